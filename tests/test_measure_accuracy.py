"""Measurements of states that are not the right-canonical ones the gate engine makes.

* FP64: a diagonal gauge on the bonds (column c of B_k times g_c, row c of B_{k+1} over g_c)
  leaves the state as it is. Every product of the contraction sums terms in which g cancels,
  so with powers of two the result has the same bits, and it is the oracle's to FP64.
"""
import numpy as np
import pytest

import paper_2207_03711_gb300 as G
from oracle import mps
from paper_2207_03711_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    G.build()
    return G.load_library()


def _polarised(n, ranks, seed):
    """Random right-canonical state with O(1) expectations of strings of Z."""
    g = syn.random_mps_gaussians(n, ranks, seed)
    r = [1] + list(ranks) + [1]
    for k in range(n):
        g[k][:r[k + 1]] *= 2.0
    return mps.random_canonical(n, ranks, g)


def _random_strings(n, count, seed):
    rng = np.random.default_rng(seed)
    codes = rng.integers(0, 4, size=(count, n)).astype(np.uint8)
    for c in codes[: count // 2]:            # some end early: closes on every level
        c[rng.integers(1, n):] = 0
    return codes


def _measure(B, lam, chi, prec, codes):
    M = G.mps_create(len(B), chi, prec)
    G.mps_set_state(M, B, lam)
    v = G.mps_expect_paulis(M, codes)
    M.close()
    return v


# bonds of 17 and up: the digit products; 130: more than one tile a side
@pytest.mark.parametrize("n,chi", [(11, 17), (12, 32), (13, 61), (16, 130)])
@pytest.mark.parametrize("spread", [4, 24, 60])
def test_fp64_does_not_depend_on_a_bond_gauge(n, chi, spread):
    ranks = syn.full_ranks(n, chi)
    st = _polarised(n, ranks, chi)
    codes = _random_strings(n, 24, chi + 1)
    plain = _measure(st.B, st.lam, chi, G.MPS_FP64, codes)
    rng = np.random.default_rng(spread)
    B = [b.copy() for b in st.B]
    for k in range(n - 1):
        g = 2.0 ** rng.integers(-spread // 2, spread // 2 + 1, ranks[k])
        B[k] = B[k] * g
        B[k + 1] = B[k + 1] / g[:, None, None]
    gauged = _measure(B, st.lam, chi, G.MPS_FP64, codes)
    assert np.array_equal(plain, gauged)
    # two products a level, each off by a few units of the last place of <psi|psi> = 1
    ref = np.array([mps.expect_string(st, c) for c in codes]) / mps.norm2(st)
    assert np.abs(gauged - ref).max() <= n * 16 * 2.0 ** -53
