"""Measurements of states that are not the right-canonical ones the gate engine makes.

* FP64: a diagonal gauge on the bonds (column c of B_k times g_c, row c of B_{k+1} over g_c)
  leaves the state as it is. Every product of the contraction sums terms in which g cancels,
  so with powers of two the result has the same bits, and it is the oracle's to FP64.
* Mixed: sites that pass a bond through are exact on the tensor cores, however many.
"""
import ctypes

import numpy as np
import pytest
import torch

import paper_2207_03711_gb300 as G
from oracle import mps
from paper_2207_03711_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    G.build()
    return G.load_library()


def _polarised(n, ranks, seed, bias=2.0):
    """Random right-canonical state that prefers |0> where its bonds leave it the choice."""
    g = syn.random_mps_gaussians(n, ranks, seed)
    r = [1] + list(ranks) + [1]
    for k in range(n):
        g[k][:r[k + 1]] *= bias
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


def _with_idle_sites(st, at, count):
    """st with `count` sites in |0> that pass bond `at` - 1 through."""
    D = st.B[at].shape[0]
    idle = np.zeros((D, 2, D), dtype=complex)
    idle[:, 0, :] = np.eye(D)
    return st.B[:at] + [idle.copy() for _ in range(count)] + st.B[at:], \
        st.lam[:at] + [st.lam[at - 1]] * count + st.lam[at:]


# a bond of one packed tile, of one tile and of two column tiles
@pytest.mark.parametrize("n,chi", [(18, 64), (20, 100), (22, 160)])
def test_mixed_sites_that_pass_a_bond_through_are_exact(n, chi):
    """100 idle sites in the middle of a state: their products are single terms with factor 1,
    exact but for the first, which may drop the last bit of an entry of L (its two 11-bit parts
    hold 23 bits and a sign of 24). <P> is sum L conj(Q) with ||L||_F <= ||rho||_F <= 1 and
    ||Q||_F <= sqrt(chi), so that is at most sqrt(chi) 2^-23, doubled for the two products."""
    ranks = syn.full_ranks(n, chi)
    st = _polarised(n, ranks, chi + 3, bias=8.0)
    at, idle = n // 2, 100
    codes = np.zeros((6, n), dtype=np.uint8)      # pairs of Z and some X around the idle sites
    for c, (p, q, l) in zip(codes, [(at - 1, at, 3), (at - 2, at, 3), (at - 2, at + 1, 3), (0, at, 3), (at - 1, at, 1), (1, at, 2)]):
        c[p], c[q] = l, 3
    long = np.concatenate([codes[:, :at], np.zeros((len(codes), idle), dtype=np.uint8), codes[:, at:]], axis=1)
    short = _measure(st.B, st.lam, chi, G.MPS_MIXED, codes)
    B, lam = _with_idle_sites(st, at, idle)
    v = _measure(B, lam, chi, G.MPS_MIXED, long)
    assert np.abs(short).max() > 0.6              # a systematic factor would be seen
    assert np.abs(v - short).max() <= 2 * np.sqrt(chi) * 2.0 ** -23


# bonds of 33..48, where few nodes and many would favour different kernels; 64: two children a tile
@pytest.mark.parametrize("n,chi", [(14, 34), (14, 48), (15, 64)])
def test_mixed_values_do_not_depend_on_the_company(n, chi):
    """A string's value is the same alone, among hundreds and with chunks of 16 nodes: every
    number of a level comes out of the same sums in the same order."""
    st = _polarised(n, syn.full_ranks(n, chi), chi + 5)
    codes = _random_strings(n, 400, chi)
    M = G.mps_create(n, chi, G.MPS_MIXED)
    G.mps_set_state(M, st.B, st.lam)
    v = G.mps_expect_paulis(M, codes)
    for i in (0, 7, 200, 399):
        assert np.array_equal(G.mps_expect_paulis(M, codes[i:i + 1]), v[i:i + 1])
    G.mps_set_meas_budget(M, 1)
    assert np.array_equal(G.mps_expect_paulis(M, codes), v)


def _pool_used():
    """Bytes in use of the device's memory pool, which the library allocates from."""
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    dev, pool, used = ctypes.c_int(), ctypes.c_void_p(), ctypes.c_uint64()
    assert cu.cuCtxGetDevice(ctypes.byref(dev)) == 0
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), dev) == 0
    assert cu.cuMemPoolGetAttribute(pool, 7, ctypes.byref(used)) == 0   # CU_MEMPOOL_ATTR_USED_MEM_CURRENT
    return used.value


@pytest.mark.parametrize("prec", [G.MPS_FP64, G.MPS_MIXED])
def test_a_smaller_budget_gives_the_memory_back(prec):
    n, chi = 16, 64
    st = _polarised(n, syn.full_ranks(n, chi), 3)
    codes = _random_strings(n, 2000, 4)
    torch.zeros(1, device="cuda")

    def held(budgets):
        before = _pool_used()
        M = G.mps_create(n, chi, prec)
        G.mps_set_state(M, st.B, st.lam)
        for b in budgets:
            G.mps_set_meas_budget(M, b)
            G.mps_expect_paulis(M, codes)
        used = _pool_used() - before
        M.close()
        return used

    small = held([1])
    assert held([0]) > 2 * small
    assert held([0, 1]) == small


def test_fp64_levels_of_many_batches():
    """chi = 256: a batch of the digit products holds 64 nodes, the levels here have hundreds,
    some without children. Against the oracle, and bit for bit against chunks of 16 nodes."""
    n, chi = 18, 256
    st = _polarised(n, syn.full_ranks(n, chi), 6)
    codes = _random_strings(n, 300, 7)
    M = G.mps_create(n, chi, G.MPS_FP64)
    G.mps_set_state(M, st.B, st.lam)
    v = G.mps_expect_paulis(M, codes)
    assert G.mps_get_stats(M)["tc_gemm_launches"] > 0
    G.mps_set_meas_budget(M, 1)
    assert np.array_equal(G.mps_expect_paulis(M, codes), v)
    some = np.arange(0, 300, 25)
    ref = np.array([mps.expect_string(st, codes[i]) for i in some]) / mps.norm2(st)
    assert np.abs(v[some] - ref).max() <= n * 16 * 2.0 ** -53


@pytest.mark.parametrize("prec,tol", [(G.MPS_FP64, 16 * 160 * 2.0 ** -53), (G.MPS_MIXED, 2e-5)])
def test_ranks_that_fall_fast(prec, tol):
    """A bond above 64 beside one below the tensor cores' smallest (neither route, nor the fused
    kernels): loaded tensors may have any ranks within the caps. They are not canonical either:
    sums of |L| |B| are up to the root of a bond above <psi|psi>."""
    n, chi = 16, 128
    ranks = [2, 4, 8, 16, 32, 64, 100, 12, 90, 64, 32, 16, 8, 4, 2]
    r = [1] + ranks + [1]
    rng = np.random.default_rng(2)
    B = [(rng.normal(size=(r[k], 2, r[k + 1])) + 1j * rng.normal(size=(r[k], 2, r[k + 1]))) / np.sqrt(4 * r[k + 1])
         for k in range(n)]
    st = mps.MPS(B, [np.ones(x) for x in ranks])
    codes = _random_strings(n, 60, 8)
    codes[:20, :6] = 0
    M = G.mps_create(n, chi, prec)
    G.mps_set_state(M, B, st.lam)
    v = G.mps_expect_paulis(M, codes)
    ref = np.array([mps.expect_string(st, c) for c in codes]) / mps.norm2(st)
    assert np.abs(v - ref).max() <= tol
    G.mps_set_meas_budget(M, 1)
    assert np.array_equal(G.mps_expect_paulis(M, codes), v)
