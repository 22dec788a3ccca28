"""The gate engine spreads one evaluation over a cluster of thread blocks whose number
depends on precision, bond cap and how many evaluations run together.

* A result has the same bits however many evaluations run beside it: the counts cover every
  number of blocks a mixed-precision evaluation of bond cap 17..64 can get.
* Single gates at the edges of the rules (caps 16/17, 64/65, 128, odd caps, tall and wide
  M', ranks below the number of blocks) against the oracle's truncated SVD step.
* Exactly degenerate Schmidt spectra (products of Bell pairs: the bidiagonal splits into
  blocks with equal singular values).
"""
import numpy as np
import pytest

import paper_2207_03711_gb300 as G
from oracle import circuit, mps
from paper_2207_03711_gb300 import serve
from paper_2207_03711_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    G.build()
    return G.load_library()


@pytest.mark.parametrize("chi", [17, 40])
def test_results_do_not_depend_on_the_batch(chi):
    n, ne = 12, 6
    H = G.ham_jw_from_integrals(*syn.random_integrals(n // 2, 3))
    C = serve.uccsd_circuit(n, ne, 5)
    M = G.mps_create(n, chi, G.MPS_MIXED, n_slots=80)
    theta = np.stack([4 * syn.random_amplitudes(C.n_params, s) for s in range(80)])
    alone = np.array([G.vqe_energy(M, C, H, t) for t in theta[:3]])
    for count in (19, 37, 80):
        assert np.array_equal(G.vqe_energy_batch(M, C, H, theta[:count])[:3], alone)


def _step(n, chi, r, bond, U, prec, seed):
    st = mps.random_canonical(n, r, syn.random_mps_gaussians(n, r, seed))
    M = G.mps_create(n, chi, prec)
    G.mps_set_state(M, st.B, st.lam)
    ll = mps.left_lambda(st, bond)
    dw_g = G.mps_apply_gates(M, np.array([bond], dtype=np.int32), U[None])
    dw_o = mps.apply_two_site(st, bond, U, chi)
    rg, sites, lams = G.mps_get_state(M)
    # eps of the tensors times the accumulation over an inner index of at most 256, with a
    # margin of 8: lambda is compared absolutely (lambda_0 <= 1), the block by its norm
    eps = 2.0 ** -53 if prec == G.MPS_FP64 else 2.0 ** -24
    tol = 8 * 16 * eps
    assert list(rg) == st.ranks()
    assert np.abs(lams[bond] - st.lam[bond]).max() <= tol
    assert abs(dw_g - dw_o) <= tol
    block = [ll[:, None, None, None] * np.einsum("aib,bjc->aijc", b[bond], b[bond + 1]) for b in (sites, st.B)]
    assert np.linalg.norm(block[0] - block[1]) <= tol * np.linalg.norm(block[1])
    V = sites[bond + 1].reshape(rg[bond], -1)
    assert np.abs(V @ V.conj().T - np.eye(len(V))).max() <= tol


# ranks around the gate's bond: (left, bond, right) of a chain that holds them
@pytest.mark.parametrize("prec", [G.MPS_FP64, G.MPS_MIXED])
@pytest.mark.parametrize("chi,rl,rm,rr", [(1, 1, 1, 1), (5, 2, 1, 2), (16, 16, 16, 16), (17, 17, 17, 17), (17, 8, 16, 17),
                                          (33, 33, 29, 15), (64, 64, 64, 64), (64, 30, 60, 63), (65, 65, 64, 65),
                                          (128, 128, 128, 128), (128, 127, 90, 46)])
def test_single_gate_at_the_edges_of_the_rules(prec, chi, rl, rm, rr):
    n, bond = 18, 8
    r = syn.full_ranks(n, chi)
    r[bond - 1], r[bond], r[bond + 1] = rl, rm, rr
    for _ in range(n):                         # a rank is at most twice either neighbour's
        for k in range(n - 1):
            r[k] = min(r[k], 2 * (r[k - 1] if k else 1), 2 * (r[k + 1] if k < n - 2 else 1))
    U = np.linalg.qr(syn.random_gate_matrices(1, chi + rl)[0])[0]
    _step(n, chi, r, bond, U, prec, chi + rm + rr)


@pytest.mark.parametrize("prec,tol", [(G.MPS_FP64, 1e-12), (G.MPS_MIXED, 1e-5)])
def test_degenerate_spectra(prec, tol):
    """Nested Bell pairs (equal Schmidt numbers on every bond), then swaps and phases that
    keep them degenerate: the state against the statevector."""
    n, chi = 10, 32
    bell = np.kron(np.eye(2), np.eye(2)) @ circuit.CNOT @ np.kron(circuit.HAD, np.eye(2))
    gates = [(q, bell) for q in range(0, n - 1, 2)]
    for q in range(1, n - 1, 2):
        gates.append((q, circuit.SWAP))
    for q in range(0, n - 1):
        gates += [(q, np.diag([1, 1j, 1j, 1]).astype(complex)), (q, circuit.SWAP)]
    psi = np.zeros(2 ** n, dtype=complex)
    psi[0] = 1.0
    for b, U in gates:
        psi = circuit.apply_two_site_sv(psi, b, U, n)
    M = G.mps_create(n, chi, prec)
    G.mps_reset(M, [0] * n)
    G.mps_apply_gates(M, np.array([b for b, _ in gates], dtype=np.int32), np.array([U for _, U in gates]))
    _, sites, lams = G.mps_get_state(M)
    assert np.abs(mps.to_statevector(mps.MPS(sites, lams)) - psi).max() <= tol


@pytest.mark.parametrize("ranks", [(128, 130, 134), (129, 128, 200)])
def test_tensor_core_levels_with_unaligned_nodes(ranks):
    """Left bonds of 2 (mod 4) give the tensor-core levels a padded stride between nodes; an
    odd one goes to the CUDA cores. Mixed precision against FP64 of the same tensors: two
    32-bit products a level over 17 levels stay below 2e-5 of O(1) expectations."""
    n, chi = 17, 256
    r = [2, 4, 8, 16, 32, 64, *ranks, 128, 64, 32, 32, 16, 8, 4]
    r = [min(x, 2 ** min(k + 1, n - 1 - k)) for k, x in enumerate(r)]
    g = syn.random_mps_gaussians(n, r, 31)
    rr = [1] + r + [1]
    for k in range(n):
        g[k][:rr[k + 1]] *= 2.0
    st = mps.random_canonical(n, r, g)
    codes = np.random.default_rng(5).integers(0, 4, size=(40, n)).astype(np.uint8)
    codes[:, 11:] = 0
    ref = np.array([mps.expect_string(st, c) for c in codes]) / mps.norm2(st)
    M = G.mps_create(n, chi, G.MPS_MIXED)
    G.mps_set_state(M, st.B, st.lam)
    assert np.abs(G.mps_expect_paulis(M, codes) - ref).max() <= 2e-5


@pytest.mark.parametrize("n,chi,prec", [(2, 2, G.MPS_FP64), (9, 16, G.MPS_FP64), (13, 64, G.MPS_FP64),
                                        (11, 16, G.MPS_FP64), (11, 17, G.MPS_FP64), (13, 50, G.MPS_FP64), (14, 65, G.MPS_FP64),
                                        (9, 5, G.MPS_MIXED), (13, 32, G.MPS_MIXED), (13, 33, G.MPS_MIXED),
                                        (13, 50, G.MPS_MIXED), (13, 63, G.MPS_MIXED), (14, 64, G.MPS_MIXED),
                                        (14, 65, G.MPS_MIXED)])
def test_fused_levels_and_energy_sum(n, chi, prec):
    """Every Pauli word of weight <= 2 and some long ones: levels of all bond sizes, parents
    with up to four children, nodes without any, and the energy against the plain sum."""
    st = mps.random_canonical(n, syn.full_ranks(n, chi), syn.random_mps_gaussians(n, syn.full_ranks(n, chi), n + chi))
    words = {tuple(np.random.default_rng(s).integers(0, 4, n)) for s in range(30)} | {(0,) * n}
    for p in range(n):
        for q in range(p, n):
            for a in range(1, 4):
                for b in range(1, 4):
                    w = [0] * n
                    w[p], w[q] = a, b
                    words.add(tuple(w))
    codes = np.array(sorted(words), dtype=np.uint8)
    coeff = np.random.default_rng(n).normal(size=len(codes))
    ref = np.array([mps.expect_string(st, c) for c in codes]) / mps.norm2(st)
    M = G.mps_create(n, chi, prec)
    G.mps_set_state(M, st.B, st.lam)
    # 32-bit (64-bit) products through n levels, each off by a few units of the last place
    tol = n * 16 * (2.0 ** -53 if prec == G.MPS_FP64 else 2.0 ** -24)
    assert np.abs(G.mps_expect_paulis(M, codes) - ref).max() <= tol
    H = G.ham_create(codes, coeff)
    assert abs(G.mps_energy(M, H) - float(coeff @ ref.real)) <= tol * np.abs(coeff).sum()


@pytest.mark.parametrize("n_threads", [3, 20])
def test_results_do_not_depend_on_calls_in_progress(n_threads):
    """Handles on streams of their own, driven from threads: the blocks per slot follow the
    number of running slots, the bits do not."""
    import threading

    import torch
    n, chi = 10, 20
    ranks = syn.full_ranks(n, chi)
    st = mps.random_canonical(n, ranks, syn.random_mps_gaussians(n, ranks, 7))
    bonds = np.tile(np.arange(n - 1, dtype=np.int32), 6)
    U = np.array([np.linalg.qr(z)[0] for z in syn.random_gate_matrices(len(bonds), 5)])
    streams = [torch.cuda.Stream() for _ in range(n_threads)]
    handles = [G.mps_create(n, chi, G.MPS_MIXED, cuda_stream=s.cuda_stream) for s in streams]
    alone = G.mps_create(n, chi, G.MPS_MIXED)

    def run(M):
        G.mps_set_state(M, st.B, st.lam)
        G.mps_apply_gates(M, bonds, U)

    run(alone)
    ref = G.mps_get_state(alone)
    threads = [threading.Thread(target=run, args=(M,)) for M in handles]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for M in handles:
        got = G.mps_get_state(M)
        for a, b in zip(ref[1] + ref[2], got[1] + got[2]):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("prec,scales", [(G.MPS_MIXED, (0, 58, 61, 62, 63)), (G.MPS_FP64, (0, 500, 509, 510, 511))])
@pytest.mark.parametrize("n,chi", [(2, 2), (8, 16), (12, 40)])
def test_gate_on_a_state_of_large_norm(prec, scales, n, chi):
    """The reduction works up to the largest norm whose square is a number: the squared norm of
    M' is 2^(2 scale) here, so twice scale stays below 128 (1024)."""
    bond = n // 2 - 1
    U = np.linalg.qr(syn.random_gate_matrices(1, n)[0])[0]
    eps = 2.0 ** -53 if prec == G.MPS_FP64 else 2.0 ** -24
    for seed in range(4):
        r = syn.full_ranks(n, chi)
        st = mps.random_canonical(n, r, syn.random_mps_gaussians(n, r, seed))
        ll = mps.left_lambda(st, bond)
        out = []
        for s in scales:
            M = G.mps_create(n, chi, prec)
            B = list(st.B)
            B[bond] = B[bond] * 2.0 ** s
            G.mps_set_state(M, B, st.lam)
            G.mps_apply_gates(M, np.array([bond], dtype=np.int32), U[None])
            rg, sites, lams = G.mps_get_state(M)
            M.close()
            V = sites[bond + 1].reshape(rg[bond], -1)
            block = ll[:, None, None, None] * np.einsum("aib,bjc->aijc", sites[bond] * 2.0 ** -s, sites[bond + 1])
            assert np.abs(V @ V.conj().T - np.eye(len(V))).max() <= 128 * eps
            out.append((lams[bond] * 2.0 ** -s, block))
        for lam, block in out[1:]:
            # the steps round differently only where sums are split at absolute places
            assert np.abs(lam - out[0][0]).max() <= 128 * eps
            assert np.linalg.norm(block - out[0][1]) <= 128 * eps


@pytest.mark.parametrize("prec", [G.MPS_FP64, G.MPS_MIXED])
@pytest.mark.parametrize("chi", [2, 16, 40])
@pytest.mark.parametrize("ranks", [[1, 1, 2, 2, 2], [2, 2, 1, 1, 1], [2, 2, 2, 2, 2]])
def test_gate_that_annihilates_the_state(prec, chi, ranks):
    """M' = 0, tall, wide and square: one Schmidt number 0, a unit vector in B_{n+1}, zeros in B_n."""
    n, bond = 6, 1
    rng = np.random.default_rng(chi)
    r = [1] + ranks + [1]
    B = [rng.normal(size=(r[k], 2, r[k + 1])) + 0j for k in range(n)]
    M = G.mps_create(n, chi, prec)
    G.mps_set_state(M, B, [np.ones(x) for x in ranks])
    G.mps_apply_gates(M, np.array([bond], dtype=np.int32), np.zeros((1, 4, 4), dtype=complex))
    rg, sites, lams = G.mps_get_state(M)
    assert rg[bond] == 1 and lams[bond][0] == 0.0
    assert not sites[bond].any()
    assert np.linalg.norm(sites[bond + 1]) == 1.0


# (cap, precision): every number of blocks a slot can get, T wholly in shared memory or partly in L2
@pytest.mark.parametrize("n,chi,prec", [(8, 9, G.MPS_FP64), (10, 24, G.MPS_FP64), (14, 64, G.MPS_FP64), (14, 80, G.MPS_FP64),
                                        (14, 65, G.MPS_MIXED), (14, 72, G.MPS_MIXED), (16, 97, G.MPS_MIXED),
                                        (16, 128, G.MPS_MIXED)])
def test_blocks_per_slot_do_not_change_results(n, chi, prec):
    rng = np.random.default_rng(chi)
    nrot = 9                                   # each doubles the rank of every bond until it is full
    C = G.circ_create(rng.integers(1, 4, (nrot, n)).astype(np.uint8), np.arange(nrot, dtype=np.int32), np.ones(nrot))
    H = G.ham_create(rng.integers(0, 4, (40, n)).astype(np.uint8), rng.normal(size=40))
    M = G.mps_create(n, chi, prec, n_slots=80)
    theta = rng.uniform(0.3, 2.5, (80, nrot))
    alone = np.array([G.vqe_energy(M, C, H, t) for t in theta[:2]])
    assert G.mps_get_stats(M)["max_rank"] > 0.75 * min(chi, 2 ** (n // 2))
    for count in (8, 16, 39, 80):
        assert np.array_equal(G.vqe_energy_batch(M, C, H, theta[:count])[:2], alone)
