"""The work this library does for its users, as cases that can be timed and checked.

Five kinds of call, each through the public Python entry points:

  energy    vqe_energy / vqe_energy_batch: the whole UCCSD circuit from the Hartree-Fock
            determinant, then the energy. Bond caps hold the state exactly (the result of a
            truncated circuit of thousands of gates is not unique under rounding).
  gradient  vqe_gradient: parameter-shift derivatives by shared-prefix forks.
  gates     mps_set_state, mps_apply_gates, then the Schmidt numbers (mps_get_state) and
            Pauli expectations: a stretch of circuit on a loaded state. The site tensors
            themselves are defined only up to a unitary per bond, so the outputs are what
            is defined: Schmidt numbers and expectations, and in FP64 the discarded weight
            (in mixed precision that number is a difference of 32-bit sums, good to three
            or four digits).
  measure   mps_energy: every Pauli string of a Jordan-Wigner Hamiltonian on a loaded state.
  expect    mps_expect_paulis: a list of strings on a loaded state, each value returned.

Handles of the mixed precision hold complex64 tensors; the numbers that come out of them
carry 32 bits, and are returned in that type. `exact` computes every case again in plain
64-bit NumPy or torch, without this package: fermionic operators on a statevector for the
circuits, truncated SVD steps for the gates, transfer matrices for the measurements.
"""
import functools
import math

import numpy as np
import torch

import paper_2207_03711_gb300 as G
from paper_2207_03711_gb300 import synthetic as syn

HAD = np.array([[1, 1], [1, -1]], dtype=complex) / math.sqrt(2)
RX90 = np.array([[1, -1j], [-1j, 1]], dtype=complex) / math.sqrt(2)
CNOT = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 0, 1], [0, 0, 1, 0]], dtype=complex)
SWAP = np.array([[1, 0, 0, 0], [0, 0, 1, 0], [0, 1, 0, 0], [0, 0, 0, 1]], dtype=complex)
PAULI = np.array([[[1, 0], [0, 1]], [[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], dtype=complex)


def listed():
    return [
        # one energy evaluation of an optimiser's loop in the default precision
        dict(name="energy_8q_fp64", kind="energy", n=8, ne=4, chi=16, prec="fp64", circuit="canonical", batch=1),
        # a batch of evaluations in flight together, ladder-cancelling compile
        dict(name="energy_8q_mixed_batch20", kind="energy", n=8, ne=4, chi=16, prec="mixed", circuit="cancel",
             batch=20),
        # the gradient an optimiser asks for beside the energy
        dict(name="gradient_6q_fp64", kind="gradient", n=6, ne=2, chi=8, prec="fp64", slots=17, n_sel=4),
        # the headline circuit's steady state: Pauli-rotation ladders at a saturated chi = 64
        dict(name="gates_24q_chi64_mixed", kind="gates", n=24, chi=64, prec="mixed", pattern="ladder", count=256),
        # the same stretch in the plain FP64 path
        dict(name="gates_24q_chi64_fp64", kind="gates", n=24, chi=64, prec="fp64", pattern="ladder", count=48),
        # random two-site gates in brickwork order at the largest bond cap gates run at
        dict(name="gates_32q_chi128_mixed", kind="gates", n=32, chi=128, prec="mixed", pattern="brickwork", count=62),
        # a medium odd bond cap
        dict(name="gates_20q_chi33_mixed", kind="gates", n=20, chi=33, prec="mixed", pattern="ladder", count=128),
        # <H> of a small state: latency and launches
        dict(name="measure_8q_fp64", kind="measure", n=8, chi=16, prec="fp64", window=8),
        # <H> of the headline state, all strings of 12 orbitals
        dict(name="measure_24q_chi64_mixed", kind="measure", n=24, chi=64, prec="mixed", window=24),
        # <H> in the plain FP64 path, all strings of 9 orbitals
        dict(name="measure_18q_chi64_fp64", kind="measure", n=18, chi=64, prec="fp64", window=18),
        # the measurement-bound size: a 10-orbital Hamiltonian inside a 64-qubit chi = 256 state
        dict(name="measure_64q_chi256_mixed", kind="measure", n=64, chi=256, prec="mixed", window=20),
        # a list of strings on a ragged state
        dict(name="expect_22q_chi49_mixed", kind="expect", n=22, chi=49, prec="mixed", strings=1500),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["energy", "gradient", "gates", "gates", "measure", "measure", "expect"])
    prec = rng.choice(["fp64", "mixed"])
    if kind == "energy":
        n = rng.choice([4, 6, 8])
        return dict(kind=kind, n=n, ne=2 * rng.randint(1, n // 2 - 1), chi=rng.randint(2 ** (n // 2), 20), prec=prec,
                    circuit=rng.choice(["canonical", "cancel"]), batch=_log_int(rng, 1, 24))
    if kind == "gradient":
        n = rng.choice([4, 6])
        return dict(kind=kind, n=n, ne=rng.choice([2, n - 2]), chi=rng.randint(2 ** (n // 2), 20),
                    prec="fp64", slots=rng.randint(5, 24), n_sel=rng.randint(1, 4))
    if kind == "gates":
        chi = _log_int(rng, 8, 128 if prec == "mixed" else 64)
        n = rng.randint(2 * math.ceil(math.log2(chi)) + 4, 32)
        each = (100 + 7.0 * chi * chi / 16) * (1 if prec == "mixed" else 8)   # rough microseconds, for the size only
        return dict(kind=kind, n=n, chi=chi, prec=prec, pattern=rng.choice(["ladder", "brickwork"]),
                    count=max(8, min(_log_int(rng, 16, 200), int(3e5 / each))))
    if kind == "measure":
        chi = _log_int(rng, 8, 256 if prec == "mixed" else 64)
        n = rng.randint(2 * math.ceil(math.log2(chi)) + 2, 40)
        top = min(n, 24) if chi <= 64 else 16
        return dict(kind=kind, n=n, chi=chi, prec=prec, window=rng.randint(4, (top if prec == "mixed" else 18) // 2) * 2)
    chi = _log_int(rng, 8, 160 if prec == "mixed" else 64)
    return dict(kind=kind, n=rng.randint(2 * math.ceil(math.log2(chi)) + 2, 40), chi=chi, prec=prec,
                strings=_log_int(rng, 10, 1500 if chi <= 64 else 300))


# ------------------------------------------------------------------------- inputs
def canonical_state(n, chi, seed, canonical):
    """Site tensors (r_{k-1}, 2, r_k) and Schmidt numbers of a seeded random MPS at the
    largest ranks, right-canonical, with Schmidt spectra that fall off over each bond as a
    correlated state's do and with O(1) local expectations. canonical: also rotated so that
    the Schmidt numbers are exact (what applying gates wants; a measurement reads only the
    tensors)."""
    r = [1] + syn.full_ranks(n, chi) + [1]
    rng = np.random.default_rng(60_000 + seed)
    B = []
    for k in range(n):
        z = rng.normal(size=(2, 2 * r[k + 1], r[k]))
        z = (z[0] + 1j * z[1]).reshape(2, r[k + 1], r[k])
        z[0] *= 2.0
        z *= np.exp(-8.0 * np.arange(r[k + 1]) / r[k + 1])[None, :, None]
        q, _ = np.linalg.qr(z.reshape(2 * r[k + 1], r[k]))
        B.append(np.ascontiguousarray(q.conj().T).reshape(r[k], 2, r[k + 1]))
    lam = []
    L = np.ones((1, 1), dtype=complex)
    for k in range(n - 1):
        if not canonical:
            lam.append(np.full(r[k + 1], r[k + 1] ** -0.5))
            continue
        L = sum(B[k][:, i].conj().T @ L @ B[k][:, i] for i in range(2))
        w, W = np.linalg.eigh(L)
        w, W = np.maximum(w[::-1], 0.0), W[:, ::-1]
        B[k] = np.einsum("aib,bc->aic", B[k], W, optimize=True)
        B[k + 1] = np.einsum("cb,bjd->cjd", W.conj().T, B[k + 1], optimize=True)
        L = np.diag(w).astype(complex)
        lam.append(np.sqrt(w))
    return B, lam


@functools.lru_cache(maxsize=4)
def hamiltonian_strings(n, window):
    """Pauli codes of a spin-conserving Jordan-Wigner Hamiltonian of window / 2 spatial
    orbitals on the middle `window` qubits of n: Z_p, Z_p Z_q, hops with their Z chains
    (also times another number operator), and double excitations with an even number of Y."""
    lo = (n - window) // 2
    sites = range(lo, lo + window)
    out = set()
    for p in sites:
        for q in range(p, lo + window):
            s = np.zeros(n, dtype=np.uint8)
            s[[p, q]] = 3
            out.add(s.tobytes())
            if q > p and (q - p) % 2 == 0:
                for a in (1, 2):
                    s[:] = 0
                    s[p + 1:q] = 3
                    s[[p, q]] = a
                    out.add(s.tobytes())
                    for t in sites:
                        if t not in (p, q):
                            u = s.copy()
                            u[t] ^= 3
                            out.add(u.tobytes())
    pairs = [(p, q) for p in sites for q in range(p + 1, lo + window)]
    for p, q in pairs:
        for r, t in pairs:
            if q < r and (p + q + r + t) % 2 == 0:
                s = np.zeros(n, dtype=np.uint8)
                s[p + 1:q] = 3
                s[r + 1:t] = 3
                up = np.array([(x - p) % 2 for x in (p, q, r, t)])
                for ab in np.ndindex(2, 2, 2, 2):   # an even number of Y on each spin
                    if sum(ab) % 2 == 0 and up @ ab % 2 == 0:
                        s[[p, q, r, t]] = np.add(ab, 1)
                        out.add(s.tobytes())
    return np.array([np.frombuffer(b, dtype=np.uint8) for b in sorted(out)])


def hamiltonian(n, window, seed):
    """The strings with seeded coefficients: diagonal terms dominate and share a sign, as in
    a molecule, the others are small and of both signs."""
    codes = hamiltonian_strings(n, window)
    rng = np.random.default_rng(70_000 + seed)
    diagonal = np.all((codes == 0) | (codes == 3), axis=1)
    return codes, np.where(diagonal, -rng.uniform(0.2, 1.0, len(codes)), rng.normal(0.0, 0.02, len(codes)))


def random_strings(n, count, seed):
    """Strings shaped like Jordan-Wigner terms anywhere on the chain, some of them twice."""
    rng = np.random.default_rng(80_000 + seed)
    out = np.zeros((count, n), dtype=np.uint8)
    for s in out:
        p, q, r, t = sorted(rng.choice(n, 4, replace=False))
        for a, b in ((p, q), (r, t))[:rng.integers(1, 3)]:
            s[a + 1:b] = rng.choice([0, 3])
            s[[a, b]] = rng.integers(1, 4, 2)
    out[rng.integers(count)] = out[0]
    return out


def rotation_gates(code, phi):
    """exp(-i phi P / 2) as fused two-site gates: basis changes, the parity carried upward by
    CNOTs (SWAPs across identities), Rz, and back."""
    S = np.nonzero(code)[0]
    lo, hi = S[0], S[-1]
    B = [np.eye(2) if c in (0, 3) else HAD if c == 1 else RX90 for c in code]
    first = np.eye(2)
    up = []
    for b in range(lo, hi):
        pre = np.kron(B[lo] if b == lo else first, B[b + 1])
        up.append((b, (CNOT if code[b + 1] else SWAP) @ pre))
    rz = np.kron(np.eye(2), np.diag([np.exp(-0.5j * phi), np.exp(0.5j * phi)]))
    top = (hi - 1, up[-1][1].conj().T @ rz @ up[-1][1])
    return up[:-1] + [top] + [(b, U.conj().T) for b, U in up[-2::-1]]


def gate_list(case, seed):
    n, count = case["n"], case["count"]
    if case["pattern"] == "brickwork":
        layers = -(-count // (n // 2 - 1))
        bonds = syn.brickwork_bonds(n, layers)[:count]
        U = np.array([np.linalg.qr(z)[0] for z in syn.random_gate_matrices(len(bonds), seed)])
        return np.array(bonds, dtype=np.int32), U
    rng = np.random.default_rng(90_000 + seed)
    gates = []
    while len(gates) < count:
        p, q, r, t = sorted(rng.choice(n, 4, replace=False))
        code = np.zeros(n, dtype=np.uint8)
        code[p + 1:q] = 3
        code[r + 1:t] = 3
        code[[p, q, r, t]] = rng.integers(1, 3, 4)
        gates += rotation_gates(code, rng.normal(0.0, 0.2))
    return np.array([b for b, _ in gates[:count]], dtype=np.int32), np.array([U for _, U in gates[:count]])


def amplitudes(case, seed):
    return [syn.random_amplitudes(len(excitations(case["n"], case["ne"])), 100 * seed + b)
            for b in range(case.get("batch", 1))]


def selection(case, seed):
    count = len(excitations(case["n"], case["ne"]))
    return np.random.default_rng(95_000 + seed).choice(count, min(case["n_sel"], count), replace=False).astype(np.int32)


def prepare(case, seed):
    n, chi, kind = case["n"], case["chi"], case["kind"]
    s = dict(kind=kind, mixed=case["prec"] == "mixed")
    prec = G.MPS_MIXED if s["mixed"] else G.MPS_FP64
    slots = case["slots"] if kind == "gradient" else case.get("batch", 1)
    s["mps"] = G.mps_create(n, chi, prec, n_slots=slots)
    if kind in ("energy", "gradient"):
        s["ham"] = G.ham_jw_from_integrals(*syn.random_integrals(n // 2, seed))
        s["circ"] = G.circ_uccsd(n, case["ne"])
        if case.get("circuit") == "cancel":
            G.circ_cancel_ladders(s["circ"])
        s["theta"] = np.array(amplitudes(case, seed))
        if kind == "gradient":
            s["sel"] = selection(case, seed)
        return s
    s["B"], s["lam"] = canonical_state(n, chi, seed, kind == "gates")
    if kind == "gates":
        s["bonds"], s["U"] = gate_list(case, seed)
        s["strings"] = random_strings(n, 48, seed)
        return s
    G.mps_set_state(s["mps"], s["B"], s["lam"])
    if kind == "measure":
        s["ham"] = G.ham_create(*hamiltonian(n, case["window"], seed))
    else:
        s["strings"] = random_strings(n, case["strings"], seed)
    return s


def _table(lam, chi):
    """Schmidt numbers as bonds x chi, zeros beyond each bond's rank."""
    out = np.zeros((len(lam), chi))
    for row, l in zip(out, lam):
        row[:len(l)] = l
    return out


def run(s):
    kind, mixed = s["kind"], s["mixed"]
    if kind == "energy":
        if len(s["theta"]) == 1:
            return G.vqe_energy(s["mps"], s["circ"], s["ham"], s["theta"][0])
        e = G.vqe_energy_batch(s["mps"], s["circ"], s["ham"], s["theta"])
        return e.astype(np.float32) if mixed else e
    if kind == "gradient":
        return G.vqe_gradient(s["mps"], s["circ"], s["ham"], s["theta"][0], s["sel"])
    if kind == "measure":
        return G.mps_energy(s["mps"], s["ham"])
    if kind == "expect":
        v = G.mps_expect_paulis(s["mps"], s["strings"])
        return v.astype(np.complex64) if mixed else v
    G.mps_set_state(s["mps"], s["B"], s["lam"])
    dropped = G.mps_apply_gates(s["mps"], s["bonds"], s["U"])
    v = G.mps_expect_paulis(s["mps"], s["strings"])
    lam = _table(G.mps_get_state(s["mps"])[2], s["mps"].chi)
    if mixed:
        return dict(expect=v.astype(np.complex64), schmidt=lam.astype(np.float32))
    return dict(dropped=dropped, expect=v, schmidt=lam)


# --------------------------------------------------------------------------- work
def _ranks(case):
    return [1] + syn.full_ranks(case["n"], case["chi"]) + [1]


def _prefix_nodes(codes):
    """Distinct prefixes of the strings that still have a letter to come, per site, and the
    number of strings."""
    last = codes.shape[1] - 1 - np.argmax(codes[:, ::-1] != 0, axis=1)
    return [len(np.unique(codes[last >= k][:, :k], axis=0)) if k else 1 for k in range(int(last.max()) + 1)]


def _measure_flops(r, codes):
    """Prefix-shared transfer matrices: one L B (both i) and one B^+ (L B) per prefix."""
    nodes = _prefix_nodes(codes)
    return sum(8.0 * u * 4 * r[k] * r[k + 1] * max(r[k], r[k + 1]) for k, u in enumerate(nodes))


def _gate_flops(m, r, n, k):
    """theta contraction, singular values and right vectors (4 m n^2 + 8 n^3 complex), update."""
    big, small = max(m, n), min(m, n)
    return 8.0 * m * r * n + 32.0 * m * n + 4.0 * (4.0 * big * small ** 2 + 8.0 * small ** 3) + 8.0 * m * n * k


def _gates_flops(case, bonds):
    r = _ranks(case)
    return sum(_gate_flops(2 * r[b], r[b + 1], 2 * r[b + 2], r[b + 1]) for b in bonds)


def _rotation_count(case):
    """Mean two-site gates of the compiled ansatz: 2 (hi - lo) - 1 per string."""
    total = 0
    for occ, vir in excitations(case["n"], case["ne"]):
        total += (2 if len(occ) == 1 else 8) * (2 * (max(vir) - min(occ)) - 1)
    return total * (0.6 if case.get("circuit") == "cancel" else 1.0)


def work(case):
    n, es = case["n"], 8 if case["prec"] == "mixed" else 16
    r = _ranks(case)
    state = float(sum(2 * r[k] * r[k + 1] for k in range(n))) * es
    if case["kind"] in ("energy", "gradient"):
        forks = case["batch"] if case["kind"] == "energy" else 1 + 8 * case["n_sel"]   # forks share half a circuit
        strings = hamiltonian_strings(n, n)
        gates = _rotation_count(case)
        mid = r[n // 2]
        flops = forks * (gates * _gate_flops(mid, mid, mid, mid) + _measure_flops(r, strings))
        return {"bytes": forks * (state + 16.0 * len(strings)) + gates * 32.0, "flops": flops}
    if case["kind"] == "gates":
        bonds, _ = gate_list(case, 0)
        return {"bytes": 2 * state + 288.0 * len(bonds), "flops": _gates_flops(case, bonds)}
    codes = hamiltonian_strings(n, case["window"]) if case["kind"] == "measure" else random_strings(n, case["strings"], 0)
    return {"bytes": state + float(codes.size) + 16.0 * len(codes), "flops": _measure_flops(r, codes)}


# -------------------------------------------------------------- the same in 64 bits
def excitations(n, ne):
    """(occupied, virtual) of the spin-conserving singles, then doubles, in order."""
    occ, vir = range(ne), range(ne, n)
    one = [((i,), (a,)) for i in occ for a in vir if (i - a) % 2 == 0]
    two = [((i, j), (a, b)) for i in occ for j in range(i + 1, ne) for a in vir for b in range(a + 1, n)
           if i % 2 + j % 2 == a % 2 + b % 2]
    return one + two


def _ladder(psi, q, create):
    """a_q or a+_q on a statevector whose index has bit q = occupation of q."""
    idx = np.arange(len(psi))
    below = idx & ((1 << q) - 1)
    sign = np.ones(len(psi))
    while np.any(below):
        sign *= 1 - 2.0 * (below & 1)
        below = below >> 1
    out = np.zeros_like(psi)
    src = idx[((idx >> q) & 1) == (0 if create else 1)]
    out[src ^ (1 << q)] = sign[src] * psi[src]
    return out


def _generator(psi, occ, vir):
    """(tau - tau+) psi, tau = a+_a a_i or a+_a a+_b a_i a_j."""
    t, u = psi, psi
    for q in occ[::-1]:
        t = _ladder(t, q, False)
    for q in vir[::-1]:
        t = _ladder(t, q, True)
    for q in vir:
        u = _ladder(u, q, False)
    for q in occ:
        u = _ladder(u, q, True)
    return t - u


def _exp_generator(psi, occ, vir, theta):
    g = _generator(psi, occ, vir)
    return psi + math.sin(theta) * g + (1 - math.cos(theta)) * _generator(g, occ, vir)   # G^3 = -G


def _apply_hamiltonian(psi, h, eri):
    m = len(h)
    down = [[_ladder(psi, 2 * q + s, False) for q in range(m)] for s in range(2)]
    out = np.zeros_like(psi)
    for s in range(2):
        for p in range(m):
            out += _ladder(sum(h[p, q] * down[s][q] for q in range(m)), 2 * p + s, True)
    # 1/2 (pq|rs) a+_ps a+_rt a_st a_qs
    for s in range(2):
        for t in range(2):
            pair = np.array([[_ladder(down[s][q], 2 * u + t, False) for u in range(m)] for q in range(m)])
            mixed = np.einsum("pqru,quv->prv", 0.5 * eri, pair, optimize=True)
            for p in range(m):
                inner = sum(_ladder(mixed[p, r], 2 * r + t, True) for r in range(m))
                out += _ladder(inner, 2 * p + s, True)
    return out


def _exact_circuit(case, seed):
    n, ne = case["n"], case["ne"]
    h, eri = syn.random_integrals(n // 2, seed)
    exc = excitations(n, ne)

    def state(theta, derivative=None):
        psi = np.zeros(2 ** n)
        psi[(1 << ne) - 1] = 1.0
        for e, (occ, vir) in enumerate(exc):
            psi = _exp_generator(psi, occ, vir, theta[e])
            if e == derivative:
                psi = _generator(psi, occ, vir)
        return psi

    thetas = amplitudes(case, seed)
    if case["kind"] == "gradient":
        hpsi = _apply_hamiltonian(state(thetas[0]), h, eri)
        return np.array([2 * hpsi @ state(thetas[0], int(e)) for e in selection(case, seed)])
    e = np.array([psi @ _apply_hamiltonian(psi, h, eri) for psi in map(state, thetas)])
    return float(e[0]) if len(e) == 1 else e


def _exact_expect(B, codes):
    """<P> / <psi|psi> of every string by transfer matrices, prefixes shared."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    B = [torch.from_numpy(np.ascontiguousarray(b)).to(dev) for b in B]
    P = torch.from_numpy(PAULI).to(dev)
    n = len(B)
    R = [torch.ones((1, 1), dtype=torch.complex128, device=dev)]
    for b in B[::-1]:
        R.append(torch.einsum("aib,bc,dic->ad", b, R[-1], b.conj()))
    R = R[::-1]
    strings, back = np.unique(codes, axis=0, return_inverse=True)
    end = np.where((strings != 0).any(axis=1), n - 1 - np.argmax(strings[:, ::-1] != 0, axis=1), -1)
    out = torch.ones(len(strings), dtype=torch.complex128, device=dev)
    norm = R[0][0, 0]
    live = np.nonzero(end >= 0)[0]
    env, at = torch.ones((1, 1, 1), dtype=torch.complex128, device=dev), np.zeros(len(live), dtype=np.int64)
    for k in range(n):
        if not len(live):
            break
        key, which = np.unique(at * 4 + strings[live, k], return_inverse=True)
        parent, letter = torch.from_numpy(key // 4).to(dev), torch.from_numpy(key % 4).to(dev)
        new = []
        for j in range(0, len(key), 256):   # sum_ij P_ij (B^i)^+ L B^j
            T = torch.einsum("uab,bjc->ujac", env[parent[j:j + 256]], B[k])
            W = torch.einsum("uij,ujac->uiac", P[letter[j:j + 256]], T)
            new.append(torch.einsum("aid,uiac->udc", B[k].conj(), W))
        env, at = torch.cat(new), which.reshape(-1)
        closed = end[live] == k
        if closed.any():
            nodes = torch.from_numpy(at[closed]).to(dev)
            # <psi| on the left index, |psi> on the right one: R is (ket, bra)
            val = torch.einsum("udc,cd->u", env, R[k + 1])
            out[torch.from_numpy(live[closed]).to(dev)] = val[nodes] / norm
        live, at = live[~closed], at[~closed]
        keep, at = np.unique(at, return_inverse=True)
        env, at = env[torch.from_numpy(keep).to(dev)], at.reshape(-1)
    return out.cpu().numpy()[back.reshape(-1)]


def _exact_gates(case, seed):
    B, lam = canonical_state(case["n"], case["chi"], seed, True)
    dropped = 0.0
    cutoff = 2.0 ** -20 if case["prec"] == "mixed" else 1e-13
    for b, U in zip(*gate_list(case, seed)):
        theta = np.einsum("aib,bjc->aijc", B[b], B[b + 1], optimize=True)
        M = np.einsum("ijkl,aklc->aijc", U.reshape(2, 2, 2, 2), theta)
        rl, _, _, rr = M.shape
        left = lam[b - 1] if b else np.ones(1)
        _, s, V = np.linalg.svd((left[:, None, None, None] * M).reshape(2 * rl, 2 * rr), full_matrices=False)
        k = min(case["chi"], int(np.count_nonzero(s > cutoff * s[0])))
        dropped += float(np.sum(s[k:] ** 2) / np.sum(s ** 2))
        B[b + 1] = V[:k].reshape(k, 2, rr)
        B[b] = (M.reshape(2 * rl, 2 * rr) @ V[:k].conj().T).reshape(rl, 2, k)
        lam[b] = s[:k]
    out = dict(expect=_exact_expect(B, random_strings(case["n"], 48, seed)), schmidt=_table(lam, case["chi"]))
    return out if case["prec"] == "mixed" else dict(out, dropped=dropped)


def exact(case, seed):
    if case["kind"] in ("energy", "gradient"):
        return _exact_circuit(case, seed)
    if case["kind"] == "gates":
        return _exact_gates(case, seed)
    B, _ = canonical_state(case["n"], case["chi"], seed, False)
    if case["kind"] == "expect":
        return _exact_expect(B, random_strings(case["n"], case["strings"], seed))
    codes, coeff = hamiltonian(case["n"], case["window"], seed)
    if _measure_flops(_ranks(case), codes) > 1e13:
        return None   # over 20 seconds of 64-bit arithmetic
    return float(coeff @ _exact_expect(B, codes).real)
