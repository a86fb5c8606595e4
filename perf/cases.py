"""The workloads whose speed counts, each through the calls a program makes.

``listed()`` gives them by name, ``draw(rng)`` gives more of the same ranges,
``prepare(case, seed)`` makes what a program has in hand before the call (the
circuit's gates or fused blocks, states, parameters, a batch handle) from the
seed, ``run(state)`` is one pass and returns every output, ``work(case)`` says
what a pass cannot do without, and ``exact(case, seed)`` computes the same
outputs in complex128 with plain torch operations.

The kinds of case:

  circuit     hq_simulate of a random grid circuit or a QFT: gate by gate on
              the default engine, in blocks fused on it, or in blocks on the
              tensor-core engines; the state and its squared norm come back
  expect      hq_expectation of a Pauli sum on a given state
  adjoint     hq_adjoint_grad of a batch of parameter sets: energies and
              gradients (a training step of a variational circuit)
  batch       Batch.run over circuits of uneven width (a serving load)
  trajectory  hq_state_init and hq_run_trajectory of a noisy circuit
  dm          hq_dm_init, hq_dm_apply and Tr(rho H) of a noisy circuit
"""
import math

import numpy as np
import torch

from paper_2111_06868_gb300 import circuits as C
from paper_2111_06868_gb300 import hq

DTYPES = {"complex64": torch.complex64, "complex128": torch.complex128}
DEV = "cuda"


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------
def _circuit(n, depth, gates, dtype, fuse=0, engine="auto", tokens="0"):
    return dict(kind="circuit", n=n, depth=depth, gates=gates, dtype=dtype, fuse=fuse, engine=engine, tokens=tokens)


def _expect(n, dtype, terms):
    return dict(kind="expect", n=n, dtype=dtype, terms=terms)


def _adjoint(n, layers, batch, dtype):
    return dict(kind="adjoint", n=n, layers=layers, batch=batch, dtype=dtype)


def _batch(count, n_min, n_max, depth_min, depth_max, tile_bits, max_high, fuse_k):
    return dict(kind="batch", count=count, n_min=n_min, n_max=n_max, depth_min=depth_min, depth_max=depth_max,
                tile_bits=tile_bits, max_high=max_high, fuse_k=fuse_k)


def _trajectory(n, depth, dtype):
    return dict(kind="trajectory", n=n, depth=depth, dtype=dtype)


def _dm(n, depth, dtype, engine):
    return dict(kind="dm", n=n, depth=depth, dtype=dtype, engine=engine)


def listed():
    return [
        # the small exact circuit (3x4 grid, CZ, depth 10) that is checked by eye and by tests: latency and launches
        dict(name="circuit_n12_c128", **_circuit(12, 10, "cz", "complex128")),
        # an ordinary circuit straight from its gate list, the default engine, a state that fits the L2 cache
        dict(name="circuit_n20_c64", **_circuit(20, 16, "cz", "complex64", tokens="+")),
        # the plain per-gate path of the random-circuit benchmark on a state far larger than L2
        dict(name="circuit_n28_c64", **_circuit(28, 20, "fsim", "complex64")),
        # the same kind of circuit fused into blocks of up to 4 qubits on the exact FP32 kernels
        dict(name="fused4_n28_c64", **_circuit(28, 20, "fsim", "complex64", fuse=4)),
        # the headline: 30 qubits, blocks of up to 6 qubits on the tensor cores (FP16 hi + lo)
        dict(name="fused6_n30_tc", **_circuit(30, 20, "fsim", "complex64", fuse=6, engine="tc_f16")),
        # double precision in blocks of up to 4 qubits on the tensor cores (digit slices)
        dict(name="fused4_n27_c128_tc", **_circuit(27, 20, "fsim", "complex128", fuse=4, engine="tc_c128")),
        # the energy of a trained state: a transverse-field Ising sum, one call
        dict(name="expect_n28_c64", **_expect(28, "complex64", 0)),
        # the training step of the 20-qubit variational ansatz, a batch of 64 parameter sets
        dict(name="adjoint_n20_c64", **_adjoint(20, 8, 64, "complex64")),
        # the same in double precision, a smaller batch
        dict(name="adjoint_n20_c128", **_adjoint(20, 8, 16, "complex128")),
        # a serving load of circuits of 10 to 24 qubits on the tuned tile shape
        dict(name="batch_128", **_batch(128, 10, 24, 8, 32, 13, 6, 3)),
        # one pure-state trajectory of a noisy circuit (depolarizing and amplitude damping)
        dict(name="trajectory_n24", **_trajectory(24, 12, "complex64")),
        # an exact noisy evolution: a 12-qubit density matrix (a 24-qubit vector)
        dict(name="dm_n12", **_dm(12, 10, "complex64", "tc_f16")),
    ]


def draw(rng):
    """One more case: a kind, then sizes over the whole range of the kind."""
    kind = rng.choice(["gates", "gates", "qft", "fused", "tc", "tc", "tcz", "expect", "adjoint", "adjoint", "batch",
                       "trajectory", "dm"])
    dtype = rng.choice(["complex64", "complex64", "complex128"])
    two = rng.choice(["cz", "fsim"])
    tokens = rng.choice(["0", "+", "mixed"])
    if kind == "gates":
        n = rng.randint(8, 27 if dtype == "complex64" else 23)
        return _circuit(n, rng.randint(3, 16), two, dtype, 0, "auto", tokens)
    if kind == "qft":
        return _circuit(rng.randint(8, 27 if dtype == "complex64" else 23), 1, "qft", dtype, 0, "auto", "mixed")
    if kind == "fused":
        n = rng.randint(10, 27 if dtype == "complex64" else 22)
        return _circuit(n, rng.randint(6, 20), two, dtype, rng.randint(2, 4), "auto", tokens)
    if kind == "tc":
        return _circuit(rng.randint(13, 29), rng.randint(4, 20), two, "complex64", rng.randint(5, 6), "tc_f16", tokens)
    if kind == "tcz":
        return _circuit(rng.randint(11, 26), rng.randint(4, 20), two, "complex128", rng.randint(3, 4), "tc_c128",
                        tokens)
    if kind == "expect":
        n = rng.randint(10, 28 if dtype == "complex64" else 26)
        return _expect(n, dtype, rng.choice([0, 0, rng.randint(3, 40)]))
    if kind == "adjoint":
        batch = int(round(2 ** rng.uniform(0, 6 if dtype == "complex64" else 4)))
        return _adjoint(rng.randint(6, 20), rng.randint(1, 8), batch, dtype)
    if kind == "batch":
        n_min = rng.randint(8, 16)
        depth = rng.randint(2, 16)
        tile, high = rng.choice([(12, 6), (13, 7), (13, 6), (11, 5)])
        return _batch(int(round(2 ** rng.uniform(2, 7))), n_min, n_min + rng.randint(0, 7), depth,
                      depth + rng.randint(0, 16), tile, high, rng.randint(2, 3))
    if kind == "trajectory":
        return _trajectory(rng.randint(8, 24), rng.randint(2, 12), dtype)
    return _dm(rng.randint(4, 12), rng.randint(2, 10), "complex64", rng.choice(["auto", "tc_f16"]))


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _tokens(case, seed):
    n = case["n"]
    if case["tokens"] == "mixed":
        rng = np.random.RandomState(seed % (1 << 31))
        return "".join("01+-"[i] for i in rng.randint(0, 4, n))
    return None if case["tokens"] == "0" else case["tokens"] * n


def _gates(case, seed):
    if case["gates"] == "qft":
        return C.qft_circuit(case["n"])
    return C.random_circuit(C.layout_for(case["n"]), case["depth"], seed, case["gates"])


def _pauli_sum(case, seed):
    """terms = 0: the transverse-field Ising sum on a chain; else that many random strings of 1..4 factors."""
    n = case["n"]
    if case["terms"] == 0:
        return C.ansatz_hamiltonian(n)
    rng = np.random.RandomState((seed + 17) % (1 << 31))
    out = []
    for _ in range(case["terms"]):
        qs = sorted(int(q) for q in rng.choice(n, min(n, rng.randint(1, 5)), replace=False))
        out.append((float(rng.uniform(-1, 1)), tuple((q, "XYZ"[rng.randint(0, 3)]) for q in qs)))
    return out


def _random_state(n, dtype, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    real = torch.float32 if dtype == torch.complex64 else torch.float64
    v = torch.randn(1 << n, 2, dtype=real, device=DEV, generator=g)
    return torch.view_as_complex(v / math.sqrt(2.0 * (1 << n)))


def _circuits(case, seed):
    """Widths and depths belong to the case, the gates to the seed."""
    rng = C.SplitMix64(case["count"])
    out = []
    for i in range(case["count"]):
        n, depth = rng.randint(case["n_min"], case["n_max"]), rng.randint(case["depth_min"], case["depth_max"])
        out.append(C.random_circuit(C.layout_for(n), depth, seed * 1_000_003 + i, "cz"))
    return out


def _noisy(case, seed):
    circ = C.random_circuit(C.layout_for(case["n"]), case["depth"], seed, "cz")
    return C.noisy_ops(circ, p1=1e-3, p2=1e-2, gamma=1e-3)


def _uniforms(ops, seed):
    nch = sum(1 for kind, _, _ in ops if kind == "kraus")
    return np.random.RandomState((seed + 29) % (1 << 31)).random_sample(max(1, nch))


def prepare(case, seed):
    kind, s = case["kind"], dict(case)
    if kind == "circuit":
        circ = _gates(case, seed)
        s["tokens"] = _tokens(case, seed)
        s["blocks"] = circ.gates
        if case["fuse"]:
            method = "beam" if case["fuse"] > 4 else "dag"
            s["blocks"] = hq.hq_fuse(case["n"], circ.gates, case["fuse"], method=method, restarts=8, width=32)
        s["state"] = torch.empty(1 << case["n"], dtype=DTYPES[case["dtype"]], device=DEV)
    elif kind == "expect":
        s["state"] = _random_state(case["n"], DTYPES[case["dtype"]], seed)
        s["H"] = _pauli_sum(case, seed)
    elif kind == "adjoint":
        s["circuit"] = C.ansatz(case["n"], case["layers"])
        s["H"] = C.ansatz_hamiltonian(case["n"])
        s["theta"] = C.ansatz_params(s["circuit"].n_params, case["batch"], seed)
        need = hq.hq_adjoint_workspace_bytes(case["n"], 0 if case["dtype"] == "complex64" else 1,
                                             len(s["circuit"].gates), s["circuit"].n_params, case["batch"])
        s["workspace"] = torch.empty(need, dtype=torch.uint8, device=DEV)
    elif kind == "batch":
        cs = _circuits(case, seed)
        flat = torch.empty(sum(1 << c.n for c in cs), dtype=torch.complex64, device=DEV)
        states, at = [], 0
        for c in cs:
            states.append(flat[at:at + (1 << c.n)])
            at += 1 << c.n
        s["flat"] = flat
        s["batch"] = hq.Batch(cs, states, tile_bits=case["tile_bits"], max_high=case["max_high"],
                              fuse_k=case["fuse_k"])
    elif kind == "trajectory":
        s["ops"] = _noisy(case, seed)
        s["u"] = _uniforms(s["ops"], seed)
        s["state"] = torch.empty(1 << case["n"], dtype=DTYPES[case["dtype"]], device=DEV)
    else:
        s["ops"] = _noisy(case, seed)
        s["H"] = C.ansatz_hamiltonian(case["n"])
        s["rho"] = torch.empty(1 << (2 * case["n"]), dtype=DTYPES[case["dtype"]], device=DEV)
    return s


# ----------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "circuit":
        norm2 = hq.hq_simulate(s["state"], s["blocks"], tokens=s["tokens"], engine=s["engine"], tc_min_k=4)
        return [s["state"], norm2]
    if kind == "expect":
        return [hq.hq_expectation(s["state"], s["H"])]
    if kind == "adjoint":
        e, g = hq.hq_adjoint_grad(s["circuit"], s["H"], s["theta"], dtype=s["dtype"], workspace=s["workspace"])
        return [e, g]
    if kind == "batch":
        s["batch"].run()
        return [s["flat"]]
    if kind == "trajectory":
        hq.hq_state_init(s["state"])
        chosen = hq.hq_run_trajectory(s["state"], s["ops"], s["u"])
        return [s["state"], chosen]
    hq.hq_dm_init(s["rho"])
    hq.hq_dm_apply(s["rho"], s["ops"], k_max=6, engine=s["engine"])
    return [s["rho"], hq.hq_dm_expectation(s["rho"], s["H"])]


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------
def _gate_flops(circ):
    """Floating-point operations per amplitude of the unfused gates, by their structure: a dense one-qubit gate two
    complex products and a sum, a controlled phase one product on a quarter, a permutation with phases one on half."""
    per = {"CZ": 0.5, "CPHASE": 1.5, "SWAP": 0.0, "fSim": 3.0, "RY": 6.0, "RZ": 6.0}
    return sum(per.get(g.name, 14.0) for g in circ.gates)


def work(case):
    kind = case["kind"]
    S = 16 if case.get("dtype") == "complex128" else 8
    if kind == "circuit":
        N = 1 << case["n"]
        return {"bytes": N * S, "flops": N * _gate_flops(_gates(case, 0))}
    if kind == "expect":
        N = 1 << case["n"]
        return {"bytes": N * S, "flops": 4.0 * N * len(_pauli_sum(case, 0))}
    if kind == "adjoint":
        circ = C.ansatz(case["n"], case["layers"])
        N = case["batch"] << case["n"]
        P = circ.n_params
        # the states live on the device between the sweeps: forward, then both states back and a sum per parameter
        return {"bytes": 16 * case["batch"] * P, "flops": N * (3.0 * _gate_flops(circ) + 4.0 * P)}
    if kind == "batch":
        cs = _circuits(case, 0)
        return {"bytes": sum(8 << c.n for c in cs), "flops": float(sum(_gate_flops(c) * (1 << c.n) for c in cs))}
    n = case["n"]
    circ = C.random_circuit(C.layout_for(n), case["depth"], 0, "cz")
    if kind == "trajectory":
        return {"bytes": (1 << n) * S, "flops": (1 << n) * (_gate_flops(circ) + 4.0 * n * case["depth"])}
    # U rho U^dag: each gate on both indices, and a channel's mixing of the entries
    return {"bytes": (1 << (2 * n)) * S, "flops": (1 << (2 * n)) * 4.0 * _gate_flops(circ)}


# ----------------------------------------------------------------------------
# the same outputs in complex128 with plain torch operations
# ----------------------------------------------------------------------------
def _split(psi, n, qubits):
    """psi viewed as (2^a0, 2, 2^a1, 2, ...) with the axes of the ascending qubits on their own."""
    shape, at = [], 0
    for q in qubits:
        shape += [1 << (q - at), 2]
        at = q + 1
    return psi.view(shape + [1 << (n - at)])


def _apply(psi, n, qubits, m):
    """psi <- (m on qubits) psi for a flat complex128 state; the first qubit is the high bit of m's index."""
    k = len(qubits)
    order = sorted(range(k), key=lambda j: qubits[j])
    m = np.asarray(m, np.complex128).reshape((2,) * (2 * k))
    m = m.transpose(order + [k + j for j in order]).reshape(1 << k, 1 << k)
    v = _split(psi, n, [qubits[j] for j in order])

    def part(r):
        idx = []
        for j in range(k):
            idx += [slice(None), (r >> (k - 1 - j)) & 1]
        return v[tuple(idx + [slice(None)])]

    rows = [r for r in range(1 << k) if m[r, r] != 1 or np.count_nonzero(m[r]) != 1]
    need = {c for r in rows for c in range(1 << k) if m[r, c] != 0 and c != r and c in rows}
    old = {c: part(c).clone() for c in need}
    for r in rows:
        p = part(r)
        p.mul_(complex(m[r, r]))
        for c in range(1 << k):
            if c != r and m[r, c] != 0:
                p.add_(old[c] if c in old else part(c), alpha=complex(m[r, c]))
    return psi


def _product_state(n, tokens):
    psi = torch.ones(1, dtype=torch.complex128, device=DEV)
    r = math.sqrt(0.5)
    vec = {"0": (1, 0), "1": (0, 1), "+": (r, r), "-": (r, -r)}
    for t in tokens or "0" * n:
        v = torch.tensor(vec[t], dtype=torch.complex128, device=DEV)
        psi = (psi[:, None] * v[None, :]).reshape(-1)
    return psi


def _pauli(psi, n, q, p):
    """P_q psi of a (batch, 2^n) state."""
    B = psi.shape[0]
    v = psi.view(B << q, 2, 1 << (n - 1 - q))
    out = torch.empty_like(v)
    if p == "Z":
        out[:, 0], out[:, 1] = v[:, 0], -v[:, 1]
    elif p == "X":
        out[:, 0], out[:, 1] = v[:, 1], v[:, 0]
    else:
        out[:, 0], out[:, 1] = v[:, 1] * -1j, v[:, 0] * 1j
    return out.view(B, -1)


def _sum_apply(psi, n, H):
    """H psi of a (batch, 2^n) state."""
    out = torch.zeros_like(psi)
    for c, term in H:
        t = psi
        for q, p in term:
            t = _pauli(t, n, q, p)
        out.add_(t, alpha=c)
    return out


def _vdot(a, b):
    """sum conj(a) b over the last axis."""
    return (a.conj() * b).sum(-1)


def _rotate(psi, n, q, axis, half):
    """exp(-i half P) on qubit q of a (batch, 2^n) state, one angle per row."""
    c = torch.cos(half)[:, None]
    s = torch.sin(half)[:, None]
    return psi * c - 1j * s * _pauli(psi, n, q, axis)


def _exact_adjoint(case, seed):
    n, B = case["n"], case["batch"]
    circ, H = C.ansatz(n, case["layers"]), C.ansatz_hamiltonian(n)
    theta = torch.from_numpy(C.ansatz_params(circ.n_params, B, seed)).to(DEV)
    psi = torch.zeros(B, 1 << n, dtype=torch.complex128, device=DEV)
    psi[:, 0] = 1

    def step(v, g, sign):
        if g.matrix is not None:  # CZ is its own inverse
            w = v.view(B << g.qubits[0], 2, 2, -1)
            w[:, 1, 1].neg_()
            return v
        return _rotate(v, n, g.qubits[0], g.axis, sign * theta[:, g.param] / 2)

    for g in circ.gates:
        psi = step(psi, g, 1.0)
    lam = _sum_apply(psi, n, H)
    e = _vdot(psi, lam).real
    grad = torch.zeros(B, circ.n_params, dtype=torch.float64, device=DEV)
    for g in reversed(circ.gates):
        if g.matrix is None:
            grad[:, g.param] += _vdot(lam, _pauli(psi, n, g.qubits[0], g.axis)).imag
        psi, lam = step(psi, g, -1.0), step(lam, g, -1.0)
    return [e.cpu().numpy(), grad.cpu().numpy()]


def _exact_trajectory(case, seed):
    n, ops = case["n"], _noisy(case, seed)
    u = _uniforms(ops, seed)
    psi, at, chosen = _product_state(n, None), 0, []
    for kind, qubits, m in ops:
        if kind == "gate":
            _apply(psi, n, qubits, m)
            continue
        forms = [np.asarray(K).conj().T @ np.asarray(K) for K in m]
        if all(np.allclose(F, F[0, 0] * np.eye(len(F)), atol=1e-13) for F in forms):
            p = np.array([F[0, 0].real for F in forms])  # the same for every state
        else:
            v = _split(psi, n, qubits)  # amplitude damping: one qubit
            a, b = v[:, 0], v[:, 1]
            rho = torch.stack([torch.stack([(x * y.conj()).sum() for y in (a, b)]) for x in (a, b)]).cpu().numpy()
            p = np.array([np.trace(F @ rho).real for F in forms])
        cum = np.cumsum(p)
        i = int(np.searchsorted(cum, u[at] * cum[-1], side="right"))
        i = min(i, len(p) - 1)
        at += 1
        chosen.append(i)
        _apply(psi, n, qubits, np.asarray(m[i]) / math.sqrt(p[i]))
    return [psi, np.asarray(chosen, np.int32)]


def _exact_dm(case, seed):
    n = case["n"]
    rho = torch.zeros(1 << (2 * n), dtype=torch.complex128, device=DEV)
    rho[0] = 1
    for kind, qubits, m in _noisy(case, seed):
        ks = [m] if kind == "gate" else m
        S = sum(np.kron(np.asarray(K), np.asarray(K).conj()) for K in ks)
        _apply(rho, 2 * n, tuple(qubits) + tuple(n + q for q in qubits), S)
    e = 0.0
    full = rho.view(1 << n, 1 << n)
    for c, term in C.ansatz_hamiltonian(n):
        t = full.t().contiguous()  # Tr(rho P) = sum_xy rho[x, y] P[y, x]; P acts on the rows of rho^T's index y
        for q, p in term:
            if p == "Z":
                t.view(1 << n, 1 << q, 2, -1)[:, :, 1].neg_()
            else:
                t = t.view(1 << n, 1 << q, 2, -1).flip(2).reshape(1 << n, 1 << n)
        e += c * torch.diagonal(t).sum().real.item()
    return [rho, e]


def exact(case, seed):
    kind = case["kind"]
    if kind == "circuit":
        n, circ = case["n"], _gates(case, seed)
        if n > 28:  # the state alone takes 16 GiB, and the circuit over 20 s
            return None
        psi = _product_state(n, _tokens(case, seed))
        for g in circ.gates:
            _apply(psi, n, g.qubits, g.matrix)
        return [psi, float(torch.view_as_real(psi).square().sum())]
    if kind == "expect":
        n = case["n"]
        psi = _random_state(n, DTYPES[case["dtype"]], seed).to(torch.complex128).view(1, -1)
        return [float(sum(c * _vdot(psi, _sum_apply(psi, n, [(1.0, term)])).real.item()
                          for c, term in _pauli_sum(case, seed)))]
    if kind == "adjoint":
        return _exact_adjoint(case, seed)
    if kind == "batch":
        out = []
        for c in _circuits(case, seed):
            psi = _product_state(c.n, None)
            for g in c.gates:
                _apply(psi, c.n, g.qubits, g.matrix)
            out.append(psi)
        return [torch.cat(out)]
    if kind == "trajectory":
        return _exact_trajectory(case, seed)
    return _exact_dm(case, seed)
