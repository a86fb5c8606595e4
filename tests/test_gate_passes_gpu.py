"""Gate lists on the exact engines (k_runs.cu: many narrow gates per pass over
the state) against the oracle, and against the same gates one call at a time
(the per-gate kernels).  Lists mix every form a pass takes (dense, real,
imaginary, diagonal of 1..6 qubits, controlled either way round, exchanges,
other permutations, dense two-qubit) with the wide gates that end a pass."""
import numpy as np
import pytest

import oracle
from paper_2111_06868_gb300 import circuits as C

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def hq():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2111_06868_gb300 import build
    from paper_2111_06868_gb300 import hq as _hq

    build.build()
    _hq.load()
    return _hq


def ctrl(U, first):
    m = np.eye(4, dtype=np.complex128)
    i = [2, 3] if first else [1, 3]
    m[np.ix_(i, i)] = U
    return m


def gate_list(n, count, seed, wide):
    rng, sm = np.random.default_rng(seed), C.SplitMix64(seed)
    ph = lambda k: np.exp(1j * rng.uniform(0, 6, k))  # noqa: E731
    two = [lambda: C.cz(), lambda: C.cphase(rng.uniform(0, 6)), lambda: C.cnot(),
           lambda: ctrl(C.random_unitary(1, sm), False), lambda: ctrl(C.random_unitary(1, sm), True),
           lambda: ctrl(C.sqrt_x(), True), lambda: C.swap(), lambda: C.fsim(np.pi / 2, rng.uniform(0, 6)),
           lambda: np.diag(ph(4)), lambda: np.diag(ph(4))[[1, 3, 0, 2]], lambda: C.random_unitary(2, sm)]
    one = [C.sqrt_x, C.sqrt_y, C.sqrt_w, C.hadamard, lambda: C.PAULI["Y"], lambda: C.PAULI["Z"],
           lambda: np.diag(ph(2)), lambda: C.random_unitary(1, sm), lambda: C.rot("X", rng.uniform(0, 6))]
    gates = []
    for _ in range(count):
        r = rng.uniform()
        if wide and r < 0.02 and n >= 5:
            k, m = 5, C.random_unitary(5, sm)
        elif wide and r < 0.06 and n >= 3:
            k, m = 3, np.kron(np.diag([0, 1]), C.cnot()) + np.kron(np.diag([1, 0]), np.eye(4))
        elif r < 0.16:
            k = int(rng.integers(1, min(n, 6) + 1))
            m = np.diag(ph(1 << k))
        elif r < 0.55:
            k, m = 2, two[rng.integers(len(two))]()
        else:
            k, m = 1, one[rng.integers(len(one))]()
        qs = tuple(int(q) for q in rng.choice(n, k, replace=False))
        gates.append(C.Gate("g", qs, np.ascontiguousarray(m, np.complex128)))
    return gates


# smallest states that take the path, tile edges of every rule (a tile of the whole state, one tile bit more, several
# tiles per SM), lists longer than one pass and than one planning window
SIZES = [(2, 12, True), (3, 30, True), (4, 40, True), (5, 60, True), (8, 300, False), (9, 200, True), (10, 250, True),
         (11, 400, True), (12, 260, False), (13, 200, True), (16, 150, True), (17, 120, False), (18, 100, True),
         (19, 100, True), (20, 80, False), (21, 60, True), (22, 60, False), (23, 60, True), (9, 5000, False)]


@pytest.mark.parametrize("n,count,wide", SIZES)
@pytest.mark.parametrize("dt", ["complex64", "complex128"])
def test_lists_match_oracle_and_single_gates(hq, n, count, wide, dt):
    gates = gate_list(n, count, 100 * n + count, wide)
    rng = np.random.default_rng(n)
    psi = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    psi /= np.linalg.norm(psi)
    dtype = getattr(torch, dt)
    start = torch.from_numpy(psi).cuda().to(dtype)
    got, one = start.clone(), start.clone()
    hq.hq_apply_blocks(got, gates)
    for g in gates:
        hq.hq_apply_gate(one, g.qubits, g.matrix)
    want = torch.from_numpy(oracle.apply_circuit(start.cpu().numpy().astype(np.complex128), C.Circuit(n, gates)))
    # the stated tolerances: complex128 max-abs 1e-12, complex64 relative L2 2e-5 per 1000 gates
    for other in (want, one.cpu().to(torch.complex128)):
        d = got.cpu().to(torch.complex128) - other
        if dt == "complex128":
            assert float(d.abs().max()) <= 1e-12
        else:
            assert float(torch.linalg.norm(d)) <= 2e-5 * max(1.0, count / 1000)


@pytest.mark.parametrize("n", [9, 10, 11, 12, 13, 14, 18, 19, 23])
@pytest.mark.parametrize("kmax", [3, 4])
def test_dense_blocks_in_passes(hq, n, kmax):
    """Lists of dense 3- and 4-qubit blocks (complex64: several per pass over the state) with narrow, diagonal and
    wider gates between them, blocks on the lowest and highest bits, more blocks than one launch takes."""
    sm, rng = C.SplitMix64(n + kmax), np.random.default_rng(n)
    gates = gate_list(n, 20, n, True)
    for _ in range(24):
        k = int(rng.integers(2, kmax + 1))
        qs = rng.choice(n, k, replace=False) if rng.uniform() < 0.7 else rng.permutation(n - k + np.arange(k))
        gates.append(C.Gate("U", tuple(int(q) for q in qs), C.random_unitary(k, sm)))
        if rng.uniform() < 0.2:
            gates += gate_list(n, 2, int(rng.integers(1000)), False)
    gates.insert(30, C.Gate("U5", (0, n - 1, 3, 1, n - 2), C.random_unitary(5, sm)))
    psi = oracle.state_init(n, "+-" * (n // 2) + "1" * (n % 2))
    st = torch.from_numpy(psi).to(torch.complex64).cuda()
    hq.hq_apply_blocks(st, gates)
    want = oracle.apply_circuit(psi.copy(), C.Circuit(n, gates))
    assert np.linalg.norm(st.cpu().numpy() - want) <= 2e-5  # the stated tolerance up to 1000 gates


@pytest.mark.parametrize("n", [12, 27])
def test_qft_list(hq, n):
    """Hundreds of controlled phases between the Hadamards: QFT of a basis state is a plane wave."""
    x = 0b101101 << (n - 8)
    circ = C.basis_prep(n, x).gates + C.qft_circuit(n).gates
    st = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
    hq.hq_simulate(st, circ, norm=False)
    y = torch.arange(1 << n, device="cuda", dtype=torch.int64)
    ang = ((x * y) % (1 << n)).to(torch.float64) * (2 * np.pi / (1 << n))
    want = torch.polar(torch.full_like(ang, 2.0 ** (-n / 2)), ang)
    assert float(torch.linalg.norm(st.to(torch.complex128) - want)) <= 2e-5


def test_list_under_capture(hq):
    """No allocation or synchronisation: a gate list can be captured into a CUDA graph and replayed."""
    n = 14
    gates = gate_list(n, 150, 5, False)
    st = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
    want = torch.empty_like(st)
    hq.hq_simulate(want, gates, norm=False)
    g = torch.cuda.CUDAGraph()
    hq.hq_simulate(st, gates, norm=False)
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        hq.hq_simulate(st, gates, norm=False)
    st.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(torch.view_as_real(st), torch.view_as_real(want))
