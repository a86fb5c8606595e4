"""Gate lists on the exact engines at the edges of what they take: gates far
from unitary, against the same gates one call at a time."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("n", [10, 12, 23])
@pytest.mark.parametrize("width", [3, 4])
@pytest.mark.parametrize("scale", [1e25, 1e-25])
@pytest.mark.parametrize("dtype", ["complex64", "complex128"])
def test_products_outside_the_float_range(hq, n, width, scale, dtype):
    """Gates scaled by 1e25 (1e-25) on a state scaled by 1e-30 (1e30): every
    state between them is in range, their product is not."""
    sm = C.SplitMix64(n)
    U = lambda k: C.random_unitary(k, sm)  # noqa: E731
    part = 1e10 if scale > 1 else 1e-10
    gates = [C.Gate("a", tuple(range(width)), U(width)), C.Gate("a", (0,), scale * U(1)),
             C.Gate("a", (1,), scale * U(1)), C.Gate("a", (1, 2), U(2)),
             C.Gate("a", (2,), np.diag([1.0, part])), C.Gate("a", (2,), np.diag([1.0, 1 / part])),
             C.Gate("a", (n - 1, 0), U(2)), C.Gate("a", (n - 2,), U(1))]
    st = torch.empty(1 << n, dtype=getattr(torch, dtype), device="cuda")
    hq.hq_state_init(st, "+")
    st *= 1e-30 if scale > 1 else 1e30
    one = st.clone()
    hq.hq_apply_blocks(st, gates)
    for g in gates:
        hq.hq_apply_gate(one, g.qubits, g.matrix)
    got, want = st.to(torch.complex128), one.to(torch.complex128)
    # 8 gates, each rounding the state by a few 2^-24 (2^-53)
    tol = 2e-6 if dtype == "complex64" else 1e-14
    top = float(want.abs().max())
    assert 0 < top < float("inf")
    assert float(torch.linalg.norm((got - want) / top)) <= tol * float(torch.linalg.norm(want / top))


def controlled(U, controls):
    m = np.eye(len(U) << controls, dtype=np.complex128)
    m[-len(U):, -len(U):] = U
    return m


@pytest.mark.parametrize("form", ["ccx", "cccx", "cswap", "ccz", "perm4"])
@pytest.mark.parametrize("n", [22, 25])
def test_lists_of_controlled_gates(hq, n, form):
    """Lists of gates that touch a part of the state on their own kernels: the
    same state as one call at a time, and no list that runs at a fraction of
    the single calls' speed."""
    rng = np.random.default_rng(n)
    m = {"ccx": controlled(C.PAULI["X"], 2), "cccx": controlled(C.PAULI["X"], 3), "cswap": controlled(C.swap(), 1),
         "ccz": controlled(C.PAULI["Z"], 2), "perm4": np.eye(16, dtype=np.complex128)[rng.permutation(16)]}[form]
    k = int(np.log2(len(m)))
    gates = [C.Gate("a", tuple(int(q) for q in rng.choice(n, k, replace=False)), m) for _ in range(16)]
    st = torch.randn(1 << n, dtype=torch.complex64, device="cuda")
    one = st.clone()
    singles = [[g] for g in gates]

    def time(runs):
        ms = []
        for _ in range(7):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda._sleep(2_000_000)  # the host is ahead of the device
            e[0].record()
            for r in runs:
                hq.hq_apply_blocks(st, r)
            e[1].record()
            torch.cuda.synchronize()
            ms.append(e[0].elapsed_time(e[1]))
        return min(ms)

    hq.hq_apply_blocks(st, gates)
    for g in gates:
        hq.hq_apply_gate(one, g.qubits, g.matrix)
    # exact products but for the sums of zeros and the order of disjoint gates: the same amplitudes
    assert float(torch.linalg.norm(st - one)) <= 2e-6 * float(torch.linalg.norm(one))
    assert time([gates]) <= 1.5 * time(singles)


@pytest.mark.parametrize("dtype", ["complex64", "complex128"])
@pytest.mark.parametrize("n", [5, 9, 12, 20, 23])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), complex(0, float("inf"))])
def test_infinities_and_nan(hq, n, dtype, bad):
    """One amplitude that is not finite: never lost by gates without a zero
    column; without blocks, amplitudes that differ in a qubit no gate acts on
    are those of the state without it."""
    sm, rng = C.SplitMix64(n), np.random.default_rng(n)
    forms = [lambda: (1, C.hadamard()), lambda: (1, C.sqrt_x()), lambda: (1, C.PAULI["Y"]), lambda: (2, C.cnot()),
             lambda: (2, C.cz()), lambda: (2, C.swap()), lambda: (2, C.fsim(np.pi / 2, 0.3)),
             lambda: (2, C.random_unitary(2, sm)), lambda: (1, np.diag(np.exp(1j * rng.uniform(0, 6, 2))))]
    act = n - 2  # qubits 0 .. n - 3 only
    gates = []
    for _ in range(40):
        k, m = forms[rng.integers(len(forms))]()
        gates.append(C.Gate("a", tuple(int(q) for q in rng.choice(act, k, replace=False)), m))
    st = torch.randn(1 << n, dtype=getattr(torch, dtype), device="cuda") * 2.0 ** (-n / 2)
    at = int(rng.integers(1 << n))
    st[at] = 0
    clean = st.clone()
    st[at] = bad
    hq.hq_apply_blocks(clean, gates)
    hq.hq_apply_blocks(st, gates)
    finite = torch.isfinite(torch.view_as_real(st)).all(dim=1)
    assert not bool(finite.all())
    assert not np.isfinite(hq.hq_expectation(st, [(1.0, ())]))
    if n < 23 or dtype == "complex128":
        apart = (torch.arange(1 << n, device="cuda") ^ at) & 3 != 0  # the two lowest bits: qubits n - 2, n - 1
        assert bool(finite[apart].all())
        assert torch.equal(torch.view_as_real(st[apart]), torch.view_as_real(clean[apart]))
