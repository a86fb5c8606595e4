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
