"""State-dependent channels two at a time (k_window) where small states do not
reach: sums outside FP32's range, many CTAs, several groups per thread."""
import numpy as np
import pytest

import oracle
from oracle import noise as N
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


@pytest.mark.parametrize("dtype", ["complex64", "complex128"])
@pytest.mark.parametrize("power", [66, 60, -50])
@pytest.mark.parametrize("n", [4, 12, 17])
def test_states_far_from_unit_norm(hq, n, power, dtype):
    """A state times 2^66 has a squared norm of 2^132, beyond FP32, while every
    thread's share is inside: the branches and the renormalised state are those
    of the unit state."""
    if n == 4 and power == 66:
        power = 58  # one thread holds all of the state
    rng = np.random.default_rng(n)
    psi = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    psi /= np.linalg.norm(psi)
    A = C.amplitude_damping(0.3, 0.1)
    ops = [("kraus", (q,), A) for q in (0, 2, n - 1, 1)] + [("gate", (1, 2), C.fsim(0.4, 0.3)), ("kraus", (2,), A)]
    u = rng.random(5)
    st = torch.from_numpy(psi).to(getattr(torch, dtype)).cuda()
    big = st * 2.0**power
    want = hq.hq_run_trajectory(st, ops, u)
    got = hq.hq_run_trajectory(big, ops, u)
    assert got.tolist() == want.tolist()
    # 6 operators, each rounding the state by a few 2^-24 (2^-53)
    assert float(torch.linalg.norm(big - st)) <= (2e-6 if dtype == "complex64" else 1e-14)
