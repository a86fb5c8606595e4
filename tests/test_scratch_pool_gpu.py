"""Device scratch of large calls is given back: a call that synchronises leaves
no more than the pool keeps, one that does not leaves it to the caller's next
synchronisation."""
import numpy as np
import pytest

from paper_2111_06868_gb300 import circuits as C

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
KEPT = 32 << 20  # what the pool keeps mapped
SLACK = 4 << 20  # other users of the device memory in this process


@pytest.fixture(scope="module")
def hq():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2111_06868_gb300 import build
    from paper_2111_06868_gb300 import hq as _hq

    build.build()
    _hq.load()
    return _hq


def free_bytes():
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("stream", ["default", "side"])
def test_expectation_of_many_groups(hq, stream):
    n = 20
    s = torch.cuda.Stream() if stream == "side" else None
    rng = np.random.default_rng(2)
    H = [(1.0, tuple((int(q), "XYZ"[rng.integers(3)]) for q in rng.choice(n, 8, replace=False))) for _ in range(15000)]
    st = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
    hq.hq_state_init(st, "+")
    hq.hq_expectation(st, H[:40])
    torch.cuda.synchronize()
    before = free_bytes()
    hq.hq_expectation(st, H, stream=s)  # scratch of about 40 MB or more
    assert before - free_bytes() <= KEPT + SLACK


def test_block_list_until_the_next_synchronisation(hq):
    n = 15
    rng = np.random.default_rng(0)
    U = [C.random_unitary(6, C.SplitMix64(i)) for i in range(4)]
    gates = [C.Gate("a", tuple(int(x) for x in rng.choice(n, 6, replace=False)), U[i % 4]) for i in range(1500)]
    st = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
    hq.hq_state_init(st)
    hq.hq_apply_blocks(st, gates[:2], engine="tc_f16")
    torch.cuda.synchronize()
    before = free_bytes()
    hq.hq_apply_blocks(st, gates, engine="tc_f16")  # matrices of about 90 MB
    torch.cuda.synchronize()
    assert before - free_bytes() <= KEPT + SLACK
    hq.hq_simulate(st, gates, engine="tc_f16")  # synchronises itself
    assert before - free_bytes() <= KEPT + SLACK
