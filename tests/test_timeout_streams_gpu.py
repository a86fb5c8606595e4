"""A bounded device-side wait that runs out on one stream is reported by the
next synchronous call on another: it waits for the work on blocking streams
before it reads the flags.  The wait is the batch runner's, shortened by the
test hook (no GPU fault)."""
import ctypes

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
    yield _hq
    _hq.hq_test_batch_wait_limit_ns(0)


def blocking_stream():
    torch.empty(1, device="cuda")  # the context
    h = ctypes.c_void_p()
    assert ctypes.CDLL("libcuda.so.1").cuStreamCreate(ctypes.byref(h), 0) == 0
    return torch.cuda.ExternalStream(h.value)


@pytest.mark.parametrize("other", ["default", "non-blocking", "blocking"])
def test_timeout_of_unfinished_work_on_a_blocking_stream(hq, other):
    cs = [C.random_circuit(C.layout_for(n), 10, seed, "cz") for n, seed in ((16, 1), (18, 2), (17, 3))]
    b = hq.Batch(cs, None, 12, 6, 0, 0)
    st = torch.empty(1 << 10, dtype=torch.complex128, device="cuda")
    hq.hq_state_init(st, "+")
    H = [(1.0, ((3, "X"),))]
    side = blocking_stream()
    mine = {"default": lambda: None, "non-blocking": torch.cuda.Stream, "blocking": blocking_stream}[other]()
    b.run(stream=side)
    torch.cuda.synchronize()
    assert abs(hq.hq_expectation(st, H, stream=mine) - 1.0) <= 1e-12
    try:
        hq.hq_test_batch_wait_limit_ns(1000)
        with torch.cuda.stream(side):
            torch.cuda._sleep(200_000_000)  # about 0.1 s before the run starts
        b.run(stream=side)
        with pytest.raises(hq.HQError) as e:
            hq.hq_expectation(st, H, stream=mine)
        assert e.value.name == "HQ_ERR_TIMEOUT"
        torch.cuda.synchronize()
        # reported once
        assert abs(hq.hq_expectation(st, H, stream=mine) - 1.0) <= 1e-12
    finally:
        torch.cuda.synchronize()
        hq.hq_test_batch_wait_limit_ns(0)
        b.close()
