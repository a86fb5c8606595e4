"""Synchronous calls from many host threads: the right values at the same
time, and nothing that stays behind when a thread ends."""
import threading

import pytest

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


def resident_kb():
    return int(next(l for l in open("/proc/self/status") if l.startswith("VmRSS")).split()[1])


def test_nothing_is_left_per_thread(hq):
    st = torch.empty(1 << 10, dtype=torch.complex64, device="cuda")
    hq.hq_state_init(st, "+")
    torch.cuda.synchronize()
    H = [(1.0, ((3, "X"),))]

    def threads(count):
        for _ in range(count):
            t = threading.Thread(target=lambda: hq.hq_expectation(st, H))
            t.start()
            t.join()

    threads(500)
    before = resident_kb()
    threads(6000)
    # a pinned buffer per thread would be 1.5 kB each, 9 MB
    assert resident_kb() - before <= 3000


def test_calls_at_the_same_time(hq):
    sums, errors = {}, []

    def work(k):
        try:
            s = torch.cuda.Stream() if k % 2 else None
            st = torch.empty(1 << (8 + k), dtype=torch.complex128, device="cuda")
            with torch.cuda.stream(s):
                hq.hq_state_init(st, "+", stream=s)
            for i in range(200):
                v = hq.hq_expectation(st, [(float(k + 1), ((i % 8, "X"),)), (2.0, ((1, "Z"),))], stream=s)
                if abs(v - (k + 1)) > 1e-12:
                    errors.append((k, i, v))
            sums[k] = True
        except Exception as e:  # noqa: BLE001
            errors.append((k, e))

    ts = [threading.Thread(target=work, args=(k,)) for k in range(8)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors and len(sums) == 8
