"""Host allocations that fail inside a gate list: HQ_ERR_ALLOC, and the state
is what some prefix of the list leaves.  A child process loads a small library
whose operator new throws std::bad_alloc after a set number of calls."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdlib>
#include <new>
static thread_local long left = -1;  // calls that still succeed; -1: all
extern "C" void fail_after(long n) { left = n; }
static void *get(std::size_t n, std::size_t al)
{
    if (left == 0) throw std::bad_alloc();
    if (left > 0) --left;
    void *p = nullptr;
    if (posix_memalign(&p, al < 16 ? 16 : al, n ? n : 1)) throw std::bad_alloc();
    return p;
}
void *operator new(std::size_t n) { return get(n, 16); }
void *operator new(std::size_t n, std::align_val_t a) { return get(n, std::size_t(a)); }
void operator delete(void *p) noexcept { std::free(p); }
void operator delete(void *p, std::size_t) noexcept { std::free(p); }
void operator delete(void *p, std::align_val_t) noexcept { std::free(p); }
void operator delete(void *p, std::size_t, std::align_val_t) noexcept { std::free(p); }
"""

CHILD = r"""
import ctypes, sys
alloc = ctypes.CDLL(sys.argv[1], mode=ctypes.RTLD_GLOBAL)  # before the library whose operator new it takes
sys.path.insert(0, sys.argv[2])
n, dt = int(sys.argv[3]), sys.argv[4]
import numpy as np, torch
from paper_2111_06868_gb300 import hq, circuits as C
sm, rng = C.SplitMix64(3), np.random.default_rng(3)
def narrow(count):
    g = []
    for _ in range(count):
        k = int(rng.choice([1, 1, 2, 2, 3] if dt == "complex64" else [1, 1, 2]))
        U = C.random_unitary(k, sm) if rng.uniform() < 0.8 else np.diag(np.exp(1j * rng.uniform(0, 6, 1 << k)))
        g.append(C.Gate("a", tuple(int(q) for q in rng.choice(n, k, replace=False)), U))
    return g
wide = C.Gate("w", (0, 3, 1, n - 1, 5), C.random_unitary(5, sm))
gates = narrow(60) + [wide] + narrow(60)
keep = []
arr, G = hq._gates_array(gates, keep)
lib = hq.load()
start = torch.randn(1 << n, dtype=getattr(torch, dt), device="cuda")
prefix = [start.clone()]
for g in gates:
    prefix.append(prefix[-1].clone())
    hq.hq_apply_gate(prefix[-1], g.qubits, g.matrix)
prefix = torch.stack(prefix)
top = float(torch.linalg.norm(start))
def run(left):
    st = start.clone()
    torch.cuda.synchronize()
    alloc.fail_after(ctypes.c_long(left))
    rc = lib.hq_apply_blocks(ctypes.c_void_p(st.data_ptr()), n, hq._dtype_code(st), arr, G, None, None)
    alloc.fail_after(ctypes.c_long(-1))
    err = torch.linalg.norm(prefix - st, dim=1) / top
    return rc, int(err.argmin()), float(err.min())
assert run(-1)[:2] == (0, G)
failures = set()
for left in range(100000):
    rc, at, err = run(left)
    assert rc in (0, -7), rc
    # 121 gates, each rounding the state by a few 2^-24 (2^-53)
    assert err <= (2e-5 if dt == "complex64" else 1e-12), (left, rc, at, err)
    if rc == 0:
        assert at == G
        break
    failures.add(at)
print("failed", left, "times, after gates", sorted(failures))
assert left > 0 and failures <= {0, 60, 61}, failures
"""


@pytest.mark.parametrize("n,dt", [(12, "complex64"), (12, "complex128"), (23, "complex64")])
def test_a_failed_plan_leaves_a_prefix(tmp_path, n, dt):
    src, lib = tmp_path / "failnew.cpp", tmp_path / "failnew.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", str(src), "-o", str(lib)], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD, str(lib), ROOT, str(n), dt], capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
