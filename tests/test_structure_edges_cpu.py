"""hq_gate_structure at the edges of its tolerance: entries within a few units
in the last place of 4 FP64 epsilon of the largest magnitude, infinities, NaN,
zero matrices, against a plain restatement with hypot on every entry."""
import math

import numpy as np
import pytest


@pytest.fixture(scope="module")
def hq():
    from paper_2111_06868_gb300 import build
    from paper_2111_06868_gb300 import hq as _hq

    build.build()
    _hq.load()
    return _hq


def restated(k, m):
    K = 1 << k
    mx = 0.0
    for e in m.ravel():
        h = math.hypot(e.real, e.imag)
        mx = h if mx < h else mx
    tiny = 4.0 * 2.220446049250313e-16 * mx
    nz = [[math.hypot(e.real, e.imag) > tiny for e in row] for row in m]
    mono = all(sum(r) == 1 for r in nz) and all(sum(c) == 1 for c in zip(*nz))
    mask = 0
    for j in range(k):
        bit = 1 << (k - 1 - j)
        if all(math.hypot(m[r, c].real - (r == c), m[r, c].imag) <= tiny
               for r in range(K) for c in range(K) if not (r & bit) or not (c & bit)):
            mask |= 1 << j
    return mono, mask


@pytest.mark.parametrize("k", [1, 2, 3, 4])
def test_entries_near_the_tolerance(hq, k):
    rng = np.random.default_rng(k)
    K = 1 << k
    eps = 2.220446049250313e-16
    seen = set()
    for trial in range(400):
        if trial % 2:  # controlled: the identity with a dense lower right corner
            m = np.eye(K, dtype=np.complex128)
            t = K >> int(rng.integers(0, k + 1))
            m[K - t:, K - t:] = (rng.standard_normal((t, t)) + 1j * rng.standard_normal((t, t))) / (1 + t)
        else:
            m = np.diag(np.exp(1j * rng.uniform(0, 6, K)))[rng.permutation(K)]
        top = max(math.hypot(e.real, e.imag) for e in m.ravel())
        for _ in range(int(rng.integers(0, 4))):  # a disturbance of about the tolerance, on or off the diagonal
            r, c = int(rng.integers(K)), int(rng.integers(K))
            size = 4 * eps * top * (1 + float(rng.choice([0, 1e-16, -1e-16, 3e-16, -3e-16, 1e-7, -1e-7, 1, -0.5])))
            ang = float(rng.choice([0, np.pi / 2, rng.uniform(0, 6)]))
            m[r, c] += size * complex(math.cos(ang), math.sin(ang))
        if trial % 29 == 0:
            m[int(rng.integers(K)), int(rng.integers(K))] = complex(*rng.choice([0.0, 1.0, np.inf, np.nan], 2))
        if trial % 97 == 0:
            m[:] = 0
        mono, mask = restated(k, m)
        s, got, _ = hq.hq_gate_structure(m)
        assert bool(s & 2) == mono and got == mask, (trial, m)
        seen.add((mono, mask))
    assert len(seen) >= min(4, 1 + k)
