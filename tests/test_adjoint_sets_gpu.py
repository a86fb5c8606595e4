"""Adjoint gradients where lambda = H phi is formed for several parameter sets
per thread (k_ham with 8 sets in complex64, 4 in complex128), which takes
enough CTAs for every SM: 18 qubits and batches of 75 up, with remainders."""
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


@pytest.mark.parametrize("dt,batch", [("complex64", 76), ("complex64", 83), ("complex64", 80), ("complex128", 41),
                                      ("complex128", 43), ("complex128", 40)])
def test_batches_with_a_remainder(hq, dt, batch):
    """Terms with repeated X masks out of order, Y factors (imaginary weights) and
    the identity; first, middle and last sets against the oracle."""
    n = 18
    circ = C.ansatz(n, 1)
    H = [(0.7, ()), (1.0, ((0, "Z"), (3, "Z"))), (-0.4, ((2, "Z"),)), (0.5, ((1, "X"),)), (0.3, ((1, "Y"),)),
         (-0.8, ((1, "X"), (14, "Z"))), (0.6, ((1, "Y"), (5, "Z"), (16, "Z"))), (0.2, ((0, "Y"), (17, "Y"))),
         (0.9, ((0, "X"), (17, "X"))), (-0.1, ((0, "Y"), (17, "X"))), (0.25, ((16, "X"),)), (0.15, ((0, "Z"),)),
         (0.35, ((1, "Y"), (7, "Y"))), (-0.2, ((1, "X"), (3, "Z")))]
    th = C.ansatz_params(circ.n_params, batch, 11)
    e, g = hq.hq_adjoint_grad(circ, H, th, dtype=dt)
    scale = sum(abs(c) for c, _ in H)
    # complex64: ~100 gates, each rounding the state by a few 2^-24
    tol = (1e-10 if dt == "complex128" else 2e-5) * scale
    for b in sorted({0, 3, 7, 8, batch // 2, batch - 3, batch - 1}):
        we, wg = oracle.adjoint_grad(circ, H, th[b])
        assert abs(e[b] - we) <= tol
        assert np.abs(g[b] - wg).max() <= tol
