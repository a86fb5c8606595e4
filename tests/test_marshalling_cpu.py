"""Gate and channel lists into the C structs: every form of a qubit index that
int() takes, the same struct as one field at a time."""
import numpy as np
import pytest

from paper_2111_06868_gb300 import circuits as C
from paper_2111_06868_gb300 import hq


class Label:
    def __int__(self):
        return 3


torch = pytest.importorskip("torch")
FORMS = [3, np.int64(3), np.uint8(3), np.array(3), np.float64(3.0), np.array(3.0), torch.tensor(3), torch.tensor(3.0),
         3.0, "3", Label(), True]


@pytest.mark.parametrize("q", FORMS, ids=[type(f).__name__ + str(i) for i, f in enumerate(FORMS)])
def test_qubit_forms(q):
    keep = []
    U = C.random_unitary(2, C.SplitMix64(1))
    arr, G = hq._gates_array([((q, 7), U), ((0,), C.hadamard())], keep)
    assert G == 2 and arr[0].k == 2 and list(arr[0].qubits[:2]) == [int(q), 7]
    assert np.array_equal(np.ctypeslib.as_array((hq.ctypes.c_double * 32).from_address(arr[0].matrix)),
                          U.ravel().view(np.float64))


@pytest.mark.parametrize("q", FORMS, ids=[type(f).__name__ + str(i) for i, f in enumerate(FORMS)])
def test_qubit_forms_of_a_noisy_circuit(q, monkeypatch):
    """The structs that hq_run_trajectory hands to the library."""
    seen = {}

    class Lib:
        def hq_run_trajectory(self, ptr, n, dt, arr, nops, *rest):
            seen["ops"] = [(o.k, list(o.qubits[: o.k]), o.nkraus) for o in arr[:nops]]
            return 0

    monkeypatch.setattr(hq, "load", lambda: Lib())
    monkeypatch.setattr(hq, "_state_args", lambda st: (None, 8, 0))
    monkeypatch.setattr(hq, "_stream", lambda st: None)
    hq.hq_run_trajectory(None, [("gate", (q, 5), C.cz()), ("kraus", (q,), C.amplitude_damping(0.1))], np.zeros(1))
    assert seen["ops"] == [(2, [int(q), 5], 0), (1, [int(q)], len(C.amplitude_damping(0.1)))]
