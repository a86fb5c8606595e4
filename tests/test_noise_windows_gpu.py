"""State-dependent channels two at a time (k_window) where small states do not
reach: sums outside FP32's range, many CTAs, several groups per thread."""
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


def sampled(psi, n, qubits, kraus, u):
    """One sampled Kraus operator, as the noise oracle's step, every operator
    applied as a gate (its dense 2^n x 2^n form does not fit at these sizes)."""
    outs = [oracle.apply_gate(psi.copy(), n, qubits, K) for K in kraus]
    p = np.array([np.vdot(o, o).real for o in outs])
    i = min(int(np.searchsorted(np.cumsum(p), u * p.sum(), side="right")), len(kraus) - 1)
    return i, outs[i] / np.sqrt(p[i])


@pytest.mark.parametrize("dtype", ["complex64", "complex128"])
@pytest.mark.parametrize("n", [15, 17, 19, 22])
def test_chains_over_many_ctas(hq, n, dtype):
    """Several CTAs' rows joined (15 qubits up), two-channel windows that feed the
    next window through the alternating sets of sums, several groups per
    thread through the three-stage ring (22 qubits), a two-qubit channel,
    lowest and highest bits, an applied gate in between: the oracle's branches
    and state."""
    rng = np.random.default_rng(n)  # input only
    sm = C.SplitMix64(n)
    order = [0, n - 1, 1, n - 2, n // 2, 2, n - 3, n // 2 + 1]
    ops = []
    for i, q in enumerate(order):
        if i % 3 == 0:
            ops.append(("gate", (q,), C.random_unitary(1, sm)))
        ops.append(("kraus", (q,), C.amplitude_damping(0.4, 0.2)))
    ops.append(("gate", (n - 1, 0), C.fsim(0.5, 0.4)))
    ops.append(("kraus", (n - 1, 0), [np.kron(a, b) for a in C.amplitude_damping(0.3) for b in C.amplitude_damping(0.2)]))
    ops += [("kraus", (q,), C.amplitude_damping(0.3)) for q in (3, n - 4, n - 1)]
    u = rng.random(sum(1 for o in ops if o[0] == "kraus"))
    tokens = "".join("+-"[int(x)] for x in rng.integers(0, 2, n))
    psi, want, c = oracle.state_init(n, tokens), [], 0
    for kind, qs, m in ops:
        if kind == "gate":
            psi = oracle.apply_gate(psi, n, qs, m)
        else:
            i, psi = sampled(psi, n, qs, m, u[c])
            want.append(i)
            c += 1
    st = torch.empty(1 << n, dtype=getattr(torch, dtype), device="cuda")
    hq.hq_state_init(st, tokens)
    got = hq.hq_run_trajectory(st, ops, u)
    assert got.tolist() == want
    # complex64: 16 operators, each rounding the state by a few 2^-24
    err = np.linalg.norm(st.cpu().numpy().astype(np.complex128) - psi)
    assert err <= (1e-12 if dtype == "complex128" else 4e-6)
