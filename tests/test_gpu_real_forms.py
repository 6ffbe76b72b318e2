"""Compiled passes that divide out the larger entry of rotations and reflections (csrc/qs_jit.cu,
real_forms): many per pass, angles on both sides of pi / 2, scaled matrices, controls in between,
against the oracle.

Bound: each gate rounds at most four times per part, 4 * 2^-24 (2^-53) of the pair's norm, so G
gates of the circuit leave at most 8 G u of the state's norm in the 2-norm."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


def _circuit(n, rng, scaled):
    gates = []
    p = 0
    for layer in range(6):
        for q in range(n):
            kind = rng.integers(0, 4)
            if kind == 0:
                gates.append(W.make_gate(q, W.H_MATRIX))
            elif kind == 1:
                a = rng.uniform(0, 2 * np.pi)
                f = 2.0 ** rng.integers(-3, 4) if scaled else 1.0
                gates.append(W.make_gate(q, f * np.array([[np.cos(a), np.sin(a)], [np.sin(a), -np.cos(a)]])))
            else:
                gates.append(W.make_gate(q, None, (), kind=W.KIND_RY, param=p))
                p += 1
                gates.append(W.make_gate(q, None, (), kind=W.KIND_RZ, param=p))
                p += 1
        a, b = (int(v) for v in rng.choice(n, 2, replace=False))
        gates.append(W.make_gate(a, np.array([[0.6, -0.8], [0.8, 0.6]]), (b,)))
        gates.append(W.make_gate(b, None, (a,), kind=W.KIND_X))
    return W.gate_list(gates), rng.uniform(0, 2 * np.pi, p)


@pytest.mark.parametrize("dtype,u", [("c64", 2.0 ** -24), ("c128", 2.0 ** -53)])
@pytest.mark.parametrize("n,scaled", [(5, False), (9, True), (14, False), (14, True)])
def test_forward(n, scaled, dtype, u):
    import paper_2411_18354_gb300 as qs

    rng = np.random.default_rng([n, scaled])
    gates, theta = _circuit(n, rng, scaled)
    psi = W.random_state(n, 5)
    with qs.State(n, dtype) as st:
        st.from_numpy(psi)
        st.apply_circuit(gates, theta, qs.QS_FLAG_FUSE | qs.QS_FLAG_JIT)
        got = st.to_numpy().astype(np.complex128)
    ref = psi.astype(np.complex64 if dtype == "c64" else np.complex128).astype(np.complex128)
    oracle.run_circuit(ref, n, gates, theta)
    assert np.linalg.norm(got - ref) <= 8 * len(gates) * u * np.linalg.norm(ref)


@pytest.mark.parametrize("dtype,tol", [("c64", 1e-4), ("c128", 1e-9)])
def test_gradient(dtype, tol):
    """Against the two-term parameter shift (rotations only uncontrolled; unitary gates)."""
    import paper_2411_18354_gb300 as qs

    n = 6
    gates, theta = _circuit(n, np.random.default_rng(8), False)
    with qs.State(n, dtype) as st:
        e, g = st.adjoint_grad(gates, theta, qs.QS_FLAG_FUSE | qs.QS_FLAG_JIT)
        back = st.to_numpy()
    assert abs(e - oracle.energy(n, gates, theta)) <= tol
    assert np.max(np.abs(g - oracle.param_shift_grad(n, gates, theta))) <= tol
    want = np.zeros(1 << n)
    want[0] = 1
    assert np.max(np.abs(back - want)) <= tol
