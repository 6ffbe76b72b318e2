"""complex128 gates in fixed point (csrc/k_fx.cuh) where a result lies just below a power of two: the
conversion to float64 then carries into the next exponent. Rotations undone, powers of two with a tiny
partner, sweeps that return to a basis state.

Bound: 2^-50 of |a||x| + |b||y| for each output of a gate (see test_gpu_fx), that is 2^-49 of the norm of
a pair for unit rows."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

N = 10


@pytest.mark.parametrize("start", ["basis", "uniform"])
@pytest.mark.parametrize("t", [0, 4])
def test_rotation_undone(t, start):
    """RY(a) then RY(-a), two calls: both rows of both matrices, 500 angles and their negatives."""
    import paper_2411_18354_gb300 as qs

    v = np.zeros(1 << N, np.complex128)
    if start == "basis":
        v[0] = 1
    else:
        v[:] = 2.0 ** (-N / 2) * (1 - 1j)
    angles = np.random.default_rng(t).uniform(-np.pi, np.pi, 500)
    with qs.State(N, "c128") as st:
        for a in np.concatenate([angles, [1.1, 1.5, 2.5, -1.1, -1.5, -2.5]]):
            st.from_numpy(v)
            st.apply_gate(t, oracle.ry(a))
            st.apply_gate(t, oracle.ry(-a))
            assert np.max(np.abs(st.to_numpy() - v)) <= 2.0 ** -48 * np.sqrt(2) * np.max(np.abs(v)), a


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("fused", [False, True])
def test_power_of_two_with_a_tiny_partner(sign, fused):
    """[[1, -e], [e, 1]] on (x, y) with x or y a power of two and the other 2^-20 .. 2^-60 of it."""
    import paper_2411_18354_gb300 as qs

    k = np.arange(1 << (N - 1))
    big = np.ldexp(1.0, k % 9 - 4) * np.where(k & 16, -1, 1)
    small = big * np.ldexp(1.0 + k / 511, -20 - k % 41) * np.where(k & 32, -1, 1)
    v = np.empty(1 << N, np.complex128)
    v[0::2] = np.where(k & 64, big, small) + 1j * np.where(k & 128, big, small)
    v[1::2] = np.where(k & 64, small, big) + 1j * np.where(k & 128, small, big)
    for e in np.ldexp([1.0, 1.3, 1.7], [-46, -30, -40]):
        U = np.array([[1.0, -sign * e], [sign * e, 1.0]])
        with qs.State(N, "c128") as st:
            st.from_numpy(v)
            if fused:  # one block's work (k_whole.cu) for two gates and more: exchanges of other qubits
                gates = [W.make_gate(0, U)] + [W.make_gate(q, None, (), kind=W.KIND_X) for q in (3, N - 1)]
                st.apply_circuit(W.gate_list(gates), None, qs.QS_FLAG_FUSE)
            else:
                st.apply_gate(0, U)
            got = st.to_numpy().astype(np.clongdouble)
        if fused:
            got = got[np.arange(1 << N) ^ (1 << 3) ^ (1 << (N - 1))]
        x, y = v[0::2].astype(np.clongdouble), v[1::2].astype(np.clongdouble)
        u = U.astype(np.longdouble)
        for out, a, b in ((got[0::2], u[0, 0], u[0, 1]), (got[1::2], u[1, 0], u[1, 1])):
            for part in (np.real, np.imag):
                size = abs(a) * abs(part(x)) + abs(b) * abs(part(y))
                assert np.all(abs(part(out) - (a * part(x) + b * part(y))) <= 2.0 ** -50 * size)


@pytest.mark.parametrize("fused", [False, True])
def test_sweep_returns_to_the_basis_state(fused):
    """20 gradients: the reverse sweep undoes every gate, so that psi comes back as |0>; each of the
    G gates forward and back adds at most 2^-49 of the norm."""
    import paper_2411_18354_gb300 as qs

    n, layers = 7, 3
    gates = W.hea_circuit(n, layers)
    want = np.zeros(1 << n)
    want[0] = 1
    with qs.State(n, "c128") as st:
        for seed in range(20):
            theta = np.random.default_rng(seed).uniform(-np.pi, np.pi, 2 * n * layers)
            st.set_basis(0)
            e, g = st.adjoint_grad(gates, theta, qs.QS_FLAG_FUSE if fused else 0)
            assert np.linalg.norm(st.to_numpy() - want) <= 2 * len(gates) * 2.0 ** -49, seed
            assert abs(e - oracle.energy(n, gates, theta)) <= 1e-12
            if seed < 3:
                assert np.max(np.abs(g - oracle.param_shift_grad(n, gates, theta))) <= 1e-11
