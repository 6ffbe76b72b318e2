"""complex128 gates in fixed point (csrc/k_fx.cuh), part by part: a real or imaginary part far below its
partner, in an entry (small phases, near-real matrices) or in an amplitude, keeps its digits.

Bound: 2^-50 of S for each part of an output, S the sum of the magnitudes of its four real products. The
fixed-point forms lose at most 2^-51.8 of S and round once (2^-53); float64 arithmetic rounds four times."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

N = 10


def _rx(a):
    return np.array([[np.cos(a / 2), -1j * np.sin(a / 2)], [-1j * np.sin(a / 2), np.cos(a / 2)]])


MATRICES = {f"phase_{p:g}": np.diag([1.0, np.exp(1j * p)]) for p in (0.9, 0.13, 0.12, 1e-2, 1e-9, 1e-12, np.pi - 1e-7)}
MATRICES.update({f"rz_{p:g}": np.diag([np.exp(-0.5j * p), np.exp(0.5j * p)]) for p in (1.0, 0.1, 1e-8)})
MATRICES.update({f"rx_{a:g}": _rx(a) for a in (1.0, 1e-6, 3.1415)})
MATRICES.update({f"haar_{s}": W.haar_2x2(np.random.default_rng(s)) for s in range(8)})
MATRICES["near_real"] = np.exp(1e-11j) * np.array([[0.6, -0.8], [0.8, 0.6]])
MATRICES["near_hadamard"] = W.H_MATRIX * np.exp(1j * np.array([[1e-9, -2e-6], [3e-12, 1e-4]]))
MATRICES["alike"] = np.array([[0.5 + 0.5j, 0.4 - 0.6j], [-0.3 + 0.7j, 0.1 - 0.45j]])


def _amplitudes(kind, rng):
    re, im = rng.standard_normal((2, 1 << N))
    if kind == "real":
        im[:] = 0
    elif kind == "small_parts":
        re, im = re * 2.0 ** -rng.integers(0, 60, 1 << N), im * 2.0 ** -rng.integers(0, 60, 1 << N)
    elif kind == "far_parts":  # beyond what one scale could hold, and where float64 arithmetic takes over
        re, im = (v * 2.0 ** rng.choice([0, -40, -300, -760, -790, -1000], 1 << N) for v in (re, im))
    return re + 1j * im


def _check(v, got, U, t):
    k = np.arange(1 << N)
    lo = k[(k >> t) & 1 == 0]
    hi = lo | (1 << t)
    u = U.astype(np.clongdouble)
    x = [v[lo].real, v[lo].imag, v[hi].real, v[hi].imag]
    x = [p.astype(np.longdouble) for p in x]
    for row, out in ((0, got[lo]), (1, got[hi])):
        (ar, ai), (br, bi) = ((z.real, z.imag) for z in u[row])
        for part, c in ((out.real, (ar, -ai, br, -bi)), (out.imag, (ai, ar, bi, br))):
            exact = sum(a * b for a, b in zip(c, x))
            size = sum(abs(a * b) for a, b in zip(c, x))
            err = abs(part.astype(np.longdouble) - exact)
            # (4e-323: roundings of subnormal results and products)
            assert np.all(err <= 2.0 ** -50 * size + 4e-323), float(np.max(err / (size + 1e-300)))


@pytest.mark.parametrize("kind", ["plain", "real", "small_parts", "far_parts"])
@pytest.mark.parametrize("name", list(MATRICES))
def test_every_part(name, kind):
    import paper_2411_18354_gb300 as qs

    U = np.asarray(MATRICES[name], dtype=np.complex128)
    rng = np.random.default_rng([list(MATRICES).index(name), len(kind)])
    for t in (0, 6):
        v = _amplitudes(kind, rng)
        with qs.State(N, "c128") as st:
            st.from_numpy(v)
            st.apply_gate(t, U)
            got = st.to_numpy()
            st.from_numpy(v)
            st.apply_gate_masked(t, U, 0)
            assert np.array_equal(got, st.to_numpy())
            _check(v, got, U, t)
            # the same gate as one block's work (k_whole.cu), with two exchanges of other qubits
            gates = [W.make_gate(t, U)] + [W.make_gate(q, None, (), kind=W.KIND_X) for q in (3, N - 1)]
            st.from_numpy(v)
            st.apply_circuit(W.gate_list(gates), None, qs.QS_FLAG_FUSE)
            assert np.array_equal(st.to_numpy()[np.arange(1 << N) ^ (1 << 3) ^ (1 << (N - 1))], got)


def test_many_small_phases_add_up():
    """20000 gates diag(1, e^{i 1e-9}): each leaves at most 2^-50 of the phase so far, 2e-11 in all."""
    import paper_2411_18354_gb300 as qs

    phi, count = 1e-9, 20000
    U = np.diag([1.0, np.exp(1j * phi)])
    with qs.State(3, "c128") as st:
        st.from_numpy(np.array([0, 0, 1, 0, 0, 0, 0, 0], np.complex128))
        for _ in range(count):
            st.apply_gate(1, U)
        z = st.to_numpy()[2]
    assert abs(np.angle(z) - count * phi) <= count * 2.0 ** -50 * count * phi


def test_small_angle_gradient_keeps_its_digits():
    """dE/dtheta of RY(theta) RZ(phi) on one qubit, theta tiny: E = cos theta, dE/dtheta = -sin theta, taken
    through every un-apply; four gates leave at most 4 * 2^-49 of it."""
    import paper_2411_18354_gb300 as qs

    gates = W.gate_list([W.make_gate(0, None, (), kind=W.KIND_RZ, param=0), W.make_gate(0, None, (), kind=W.KIND_RY, param=1),
                         W.make_gate(0, None, (), kind=W.KIND_RZ, param=2), W.make_gate(1, None, (), kind=W.KIND_RZ, param=3)])
    for theta in (1e-6, 1e-10):
        th = np.array([0.7, theta, 1e-7, 1e-9])
        with qs.State(2, "c128") as st:
            e, g = st.adjoint_grad(gates, th)
        assert abs(e - (1 + np.cos(theta))) <= 1e-15
        assert abs(g[1] + np.sin(theta)) <= 4 * 2.0 ** -49 * np.sin(theta)
