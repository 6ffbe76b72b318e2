"""complex128 gates in fixed point (csrc/k_fx.cuh): every form and its edges against extended
precision, per pair.

Bound: 2^-50 of |a||x| + |b||y| for each output. The fixed-point forms lose at most 2^-51.9 of it
and round once (2^-53 per part); float64 arithmetic, which out-of-range pairs take, rounds each part
four times, at most 2^-51 per part."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

N = 11
H, S = 0.5, np.sqrt(0.75)
MATRICES = {
    "balanced": W.haar_2x2(np.random.default_rng(3)),
    "wide": np.array([[np.cos(1e-5) * np.exp(0.3j), -1j * np.sin(1e-5)], [1j * np.sin(1e-5), np.cos(1e-5)]]),
    "wide_rows": np.array([[1e10 + 2j, 3e-12 - 1e-9j], [1e-9j, 5.0 - 1e-12j]]),
    "zero_entry": np.array([[0, -1j], [1j, 0]]),
    "triangular": np.array([[0.5 + 1j, 0], [1e-9j, 2.0]]),
    "huge": np.array([[1e60j, 1.0], [1.0, 1e-60j]]),
    "real": np.array([[H, -S], [S, H]]),
    "real_small": np.array([[1.0, -1e-14], [1e-14, 1.0]]),
    "real_monomial": np.array([[0, -1.0], [1.0, 0]]),
    "diag": np.diag(np.exp([0.7j, -1.1j])),
    "diag_z": np.diag([2.0, -1.0]),
    "side": np.diag([1.0, np.exp(0.2j)]),
    "side_lo": np.diag([1e-3 + 2j, 1.0]),
}


def _amplitudes(kind, rng):
    v = rng.standard_normal(1 << N) + 1j * rng.standard_normal(1 << N)
    if kind == "zeros":  # whole pairs, one side, one part
        v[rng.random(1 << N) < 0.5] = 0
        v.real[rng.random(1 << N) < 0.2] = 0
    elif kind == "spread":  # 2^-120 .. 2^120, each part its own
        v = v.real * 2.0 ** rng.integers(-120, 121, 1 << N) + 1j * v.imag * 2.0 ** rng.integers(-120, 121, 1 << N)
    elif kind == "edges":  # around the exponents where float64 arithmetic takes over, and subnormals
        e = rng.choice([-1060, -1022, -960, -769, -768, -767, -766, -765, -400, 0, 700, 765, 766, 767, 768], 1 << N)
        v = np.ldexp(v.real, e) + 1j * np.ldexp(v.imag, e)
    return v


@pytest.mark.parametrize("kind", ["plain", "zeros", "spread", "edges"])
@pytest.mark.parametrize("name", list(MATRICES))
def test_forms_against_extended_precision(name, kind):
    import paper_2411_18354_gb300 as qs

    U = np.asarray(MATRICES[name], dtype=np.complex128)
    rng = np.random.default_rng([list(MATRICES).index(name), len(kind)])
    for t, mask in ((0, 0), (0, 0b10010), (5, 0), (N - 1, 0b11), (3, 0b1100000100)):
        v = _amplitudes(kind, rng)
        with qs.State(N, "c128") as st, qs.State(N, "c128") as sm:
            st.from_numpy(v)
            sm.from_numpy(v)
            st.apply_gate(t, U, mask)
            sm.apply_gate_masked(t, U, mask)
            got, got_masked = st.to_numpy(), sm.to_numpy()
        assert np.array_equal(got, got_masked)
        k = np.arange(1 << N)
        lo = k[((k >> t) & 1 == 0) & (k & mask == mask)]
        hi = lo | (1 << t)
        touched = np.zeros(1 << N, bool)
        touched[lo] = touched[hi] = True
        assert np.array_equal(got[~touched], v[~touched])
        x, y = v[lo].astype(np.clongdouble), v[hi].astype(np.clongdouble)
        u = U.astype(np.clongdouble)
        for out, a, b in ((got[lo], u[0, 0], u[0, 1]), (got[hi], u[1, 0], u[1, 1])):
            size = abs(a) * abs(x) + abs(b) * abs(y)
            err = abs(out.astype(np.clongdouble) - (a * x + b * y))
            # (5e-324 * 8: roundings of subnormal results and products)
            fine = np.isfinite(np.float64(size)) & (size < 1e308)
            assert np.all(err[fine] <= 2.0 ** -50 * size[fine] + 4e-323), (t, mask, float(np.max(err[fine] / (size[fine] + 1e-300))))


def test_infinities_and_nan_stay_in_their_pairs():
    import paper_2411_18354_gb300 as qs

    v = np.random.default_rng(1).standard_normal(1 << N) + 0.5j
    v[4], v[9], v[300] = np.inf, np.nan, -np.inf * 1j
    for U in (MATRICES["balanced"], MATRICES["wide"], MATRICES["real"], MATRICES["diag"]):
        for t in (0, 4):
            with qs.State(N, "c128") as st:
                st.from_numpy(v)
                st.apply_gate(t, U)
                got = st.to_numpy()
            bad = np.zeros(1 << N, bool)
            for k in (4, 9, 300):
                bad[k] = bad[k ^ (1 << t)] = True
            assert np.all(np.isfinite(got[~bad]))
            assert not np.any(np.isfinite(got[[4, 9, 300]]))


@pytest.mark.parametrize("n", [12, 13, 16])
@pytest.mark.parametrize("kind", ["plain", "zeros", "spread", "small", "tiny"])
def test_expect_z_integer_sums(n, kind):
    """<Z_i> of complex128 with 16 values per thread summed as integers. Bound 2^-47 of the norm: each
    value loses at most 2^-54 of its thread's largest (16 of them: 2^-50 of that thread's sum), and the
    float64 additions above round at most 2^6 times along any path."""
    import paper_2411_18354_gb300 as qs

    rng = np.random.default_rng([n, len(kind)])
    v = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    if kind == "zeros":
        v[rng.random(1 << n) < 0.9] = 0
    elif kind == "spread":
        v *= 2.0 ** rng.integers(-60, 61, 1 << n)
    elif kind == "small":  # around the exponents where float64 squares take over
        v *= 2.0 ** rng.integers(-440, -400, 1 << n)
    elif kind == "tiny":
        v *= 2.0 ** -500
    with qs.State(n, "c128") as st:
        st.from_numpy(v)
        z, norm2 = st.expect_z()
    p = v.real.astype(np.longdouble) ** 2 + v.imag.astype(np.longdouble) ** 2
    k = np.arange(1 << n)
    total = p.sum()
    assert abs(norm2 - total) <= 2.0 ** -47 * total
    for q in range(n):
        assert abs(z[q] - (p * (1 - 2 * ((k >> q) & 1))).sum()) <= 2.0 ** -47 * total


@pytest.mark.parametrize("n", [24, 25, 26, 27])
def test_expect_z_runs_of_tiles(n):
    """Runs of 1, 2, 4, 8 tiles: basis states whose bits differ in and around the run's tile bits."""
    import paper_2411_18354_gb300 as qs

    with qs.State(n, "c128") as st:
        for k in (0, 1 << 12, 5 << 13, 3 << 15, (1 << n) - 1, (1 << (n - 1)) | 0x5A5A):
            st.set_basis(k)
            z, norm2 = st.expect_z()
            assert norm2 == 1.0
            assert np.array_equal(z, np.array([1.0 - 2.0 * ((k >> i) & 1) for i in range(n)]))
