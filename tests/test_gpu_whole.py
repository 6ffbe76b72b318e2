"""States that fit one block (csrc/k_whole.cu): every size, operation class and control pattern against
the oracle, across chunks of descriptors, as a call, a graph and with new angles.

Bounds: those of the fused circuit tests, complex64 3e-5 and complex128 1e-12 per amplitude of a
normalised state."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

ATOL = {"c64": 3e-5, "c128": 1e-12}


def _gates(n, count, rng):
    out = []
    for i in range(count):
        t = int(rng.integers(0, n))
        others = [q for q in range(n) if q != t]
        c = int(rng.integers(0, n)) if rng.random() < 0.3 else int(rng.integers(0, min(3, n - 1) + 1))
        ctrls = sorted(int(q) for q in rng.choice(others, size=c, replace=False)) if c else []
        vals = [int(b) for b in rng.integers(0, 2, size=c)]
        k = rng.integers(0, 7)
        if k == 0:
            out.append(W.make_gate(t, None, ctrls, vals, kind=W.KIND_X))
        elif k == 1:
            out.append(W.make_gate(t, None, ctrls, vals, kind=W.KIND_RY, param=int(rng.integers(0, 4))))
        elif k == 2:
            out.append(W.make_gate(t, np.diag(np.exp(1j * rng.uniform(0, 6, 2))), ctrls, vals))
        elif k == 3:
            out.append(W.make_gate(t, np.diag([1.0, 1j] if rng.random() < 0.5 else [np.exp(0.3j), 1.0]), ctrls, vals))
        else:
            out.append(W.make_gate(t, W.haar_2x2(rng), ctrls, vals))
    return W.gate_list(out)


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n", range(1, 13))
def test_against_oracle(n, dtype):
    import paper_2411_18354_gb300 as qs

    rng = np.random.default_rng(n)
    for count in (2, 128, 300):  # one chunk of descriptors, exactly one, several
        gates = _gates(n, count, rng)
        for theta in (rng.uniform(0, 6, 4), np.zeros(4)):
            psi = W.random_state(n, count)
            ref = psi.copy()
            oracle.run_circuit(ref, n, gates, theta)
            for flags in (qs.QS_FLAG_FUSE, qs.QS_FLAG_FUSE | qs.QS_FLAG_GRAPH):
                with qs.State(n, dtype) as st:
                    st.from_numpy(psi)
                    st.apply_circuit(gates, theta, flags)
                    got = st.to_numpy()
                assert np.max(np.abs(got - ref)) <= ATOL[dtype], (count, flags)


def test_exchanges_move_bits():
    import paper_2411_18354_gb300 as qs

    n = 11
    gates = W.streaming_circuit(n)
    for dtype in ("c64", "c128"):
        psi = W.random_state(n, 3, np.complex64 if dtype == "c64" else np.complex128)
        with qs.State(n, dtype) as st:
            st.from_numpy(psi)
            st.apply_circuit(gates, flags=qs.QS_FLAG_FUSE)
            assert np.array_equal(st.to_numpy(), np.roll(psi, -1))
