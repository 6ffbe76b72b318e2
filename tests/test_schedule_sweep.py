"""The reverse sweep in qs_circuit_schedule (host only): launches, bytes and operations of the gradient of an
ansatz as qs_adjoint_grad issues it."""
import pytest

import workloads as W


@pytest.fixture(scope="module")
def qs():
    import paper_2411_18354_gb300 as q

    q.build()
    return q


@pytest.mark.parametrize("dtype,size", [("c64", 8), ("c128", 16)])
@pytest.mark.parametrize("n,layers", [(6, 1), (6, 3), (13, 2)])
def test_unfused_ansatz_gradient(qs, n, layers, dtype, size):
    """RZ and RY of a qubit un-apply in one launch, one-sided and real, except the first un-applied RZ,
    which keeps both sides and runs apart; CNOTs touch half of both vectors."""
    state = size * 2.0**n
    s = qs.circuit_schedule(n, W.hea_circuit(n, layers), W.hea_params(n, layers, seed=1),
                            flags=qs.QS_FLAG_ADJOINT, dtype=dtype)
    merged, cnots, joined = layers * n, layers * (n - 1), layers * n - 1
    assert s["single_gates"] == merged + cnots + joined + 2 + cnots
    # complex64: energy and lambda in one kernel; complex128: reduction (two kernels above one tile), the
    # sum, lambda. One kernel of gradient sums.
    tail = 2 if dtype == "c64" else (1 if n < 12 else 2) + 3
    assert s["launches"] == s["single_gates"] + tail
    forward = 2 * state * (merged + 0.5 * cnots)
    sweep = 2 * 2 * state * (joined + 2 + 0.5 * cnots)
    assert s["algorithmic_bytes"] == forward + sweep + (2 if dtype == "c64" else 3) * state
    pairs = 2.0 ** (n - 1)
    # forward: a general product; un-apply of two vectors; derivative products 8, one-sided 4
    flops = pairs * (28 * merged + 2 * (12 * layers * n + 6 * joined + 12) + 8 * layers * n + 4 * joined + 8) + 16 * pairs
    assert s["algorithmic_flops"] == flops


@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_shared_parameters_take_one_launch_more(qs, dtype):
    """Rows of a parameter with more than two gates are summed in a launch of their own."""
    def circuit(owner):
        return W.gate_list([W.make_gate(q, None, (), kind=W.KIND_RY, param=owner(q)) for q in range(5)])

    theta = [0.3] * 5
    flags = qs.QS_FLAG_ADJOINT
    apart = qs.circuit_schedule(5, circuit(lambda q: q), theta, flags=flags, dtype=dtype)
    two = qs.circuit_schedule(5, circuit(lambda q: q // 2), theta, flags=flags, dtype=dtype)
    one = qs.circuit_schedule(5, circuit(lambda q: 0), theta, flags=flags, dtype=dtype)
    assert apart["launches"] == two["launches"] == one["launches"] - 1


def test_fused_sweep_counts_joined_steps_once(qs):
    """complex128 rotations run alone (forward merged, one sweep launch a qubit and layer and one more) and
    exchanges in passes, except a few of the 2 * 19 a layer."""
    n, layers = 20, 8
    s = qs.circuit_schedule(n, W.hea_circuit(n, layers), W.hea_params(n, layers, seed=1),
                            flags=qs.QS_FLAG_ADJOINT | qs.QS_FLAG_FUSE, dtype="c128")
    rotations = 2 * layers * n + 1
    assert rotations <= s["single_gates"] < rotations + layers * (n - 1)
    assert s["launches"] == s["single_gates"] + s["tile_passes"] + s["diag_runs"] + 5
