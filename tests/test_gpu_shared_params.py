"""Gradients of circuits whose gates share parameters: one parameter per gate, two, three and all gates on
one, against the oracle's sum of two-term shifts (each gate shifted by itself)."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


def _circuit(n, layers, owner):
    """RY and RZ on every qubit, CNOT ladders; rotation k takes parameter owner(k)."""
    gates, k = [], 0
    for _ in range(layers):
        for q in range(n):
            for kind in (W.KIND_RY, W.KIND_RZ):
                gates.append(W.make_gate(q, None, (), kind=kind, param=owner(k)))
                k += 1
        gates += [W.make_gate(q + 1, None, (q,), kind=W.KIND_X) for q in range(n - 1)]
    return W.gate_list(gates), k


@pytest.mark.parametrize("dtype,tol", [("c64", 2e-4), ("c128", 1e-9)])
@pytest.mark.parametrize("share", [1, 2, 3, 1000])
def test_shared_parameters(share, dtype, tol):
    import paper_2411_18354_gb300 as qs

    n, layers = 5, 4
    gates, count = _circuit(n, layers, lambda k: k // share)
    apart, _ = _circuit(n, layers, lambda k: k)
    theta = np.random.default_rng(share).uniform(-2, 2, (count + share - 1) // share)
    every = theta[np.arange(count) // share]
    want = np.bincount(np.arange(count) // share, oracle.param_shift_grad(n, apart, every))
    for flags in (0, qs.QS_FLAG_FUSE, qs.QS_FLAG_FUSE | qs.QS_FLAG_JIT):
        with qs.State(n, dtype) as st:
            e, g = st.adjoint_grad(gates, theta, flags)
        assert abs(e - oracle.energy(n, apart, every)) <= tol
        assert np.max(np.abs(g - want)) <= tol
