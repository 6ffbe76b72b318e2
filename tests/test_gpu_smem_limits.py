"""Kernels with dynamic shared memory serve callers of different sizes at the same time: the limit a call
raises is not lowered by a smaller call on another thread or of another batch."""
import threading

import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns,perm", [((11, 12), 0.0), ((13, 14), 1.0)])
def test_threads_with_states_of_different_sizes(ns, perm):
    """complex128 circuits, fused: one block's work (n <= 12: 68 and 100 KB), and tile passes of other
    sizes. Every call succeeds, and the results are those of a call alone."""
    import torch

    import paper_2411_18354_gb300 as qs

    qs._lib.lib()
    errors = []

    def work(n):
        try:
            torch.cuda.set_device(0)
            gates = W.random_circuit(n, 30, 2, seed=n, perm_fraction=perm)
            with qs.State(n, "c128", stream=0) as st:
                st.apply_circuit(gates, None, qs.QS_FLAG_FUSE)
                want = st.to_numpy()
                for _ in range(1000):
                    st.set_basis(0)
                    st.apply_circuit(gates, None, qs.QS_FLAG_FUSE)
                if not np.array_equal(st.to_numpy(), want):
                    errors.append((n, "different amplitudes"))
        except Exception as e:  # noqa: BLE001 (reported below)
            errors.append((n, str(e)))

    threads = [threading.Thread(target=work, args=(n,)) for n in ns * 2]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors


@pytest.mark.parametrize("dtype,tol", [("c64", 1e-4), ("c128", 1e-9)])
def test_batches_of_different_sizes(dtype, tol):
    """A batch runs after a batch of smaller states has been created."""
    import torch

    import paper_2411_18354_gb300 as qs

    big, small = (10, W.hea_circuit(10, 2), 40), (3, W.hea_circuit(3, 1), 6)
    a = qs.Batch([big[0]], [big[1]], [big[2]], dtype)
    b = qs.Batch([small[0]], [small[1]], [small[2]], dtype)
    for batch, (n, gates, count) in ((a, big), (b, small), (a, big)):
        theta = np.random.default_rng(n).uniform(-3, 3, count)
        th = torch.tensor(theta, device="cuda")
        energy = torch.zeros(1, dtype=torch.float64, device="cuda")
        grad = torch.zeros(count, dtype=torch.float64, device="cuda")
        for flags in (0, qs.QS_FLAG_GRAPH):
            batch.run(th, energy, grad, flags)
            assert abs(energy.item() - oracle.energy(n, gates, theta)) <= tol
    a.close()
    b.close()
