"""The two paths of one batch, run in turn: each plans for itself (the compiled one on its first run), the
answers agree, and the bytes reported are those of the path that ran."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_bytes_are_those_of_the_path_that_ran():
    """RY and RZ on two qubits of a state larger than a tile, two gates to a pass. Persistent kernel: RY RZ
    merge, one forward pass, two sweep passes. Compiled: two of each. Three vectors beside the passes."""
    import torch

    import paper_2411_18354_gb300 as qs

    gates = W.gate_list([W.make_gate(q, None, (), kind=k, param=2 * q + (k == W.KIND_RZ))
                         for q in (0, 1) for k in (W.KIND_RY, W.KIND_RZ)])
    b = qs.Batch([6, 6], [gates] * 2, [4, 4], "c64", small_bits=5, tile_bits=5, max_pass_gates=2)
    vector = 2 * (1 << 6) * 8
    theta = torch.tensor(np.linspace(0.1, 2.0, 8), device="cuda")
    out = []
    assert b.algorithmic_bytes() == (3 + 2 + 2 * 4) * vector
    for flags, passes in ((0, 2 + 2 * 4), (qs.QS_FLAG_JIT, 2 * 2 + 2 * 4), (qs.QS_FLAG_GRAPH, 2 + 2 * 4),
                          (qs.QS_FLAG_GRAPH | qs.QS_FLAG_JIT, 2 * 2 + 2 * 4)):
        energy = torch.zeros(2, dtype=torch.float64, device="cuda")
        grad = torch.zeros(8, dtype=torch.float64, device="cuda")
        b.run(theta, energy, grad, flags)
        torch.cuda.synchronize()
        assert b.algorithmic_bytes() == (3 + passes) * vector
        out.append(np.concatenate([energy.cpu().numpy(), grad.cpu().numpy()]))
    b.close()
    for o in out[1:]:
        assert np.max(np.abs(o - out[0])) <= 1e-5
