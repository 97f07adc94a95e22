"""The merge launch of queries over 1 to 64 subcircuits: which descriptor a
block belongs to is found by a lane per descriptor, in two halves of 32.
Unconnected subcircuits, so that the bins are products of small integers."""
import numpy as np
import pytest

import oracle as O
from synthetic import workloads as W
from synthetic.circuits import chain_line_circuit

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 34, 63, 64])
def test_many_subcircuits(n):
    import torch
    from paper_2207_00933_gb300 import Context, _build
    _build.build()
    widths = [4 + i % 3 for i in range(n)]
    c = chain_line_circuit(n, widths, [0] * (n - 1), 1)
    rng = np.random.default_rng(n)
    probs = []
    for w in widths:
        p = np.zeros((1, 1 << w), dtype=np.float32)
        p[0, rng.integers(1 << w)] = 1
        probs.append(p)
    open_ones = sorted({0, n // 2, min(n - 1, 32), n - 1})
    for i in open_ones:
        probs[i][:] = rng.integers(0, 4, probs[i].shape)
    roles = W.lowest_active_roles(c, [3 if i in open_ones else 0 for i in range(n)])
    g = O.Graph.from_arrays(c.n_qubits, *c.graph_arrays())
    want = O.reconstruct_pairwise(g, O.subcircuit_tensors(g, [p.astype(np.float64) for p in probs], roles), roles)
    with Context(0) as ctx:
        cid = ctx.load_subcircuit_outputs(c.n_qubits, *c.graph_arrays(), [torch.from_numpy(p).cuda() for p in probs])
        qid, na = ctx.set_qubit_roles(cid, roles)
        out = torch.full((1 << na,), float("nan"), dtype=torch.float64, device="cuda")
        ctx.reconstruct(qid, out)
        torch.cuda.synchronize()
        assert want.max() > 0 and np.array_equal(out.cpu().numpy(), want)
