"""The probability check of a contraction step at sizes between two tile
shapes.  The outputs are integers below 2^20 that only the I labels of the cut
edges carry: FP32 sums of 16 bins are exact, those of 64 are not.  A step too
small for 128 x 128 tiles adds at most 16 bins in FP32, so its FP64 sum must be
exact."""
import numpy as np
import pytest

import oracle as O
from synthetic import workloads as W
from synthetic.circuits import chain_line_circuit

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths,cut,active,shape", [
    ([14, 10], 3, [11, 10], (1024, 2048, 64)),
    ([13, 11], 3, [10, 11], (1024, 2048, 64)),
    ([18, 7], 4, [14, 7], (128, 16384, 256)),
    ([13, 10], 3, [10, 10], (1024, 1024, 64)),
    ([13, 10], 2, [11, 10], (1024, 2048, 16)),
])
def test_exact_total(widths, cut, active, shape):
    import torch
    from paper_2207_00933_gb300 import Context, _build
    _build.build()
    c = chain_line_circuit(3, widths, [cut], 1)
    rng = np.random.default_rng(3)
    up = rng.integers(800 >> cut, 1000 >> cut, (4 ** cut, 1 << widths[0])).astype(np.float32)
    down = np.tile(rng.integers(900, 1001, 1 << widths[1]).astype(np.float32), (4 ** cut, 1))
    roles = W.lowest_active_roles(c, active)
    g = O.Graph.from_arrays(c.n_qubits, *c.graph_arrays())
    ref = O.reconstruct_pairwise(g, O.subcircuit_tensors(g, [up.astype(np.float64), down.astype(np.float64)], roles), roles)
    assert np.array_equal(ref, np.rint(ref)) and 2 ** 18 < ref.min() and ref.max() < 2 ** 20
    with Context(0) as ctx:
        cid = ctx.load_subcircuit_outputs(c.n_qubits, *c.graph_arrays(), [torch.from_numpy(p).cuda() for p in (up, down)])
        qid, na = ctx.set_qubit_roles(cid, roles)
        assert tuple(sorted(ctx.query_steps(qid)[-1][:2])) + ctx.query_steps(qid)[-1][2:] == shape
        out = torch.empty(1 << na, dtype=torch.float32, device="cuda")
        tot = torch.zeros(1, dtype=torch.float64, device="cuda")
        ctx.reconstruct(qid, out, "fp32", tot)
        torch.cuda.synchronize()
        assert np.array_equal(out.double().cpu().numpy(), ref)
        assert tot.item() == ref.sum()
