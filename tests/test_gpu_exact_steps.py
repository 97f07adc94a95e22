"""Bit-exact parity of the merge and contraction kernels at the edges of
their tile shapes.  The variant outputs are small integers and every partial
sum stays below 2^24, so FP32 arithmetic is exact whatever the order: the
bins must equal the FP64 oracle's exactly."""
import numpy as np
import pytest

import oracle as O
from synthetic import workloads as W
from synthetic.circuits import chain_line_circuit

pytestmark = pytest.mark.gpu


def _chain(seed, widths, cuts, most=2):
    c = chain_line_circuit(seed, widths, cuts, 1)
    rng = np.random.default_rng(seed)
    probs = [rng.integers(0, most + 1, (4 ** len(c.incident[i]), 1 << c.width(i))).astype(np.float32)
             for i in range(c.n_subcircuits)]
    return c, probs


def _run(c, probs, roles, precision="fp32", out="float32", **cfg):
    import torch
    from paper_2207_00933_gb300 import Context, _build
    _build.build()
    with Context(0, **cfg) as ctx:
        cid = ctx.load_subcircuit_outputs(c.n_qubits, *c.graph_arrays(), [torch.from_numpy(p).cuda() for p in probs])
        qid, na = ctx.set_qubit_roles(cid, roles)
        res = torch.full((1 << na,), float("nan"), dtype=getattr(torch, out), device="cuda")
        tot = torch.zeros(1, dtype=torch.float64, device="cuda")
        ctx.reconstruct(qid, res, precision, tot)
        torch.cuda.synchronize()
        return res.double().cpu().numpy(), tot.item(), ctx.query_steps(qid)


def _check(c, probs, roles, **kw):
    g = O.Graph.from_arrays(c.n_qubits, *c.graph_arrays())
    ref = O.reconstruct(g, [p.astype(np.float64) for p in probs], roles)
    got, tot, steps = _run(c, probs, roles, **kw)
    assert np.array_equal(got, ref), (steps, np.abs(got - ref).max())
    assert abs(tot - ref.sum()) <= 1e-6 * np.abs(ref).sum()
    return steps


@pytest.mark.parametrize("widths,cut,active,shape", [
    ([13, 10], 3, [10, 10], (1024, 1024, 64)),       # 128 whole tiles of the pipelined form: too few, the plain tiles
    ([14, 10], 3, [11, 10], (1024, 2048, 64)),       # 256 tiles
    ([10, 14], 3, [7, 14], (16384, 128, 64)),        # one tile row of columns
    ([11, 13], 3, [8, 13], (8192, 256, 64)),
    ([16, 10], 4, [11, 10], (1024, 2048, 256)),
])
def test_pipelined_step(widths, cut, active, shape):
    c, probs = _chain(sum(widths) + cut, widths, [cut], most=1)
    steps = _check(c, probs, W.lowest_active_roles(c, active))
    assert tuple(sorted(steps[-1][:2])) == tuple(sorted(shape[:2])) and steps[-1][2] == shape[2]
