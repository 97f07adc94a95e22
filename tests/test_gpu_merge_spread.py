"""Merges whose merged qubits do not lie together: alternating with active and
zoomed ones, in runs, a single one, none; one to 32 lanes per output and a few
to 2^16 states, in a query's own merge, a one-launch query and a batch.
Integer outputs: the bins equal the FP64 oracle's exactly."""
import numpy as np
import pytest

import oracle as O
from synthetic import workloads as W
from synthetic.circuits import chain_line_circuit

pytestmark = pytest.mark.gpu

A, M, Z, T = W.ACTIVE, W.MERGED, W.ZOOM0, W.ZOOM1
PATTERNS = {
    "alternating": [M, A, M, Z],
    "merged_low": [A, M, M, M, M, M, M],          # (data qubit 0 is the highest storage bit)
    "one": [A, A, A, A, M, A, T],
    "runs": [M, M, M, A, Z, M, M, M, M, T],
    "none": [A, Z, A],
    "mostly": [M] * 9 + [A] + [M] * 7 + [T],
}


@pytest.mark.parametrize("pattern", sorted(PATTERNS))
@pytest.mark.parametrize("widths,cuts", [([8, 7], [1]), ([18, 6], [1]), ([6, 17, 5], [1, 1])])
def test_spread_merge(pattern, widths, cuts):
    import torch
    from paper_2207_00933_gb300 import Context, _build
    _build.build()
    c = chain_line_circuit(sum(widths), widths, cuts, 1)
    rng = np.random.default_rng(sum(widths))
    probs = []
    for i in range(c.n_subcircuits):
        p = np.zeros((4 ** len(c.incident[i]), 1 << c.width(i)), dtype=np.float32)
        p[np.arange(len(p))[:, None], rng.integers(0, p.shape[1], (len(p), min(p.shape[1], 200)))] = 1
        probs.append(p)
    roles = np.array((PATTERNS[pattern] * c.n_qubits)[:c.n_qubits], dtype=np.int8)
    for q in np.nonzero(roles == A)[0][14:]:
        roles[q] = M
    g = O.Graph.from_arrays(c.n_qubits, *c.graph_arrays())
    T_ = O.subcircuit_tensors(g, [p.astype(np.float64) for p in probs], roles)
    assert O.reconstruct_pairwise(g, [np.abs(t) for t in T_], roles).max() * 2.0 ** c.n_edges < 2 ** 24
    want = O.reconstruct_pairwise(g, T_, roles)
    dev = [torch.from_numpy(p).cuda() for p in probs]
    for fused in (False, True):
        with Context(0, fused_query=fused) as ctx:
            cid = ctx.load_subcircuit_outputs(c.n_qubits, *c.graph_arrays(), dev)
            qid, na = ctx.set_qubit_roles(cid, roles)
            outs = [torch.full((1 << na,), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2)]
            ctx.reconstruct(qid, outs[0])
            b = ctx.batch_create([qid], [outs[1]])
            ctx.batch_run(b)
            ctx.batch_status(b)
            for o in outs:
                assert np.array_equal(o.cpu().numpy(), want)
