"""Attribution of small subcircuits beside one whose reads call for large
tiles: 7 to 10 data qubits at the end of a chain (the ring-buffered form has 9
bits of state per tile) and unconnected (the form without incoming edges takes
four 8-bit tiles at once), alone and several in one launch.  Integer outputs,
sums below 2^24: the bins equal the FP64 oracle's exactly."""
import numpy as np
import pytest

import oracle as O
from synthetic import workloads as W
from synthetic.circuits import chain_line_circuit

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pyramid", [False, True])
@pytest.mark.parametrize("widths,cuts", [
    ([19, 7], [1]), ([19, 8], [1]), ([19, 9], [1]), ([19, 10], [1]), ([18, 8], [2]), ([17, 8], [3]),
    ([20, 7], [0]), ([20, 8], [0]), ([20, 9], [0]), ([20, 10], [0]), ([21, 8], [0]),
    ([19, 8, 9], [1, 0]), ([18, 8, 18, 8], [1, 0, 1]), ([18, 8, 8, 9, 8], [1, 0, 1, 0]), ([8], []), ([9], []),
])
def test_small_beside_large(widths, cuts, pyramid):
    import torch
    from paper_2207_00933_gb300 import Context, _build
    _build.build()
    c = chain_line_circuit(sum(widths), widths, cuts, 1)
    rng = np.random.default_rng(sum(widths))
    probs = []
    for i in range(c.n_subcircuits):
        p = np.zeros((4 ** len(c.incident[i]), 1 << c.width(i)), dtype=np.float32)
        p[np.arange(len(p))[:, None], rng.integers(0, p.shape[1], (len(p), 12))] = 1
        probs.append(p)
    n = [len(d) for d in c.data_qubits]
    g = O.Graph.from_arrays(c.n_qubits, *c.graph_arrays())
    with Context(0, merge_pyramid=pyramid) as ctx:
        dev = [torch.from_numpy(p).cuda() for p in probs]
        cid = ctx.load_subcircuit_outputs(c.n_qubits, *c.graph_arrays(), dev)
        for small in [i for i in range(len(n)) if n[i] <= 10]:      # each small block whole, once
            roles = W.lowest_active_roles(c, [n[i] if i == small else min(n[i], 2) for i in range(len(n))])
            T = O.subcircuit_tensors(g, [p.astype(np.float64) for p in probs], roles)
            assert O.reconstruct_pairwise(g, [np.abs(t) for t in T], roles).max() * 2.0 ** c.n_edges < 2 ** 24
            qid, na = ctx.set_qubit_roles(cid, roles)
            out = torch.full((1 << na,), float("nan"), dtype=torch.float64, device="cuda")
            ctx.reconstruct(qid, out)
            torch.cuda.synchronize()
            assert np.array_equal(out.cpu().numpy(), O.reconstruct_pairwise(g, T, roles)), small
