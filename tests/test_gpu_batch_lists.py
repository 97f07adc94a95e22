"""Batched levels whose work lists are shorter than the launch's CTAs, about as
long, and several times as long (items are claimed ahead of the one at hand
only while many are left): the bins equal the single queries' bit for bit, run
after run and after a wait that runs out."""
import numpy as np
import pytest

from synthetic import workloads as W
from synthetic.circuits import chain_line_circuit

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 24, 150])
def test_list_lengths(n):
    import torch
    from paper_2207_00933_gb300 import Context, SQCError, _build
    _build.build()
    rng = np.random.default_rng(n)
    with Context(0, wait_limit_ms=200) as ctx:
        queries, outs, want = [], [], []
        circuits = []
        for widths, cuts in (([7, 8, 7], [1, 2]), ([9, 8], [2]), ([6, 7, 6, 7], [1, 1, 1])):
            c = chain_line_circuit(sum(widths), widths, cuts, 1)
            probs = [torch.from_numpy(rng.random((4 ** len(c.incident[i]), 1 << c.width(i)), dtype=np.float32)).cuda()
                     for i in range(c.n_subcircuits)]
            circuits.append((c, ctx.load_subcircuit_outputs(c.n_qubits, *c.graph_arrays(), probs)))
        for j in range(n):
            c, cid = circuits[j % 3]
            active = [int(rng.integers(1, len(d) + 1)) for d in c.data_qubits]
            qid, na = ctx.set_qubit_roles(cid, W.lowest_active_roles(c, active))
            ref = torch.empty(1 << na, dtype=torch.float32, device="cuda")
            ctx.reconstruct(qid, ref)
            queries.append(qid)
            want.append(ref)
            outs.append(torch.empty_like(ref))
        totals = torch.zeros(n, dtype=torch.float64, device="cuda")
        b = ctx.batch_create(queries, outs, totals)

        def check():
            for o in outs:
                o.fill_(float("nan"))
            ctx.batch_run(b)
            ctx.batch_status(b)
            for o, w, t in zip(outs, want, totals.cpu().tolist()):
                assert torch.equal(o, w)
                assert abs(t - w.double().sum().item()) <= 1e-6 * w.double().abs().sum().item()

        for _ in range(3):
            check()
        ctx.batch_inject_stall(b, True)
        ctx.batch_run(b)
        with pytest.raises(SQCError):
            ctx.batch_status(b)
        ctx.batch_release(b)
        b = ctx.batch_create(queries, outs, totals)
        check()
        ctx.batch_release(b)
