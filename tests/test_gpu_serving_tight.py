"""A server whose memory holds one request whole and a second one's plan and
bins, but not its batch's state: the second waits until the first retires."""
import numpy as np
import pytest

from synthetic import workloads as W
from synthetic.circuits import chain_line_circuit

pytestmark = pytest.mark.gpu


def test_only_request_waits_for_memory():
    import torch
    from paper_2207_00933_gb300 import Context, Server, _build
    _build.build()
    c = chain_line_circuit(4, [16, 14], [2], 1)
    rng = np.random.default_rng(4)
    probs = [torch.from_numpy(rng.random((4 ** len(c.incident[i]), 1 << c.width(i)), dtype=np.float32)).cuda()
             for i in range(c.n_subcircuits)]
    roles = W.lowest_active_roles(c, [10, 11])
    with Context(0) as ctx:
        cid = ctx.load_subcircuit_outputs(c.n_qubits, *c.graph_arrays(), probs)
        resident = ctx.memory_info()["held"]
        qid, na = ctx.set_qubit_roles(cid, roles)
        want = torch.empty(1 << na, dtype=torch.float32, device="cuda")
        plan = ctx.memory_info()["held"] - resident
        bid = ctx.batch_create([qid], [want])
        state = ctx.memory_info()["held"] - resident - plan
        ctx.batch_run(bid)
        ctx.batch_status(bid)
        want = want.cpu().numpy()
    one = plan + (4 << na) + state
    with Context(0, hbm_budget_bytes=resident + one + plan + (4 << na) + state // 2) as ctx:
        cid = ctx.load_subcircuit_outputs(c.n_qubits, *c.graph_arrays(), probs)
        with Server(ctx, max_batch=1, n_streams=2) as srv:
            tickets = [srv.submit(cid, roles) for _ in range(40)]
            srv.drain(60.0)
            for t in tickets:
                assert np.array_equal(srv.result(t), want)
            assert srv.stats()["busy_refusals"] > 0
