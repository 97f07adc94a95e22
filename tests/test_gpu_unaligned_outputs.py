"""Bins written to an address that is not 16-byte aligned: the same values, bit
for bit, as to an aligned one, and nothing beside them, in every form of the
last step (bands, pipelined and plain tiles, the tensor cores, FP64 chunks,
slices, one-launch queries, one subcircuit) and in the calls around it."""
import numpy as np
import pytest

from synthetic import workloads as W
from synthetic.circuits import chain_line_circuit

pytestmark = pytest.mark.gpu

CASES = {
    "band": ([13, 10], [2], [10, 10], {}),                  # 1024 x 1024, K = 16
    "outer_product": ([10, 10], [0], [10, 10], {}),         # K = 1
    "pipelined": ([14, 10], [3], [11, 10], {}),             # 1024 x 2048, K = 64
    "small": ([7, 6], [2], [5, 6], {}),
    "tensor": ([16, 12], [4], [11, 12], {}),                # 2048 x 4096, K = 256 (split-BF16)
    "chunks": ([14, 10], [3], [11, 10], {"fp64_chunk_min_edges": 1, "chunk_terms": 16}),
    "slices": ([13, 10], [3], [10, 10], {"slice_edges": 1}),
    "one_launch": ([13, 10], [2], [10, 10], {"fused_query": True}),
    "one_subcircuit": ([14], [], [12], {}),
}


@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("case", sorted(CASES))
def test_unaligned_outputs(case, dtype):
    import torch
    from paper_2207_00933_gb300 import Context, _build
    _build.build()
    widths, cuts, active, cfg = CASES[case]
    c = chain_line_circuit(9, widths, cuts, 1)
    rng = np.random.default_rng(9)
    probs = [torch.from_numpy(rng.random((4 ** len(c.incident[i]), 1 << c.width(i)), dtype=np.float32)).cuda()
             for i in range(c.n_subcircuits)]
    with Context(0, **cfg) as ctx:
        cid = ctx.load_subcircuit_outputs(c.n_qubits, *c.graph_arrays(), probs)
        qid, na = ctx.set_qubit_roles(cid, W.lowest_active_roles(c, active))
        n, dt = 1 << na, getattr(torch, dtype)
        total = [torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(2)]
        for precision in ("fp32", "split_bf16"):
            for call in ("reconstruct", "outputs", "select"):
                if call != "reconstruct" and cfg.get("slice_edges"):
                    continue                                     # (refused: sliced queries)
                room = [torch.full((n + 8,), -7.0, dtype=dt, device="cuda") for _ in range(2)]
                outs = [room[0][:n], room[1][1:n + 1]]
                assert outs[0].data_ptr() % 16 == 0 and outs[1].data_ptr() % 16 != 0
                top = []
                for o, t in zip(outs, total):
                    if call == "reconstruct":
                        ctx.reconstruct(qid, o, precision, t)
                    elif call == "outputs":
                        ctx.reconstruct_outputs(qid, probs, o, precision, t)
                    else:
                        top.append(ctx.reconstruct_select(qid, o, 100, precision=precision, total_prob=t))
                assert torch.equal(outs[0], outs[1]), (precision, call)
                assert (room[1][n + 1:] == -7).all() and room[1][0] == -7
                # (one-launch queries and steps of other tiles add the sum's parts in another order)
                assert abs(total[0].item() - total[1].item()) <= 1e-5 * outs[0].double().abs().sum().item()
                if top:
                    assert all(torch.equal(a, b) for a, b in zip(*top))
