"""GPU parity of the one-CTA selection (few values, few bins) where it can go
wrong: one value to the most, either side of a value per thread and of the
limit, exact ties of the k-th value in numbers that only the bin can decide,
NaN, infinities and a threshold.  Compared exactly with a full sort of the
same values."""
import math

import pytest

from synthetic import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("n", [1, 31, 1024, 1025, 4095, 4096, 4097])
def test_small_selection(dtype, n):
    import torch
    from paper_2207_00933_gb300 import Context, _build
    _build.build()
    w = W.full_state_12q()
    c = w.circuit
    dt = getattr(torch, dtype)
    with Context(0) as ctx:
        cid = ctx.load_subcircuit_outputs(c.n_qubits, *c.graph_arrays(), [torch.from_numpy(p).cuda() for p in w.probs])
        qid, _ = ctx.set_qubit_roles(cid, w.roles)
        g = torch.Generator(device="cuda").manual_seed(n)
        spread = torch.empty(n + 1, dtype=dt, device="cuda").exponential_(1.0, generator=g)
        odd = spread.clone()
        odd[n // 2] = math.nan
        odd[n // 3] = math.inf
        odd[n // 5] = -math.inf
        few = torch.randint(-2, 3, (n + 1,), device="cuda", generator=g).to(dt) / 8
        zeros = torch.zeros(n + 1, dtype=dt, device="cuda")
        last = zeros.clone()
        last[-2:] = 1.0
        none = torch.full((n + 1,), math.nan, dtype=dt, device="cuda")
        for x in (spread[:n], spread[1:], odd[:n], few[:n], zeros[:n], last[1:], none[:n]):
            for k, thr in ((1, -math.inf), (16, 0.0), (128, -math.inf), (128, 0.25), (129, -math.inf)):
                b, v, nf = ctx.top_bins(qid, x, k, thr)
                idx = torch.nonzero(x >= thr).flatten()                # false for NaN
                val, order = torch.sort(x[idx], descending=True, stable=True)
                m = min(k, idx.numel())
                assert int(nf.item()) == m
                assert torch.equal(b[:m], idx[order[:m]])
                assert torch.equal(v[:m], val[:m].double())
