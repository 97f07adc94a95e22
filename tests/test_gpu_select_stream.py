"""GPU parity of the filtering selection (inputs beyond the shared-memory
resident form, and every input with select_resident=False) where it can go
wrong: the edge between keeping every value and sampling, ragged and
misaligned slices, ties of the filter's key, values that crowd into one
CTA's slice or into one prefix of the sample's digits (both fall back to the
radix passes).  Compared exactly with a full sort of the same values."""
import math

import numpy as np
import pytest

from synthetic import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sel():
    import torch
    from paper_2207_00933_gb300 import Context, _build
    _build.build()
    w = W.full_state_12q()
    c = w.circuit
    ctx = Context(0, select_resident=False)
    cid = ctx.load_subcircuit_outputs(c.n_qubits, *c.graph_arrays(), [torch.from_numpy(p).cuda() for p in w.probs])
    qid, _ = ctx.set_qubit_roles(cid, w.roles)
    yield ctx, qid
    torch.cuda.synchronize()
    ctx.close()


def _check(sel, x, k, thr=-math.inf):
    """Against a stable descending sort (ties by bin ascending); NaN never selected."""
    import torch
    ctx, qid = sel
    b, v, nf = ctx.top_bins(qid, x, k, thr)
    ok = x >= thr                                        # false for NaN
    idx = torch.nonzero(ok).flatten()
    val, order = torch.sort(x[idx], descending=True, stable=True)
    m = min(k, idx.numel())
    assert int(nf.item()) == m
    assert torch.equal(b[:m], idx[order[:m]])
    assert torch.equal(v[:m], val[:m].double())


@pytest.mark.parametrize("dtype", ["float32", "float64"])
@pytest.mark.parametrize("n", [1, 152 * 4 + 1, (1 << 18) - 1, 1 << 18, (1 << 18) + 3, (1 << 23) + 5])
def test_sizes(sel, dtype, n):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.empty(n + 1, dtype=getattr(torch, dtype), device="cuda").exponential_(1.0, generator=g)
    for y in (x[:n], x[1:]):                             # 16-byte aligned, and not
        for k in (1, 1000, 4096):
            _check(sel, y, k)
        _check(sel, y, 4096, 3.0)


@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_ties_of_the_filter(sel, dtype):
    import torch
    g = torch.Generator(device="cuda").manual_seed(3)
    n = (1 << 22) + 7
    dt = getattr(torch, dtype)
    zeros = torch.zeros(n, dtype=dt, device="cuda")
    zeros[n // 3] = 1.0
    few = torch.randint(0, 4, (n,), device="cuda", generator=g).to(dt) / 8
    neg = -few                                           # -0.0 among them
    sparse = torch.where(torch.rand(n, device="cuda", generator=g) < 5e-4, 0.5, 0.25).to(dt)
    spread = zeros.clone()                               # the ties needed spread over every slice
    spread[torch.randperm(n, device="cuda", generator=g)[:3000]] = 0.75
    for x in (zeros, few, neg + 0.25, sparse, spread, torch.full_like(zeros, math.inf)):
        for k in (1, 2500, 4096):
            _check(sel, x, k)
    mixed = few.clone()
    mixed[torch.randperm(n, device="cuda", generator=g)[:5000]] = math.nan
    mixed[torch.randperm(n, device="cuda", generator=g)[:7]] = math.inf
    mixed[torch.randperm(n, device="cuda", generator=g)[:7]] = -math.inf
    _check(sel, mixed, 4096)
    _check(sel, mixed, 4096, 0.375)


@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_fallback(sel, dtype):
    import torch
    g = torch.Generator(device="cuda").manual_seed(9)
    n = (1 << 23) + 11
    x = torch.rand(n, dtype=getattr(torch, dtype), device="cuda", generator=g)
    x[5000:95000] += 1.0                                 # more than a CTA keeps, in one slice
    for k in (1, 4096):
        _check(sel, x, k)
    x[5000:95000] -= 1.0
    x[77:77 + 4000] += 2.0                               # the best in one short run the sample may miss
    _check(sel, x, 4096)
    if dtype == "float64":                               # every value in one prefix of the sample's digits
        y = 1.0 + 1e-12 * torch.rand(1 << 20, dtype=torch.float64, device="cuda", generator=g)
        for k in (1, 4096):
            _check(sel, y, k)
    _check(sel, x, 100)                                  # the workspace is left as it was found
