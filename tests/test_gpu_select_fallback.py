"""The filtering selection on inputs made against it: a CTA of the filter keeps
more values than its buffer holds, or the sample's key lies above all but a few
values.  Both go to the radix passes inside the launch.  The inputs are built
from a restatement of the filter's rule, which also has to say that they take
that branch, so that a change of its constants cannot empty the test."""
import math

import numpy as np
import pytest

from synthetic import workloads as W

N = (1 << 23) + 11
THREADS, BUFFER = 1024, (200 * 1024 - 4096 * 4 - 8 * 1024 * 16) // 8


def _sampled(n):
    """Positions of the sampled chunks of 4 values, [chunks a thread reads, threads]."""
    chunks = min(max(n >> 26, 2), 64)
    strata = min(n // 16, chunks * THREADS)
    span = n // strata
    h = np.arange(strata, dtype=np.uint64) * np.uint64(0x9E3779B1) & np.uint64(0xFFFFFFFF)
    h ^= h >> np.uint64(15)
    h = h * np.uint64(0x85EBCA77) & np.uint64(0xFFFFFFFF)
    h ^= h >> np.uint64(13)
    at = np.arange(strata, dtype=np.uint64) * np.uint64(span) + np.uint64(4) * (h * np.uint64(span >> 2) >> np.uint64(32))
    return (at & ~np.uint64(3)).astype(np.int64).reshape(chunks, -1)


def _branch(x, k, ctas, thr=-math.inf):
    """What the filter finds: "over" (a buffer runs over), "misled" (too few values reach the key) or "fits"."""
    n, at = len(x), _sampled(len(x))
    v = np.where(x >= thr, x, -math.inf).astype(x.dtype)                 # NaN and values below the threshold: never
    most = v[(at[:, :, None] + np.arange(4)).clip(max=n - 1)].max(axis=(0, 2))
    j = min(max(4 * max(k, 2048) * 4 * at.size // n, 16), 256)
    some = (most > -math.inf).sum() > j
    tau = np.sort(most)[-j] if some else -math.inf                       # (none: every value from the threshold on)
    per = 16 // x.itemsize                                              # values per 16-byte vector
    kept = np.flatnonzero(v > tau)
    cta = np.where(kept < n // per * per, kept // per // THREADS % ctas, 0)
    if np.bincount(cta, minlength=ctas).max() > BUFFER:
        return "over"
    return "misled" if some and len(kept) + (v == tau).sum() < k else "fits"


def _inputs(dtype, ctas):
    """(name, values, branch, [(k, threshold)])"""
    rng = np.random.default_rng(11)
    at = _sampled(N)
    free = np.ones(N, dtype=bool)
    free[(at[:, :, None] + np.arange(4)).ravel()] = False
    per = 16 // np.dtype(dtype).itemsize
    one_cta = np.flatnonzero(free & (np.arange(N) // per // THREADS % ctas == 0))[:BUFFER + 400]
    base = rng.random(N).astype(dtype)
    nan = rng.random(N) < 0.01
    over = base.copy()
    over[one_cta] += 1 + rng.random(len(one_cta)).astype(dtype)
    yield "over", over, "over", [(1, -math.inf), (4096, -math.inf), (4096, 1.0)]
    holes = np.where(nan & free & (over < 1), np.nan, over).astype(dtype)
    holes[one_cta[:3]] = math.inf
    yield "over, NaN and infinities", holes, "over", [(4096, -math.inf)]
    equal = base.copy()
    equal[one_cta] = 2
    yield "over, all equal", equal, "over", [(1, -math.inf), (4096, -math.inf)]
    misled = base.copy()
    misled[~free] = 2 + rng.permutation((~free).sum()).astype(dtype) / 8192
    yield "misled", misled, "misled", [(100, -math.inf), (4096, -math.inf), (4096, 2.25)]
    yield "misled, NaN", np.where(nan & free, np.nan, misled).astype(dtype), "misled", [(4096, -math.inf)]
    ties = np.full(N, -0.5, dtype=dtype)
    ties[at[0, :40]] = 1 + np.arange(40, dtype=dtype)
    yield "misled, ties of the k-th", ties, "misled", [(100, -math.inf), (4096, -math.inf)]


@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_restated_rule(dtype):
    for name, x, branch, calls in _inputs(dtype, 152):
        for k, thr in calls:
            assert _branch(x, k, 152, thr) == branch, (name, k)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_fallback_is_exact(dtype):
    import torch
    from paper_2207_00933_gb300 import Context, _build
    _build.build()
    w = W.full_state_12q()
    c = w.circuit
    ctas = torch.cuda.get_device_properties(0).multi_processor_count

    def check(ctx, qid, x, k, thr):
        b, v, nf = ctx.top_bins(qid, x, k, thr)
        idx = torch.nonzero(x >= thr).flatten()
        val, order = torch.sort(x[idx], descending=True, stable=True)
        m = min(k, idx.numel())
        assert int(nf.item()) == m
        assert torch.equal(b[:m], idx[order[:m]]) and torch.equal(v[:m], val[:m].double())

    with Context(0) as ctx:
        cid = ctx.load_subcircuit_outputs(c.n_qubits, *c.graph_arrays(), [torch.from_numpy(p).cuda() for p in w.probs])
        qid, _ = ctx.set_qubit_roles(cid, w.roles)
        plain = torch.rand(N, dtype=getattr(torch, dtype), device="cuda")
        shifted = torch.empty(N + 1, dtype=plain.dtype, device="cuda")
        for name, x, branch, calls in _inputs(dtype, ctas):
            dev = torch.from_numpy(x).cuda()
            shifted[1:] = dev
            for k, thr in calls:
                assert _branch(x, k, ctas, thr) == branch, (name, k)
                for y in (dev, shifted[1:]):                  # 16-byte aligned, and not
                    check(ctx, qid, y, k, thr)
            check(ctx, qid, plain, 1000, -math.inf)           # the workspace is left as it was found


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_more_sampled_chunks(dtype):
    """Beyond 2^27 values a thread samples more than two chunks."""
    import torch
    from paper_2207_00933_gb300 import Context, _build
    _build.build()
    w = W.full_state_12q()
    c = w.circuit
    with Context(0) as ctx:
        cid = ctx.load_subcircuit_outputs(c.n_qubits, *c.graph_arrays(), [torch.from_numpy(p).cuda() for p in w.probs])
        qid, _ = ctx.set_qubit_roles(cid, w.roles)
        n = (1 << 28) + 5
        x = torch.empty(n, dtype=getattr(torch, dtype), device="cuda").exponential_(1.0)
        for k in (1, 4096):
            b, v, nf = ctx.top_bins(qid, x, k)
            val = torch.topk(x, k).values
            assert int(nf.item()) == k
            assert torch.equal(v, val.double()) and torch.equal(x[b].double(), v)
            assert b.unique().numel() == k
