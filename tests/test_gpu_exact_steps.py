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


def _chain(seed, widths, cuts, most=2, ones=None):
    """A chain with outputs in 0..most, or with `ones` ones per variant."""
    c = chain_line_circuit(seed, widths, cuts, 1)
    rng = np.random.default_rng(seed)
    probs = []
    for i in range(c.n_subcircuits):
        shape = (4 ** len(c.incident[i]), 1 << c.width(i))
        if ones is None:
            p = rng.integers(0, most + 1, shape)
        else:
            p = np.zeros(shape)
            p[np.arange(shape[0])[:, None], rng.integers(0, shape[1], (shape[0], ones))] = 1
        probs.append(p.astype(np.float32))
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
    T = O.subcircuit_tensors(g, [p.astype(np.float64) for p in probs], roles)
    # the premise: no partial sum of the contraction reaches 2^24 (the 2^-K is exact)
    assert O.reconstruct_pairwise(g, [np.abs(t) for t in T], roles).max() * 2.0 ** c.n_edges < 2 ** 24
    ref = O.reconstruct_pairwise(g, T, roles)
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


@pytest.mark.parametrize("precision", ["fp32", "split_bf16"])
@pytest.mark.parametrize("widths,cut,active", [
    ([14, 13], 2, [12, 13]),          # 16 rows: 2^16 and 2^17 outputs, value by value
    ([16, 14], 2, [14, 14]),          # 16 rows, 2^18 outputs: half-height tiles
    ([15, 14], 3, [12, 12]),          # 64 rows, one and four states per bin
    ([14, 14], 4, [10, 10]),          # 256 rows, 1 and 16 states per bin
    ([14, 13], 4, [9, 10]),           # 2 and 8 states per bin; the first below the tiles' size
])
def test_turned_merge(widths, cut, active, precision):
    c, probs = _chain(sum(widths) + cut, widths, [cut], most=1)
    _check(c, probs, W.lowest_active_roles(c, active), precision=precision)


def test_turned_merge_other_roles():
    """Bins that are not the lowest data qubits, a zoomed qubit, a three-block
    chain whose middle tensor keeps edges beside its shared ones, the merge
    pyramid and slices."""
    c, probs = _chain(5, [14, 14], [4], most=1)
    rng = np.random.default_rng(5)
    roles = np.zeros(c.n_qubits, dtype=np.int8)
    roles[rng.permutation(10)[:1]] = W.MERGED
    roles[10 + rng.permutation(14)[:3]] = [W.ZOOM1, W.MERGED, W.MERGED]
    _check(c, probs, roles)
    c, probs = _chain(6, [8, 13, 8], [2, 2], most=1)
    _check(c, probs, W.lowest_active_roles(c, [4, 11, 5]))
    c, probs = _chain(7, [15, 14], [3], most=1)
    for cfg in ({"merge_pyramid": True}, {"slice_edges": 1}):
        _check(c, probs, W.lowest_active_roles(c, [12, 12]), **cfg)


@pytest.mark.parametrize("widths,cuts,active,zoom", [
    ([14, 13, 12], [1, 1], [1, 1, 0], {}),          # 2^11-state runs at the edge, 2^12 and 2^12
    ([15, 14], [2], [2, 0], {0: 1, 13: 0}),
    ([14], [], [1], {}),                             # one subcircuit: straight into the bins
])
def test_long_merge(widths, cuts, active, zoom):
    c, probs = _chain(sum(widths), widths, cuts, ones=40)
    for out in ("float32", "float64"):
        _check(c, probs, W.lowest_active_roles(c, active, zoom), out=out)


@pytest.mark.parametrize("widths,cuts,active", [
    ([18, 6], [1], [2, 5]), ([6, 18], [1], [4, 3]), ([6, 18, 7], [1, 1], [3, 2, 5]),
    ([17, 5, 18], [1, 1], [2, 2, 3]), ([16, 6], [1], [2, 5]), ([15, 6], [1], [0, 4])])
def test_long_merge_beside_others(widths, cuts, active):
    """Runs of 2^13 to 2^15 states, in each place among subcircuits of short
    ones: merged in a launch of their own from 2^14 on."""
    c, probs = _chain(7 + sum(widths), widths, cuts, ones=40)
    for out in ("float32", "float64"):
        _check(c, probs, W.lowest_active_roles(c, active), out=out)


@pytest.mark.parametrize("policy", [0, 2])
def test_batch_bands(policy):
    """The batched launch's bands (shared index 1, 4 and 16, from the smallest
    to several bands, more rows than columns and fewer) and its merges, for
    queries of one launch that differ in every shape; and an output that is
    not 16-byte aligned, which takes the plain tiles."""
    import torch
    from paper_2207_00933_gb300 import Context, _build
    _build.build()
    shapes = [([7, 7], [1], [6, 7]), ([7, 8], [2], [5, 8]), ([9, 12], [1], [5, 11]), ([12, 9], [2], [10, 4]),
              ([5, 14], [2], [3, 12]), ([13, 5], [1], [12, 3]), ([8, 9, 8], [1, 2], [5, 5, 6]), ([9, 9], [0], [6, 8]),
              ([10, 10, 9], [2, 2], [4, 3, 5]), ([12, 12], [2], [9, 9]), ([13, 13], [2], [11, 11])]
    with Context(0) as ctx:
        queries, outs, want, store = [], [], [], []
        for j, (widths, cuts, active) in enumerate(shapes):
            c, probs = _chain(100 + j, widths, cuts, most=1)
            roles = W.lowest_active_roles(c, active)
            cid = ctx.load_subcircuit_outputs(c.n_qubits, *c.graph_arrays(), [torch.from_numpy(p).cuda() for p in probs])
            q, na = ctx.set_qubit_roles(cid, roles)
            buf = torch.full(((1 << na) + 1,), float("nan"), dtype=torch.float32, device="cuda")
            queries.append(q)
            store.append(buf)
            outs.append(buf[j == 3:][:1 << na])
            g = O.Graph.from_arrays(c.n_qubits, *c.graph_arrays())
            T = O.subcircuit_tensors(g, [p.astype(np.float64) for p in probs], roles)
            assert O.reconstruct_pairwise(g, [np.abs(t) for t in T], roles).max() * 2.0 ** c.n_edges < 2 ** 24
            want.append(O.reconstruct_pairwise(g, T, roles))
        totals = torch.zeros(len(queries), dtype=torch.float64, device="cuda")
        if policy:
            ctx.batch_autotune(queries, outs, totals, reps=1)
        b = ctx.batch_create(queries, outs, totals)
        for _ in range(2):
            ctx.batch_run(b)
        ctx.batch_status(b)
        for o, w, t in zip(outs, want, totals.cpu().numpy()):
            assert np.array_equal(o.double().cpu().numpy(), w)
            assert abs(t - w.sum()) <= 1e-6 * np.abs(w).sum()
        ctx.batch_release(b)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("widths,cuts", [
    ([3, 4, 4], [1, 2]),              # two data qubits in the middle block: the least the streaming form takes
    ([4, 6, 5], [1, 3]),
    ([7, 9, 9], [3, 3]),              # 64 prepared states x 8 outcomes: 16-state tiles of 64
    ([9, 11, 8], [3, 3]),
    ([8, 8, 8], [4, 2]),              # 256 x 4: 8-state tiles
    ([8, 9, 7], [4, 3]),              # 256 x 8: 4-state tiles
    ([8, 8, 7], [5, 1]),              # 1024 x 2
    ([10, 9], [6]),                   # 4096 prepared states: too many for a tile
    ([13, 10], [1]),                  # no incoming edge, and no outgoing one
    ([9], []),
])
def test_attribution_forms(widths, cuts, offset):
    """Every attributed value shows in some bin when all qubits are active;
    inputs at a 16-byte address and one value beyond it."""
    import torch
    from paper_2207_00933_gb300 import Context, _build
    _build.build()
    c, probs = _chain(sum(widths), widths, cuts, ones=6)
    g = O.Graph.from_arrays(c.n_qubits, *c.graph_arrays())
    roles = np.zeros(c.n_qubits, dtype=np.int8)
    T = O.subcircuit_tensors(g, [p.astype(np.float64) for p in probs], roles)
    assert O.reconstruct_pairwise(g, [np.abs(t) for t in T], roles).max() * 2.0 ** c.n_edges < 2 ** 24
    want = O.reconstruct_pairwise(g, T, roles)
    dev = []
    for p in probs:
        buf = torch.zeros(p.size + 4, dtype=torch.float32, device="cuda")
        buf[offset:offset + p.size] = torch.from_numpy(p).cuda().flatten()
        dev.append(buf[offset:offset + p.size].view(p.shape))
    for cfg in ({}, {"merge_pyramid": True}):
        with Context(0, **cfg) as ctx:
            cid = ctx.load_subcircuit_outputs(c.n_qubits, *c.graph_arrays(), dev)
            ctx.update_subcircuit_outputs(cid, dev)
            qid, na = ctx.set_qubit_roles(cid, roles)
            res = torch.full((1 << na,), float("nan"), dtype=torch.float64, device="cuda")
            ctx.reconstruct(qid, res)
            torch.cuda.synchronize()
            assert np.array_equal(res.cpu().numpy(), want)
