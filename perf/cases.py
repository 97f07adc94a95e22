"""Measured cases: the calls a user of this framework has it do, over the sizes they meet.

Circuits are chains of blocks joined by cut wires, written as texts of comma-separated numbers: `widths` (wires of
each block), `cuts` (wires handed from each block to the next; 0 starts a new, unconnected chain), `zoom` and `active`
(data qubits of each block fixed by earlier recursions, and kept as bins; the rest are merged).  Variant outputs are
those of Haar-random blocks ("haar": exact, physical, what deep random circuits tend to) or of a Bernstein-Vazirani
circuit ("bv": sparse, with one solution).
"""
import math
import random

import numpy as np
import torch

from paper_2207_00933_gb300 import Context, Server, recursion_roles

ACTIVE, MERGED, ZOOM0, ZOOM1 = 0, 1, 2, 3
MOST_BINS = 24          # log2 of the most bins of a drawn reconstruction


def listed():
    grid = {"widths": "8,11,11,11,11", "cuts": "3,3,3,3", "zoom": "0,0,0,0,0", "active": "4,4,4,5,5"}
    line = {"widths": "10,10,10,8", "cuts": "3,2,3", "zoom": "0,0,0,0", "active": "5,5,5,5"}
    join = {"widths": "16,16", "cuts": "4", "zoom": "0,0", "active": "12,12"}
    step = {"kind": "step", "values": "haar", "inputs": "f32", "out": "f32", "precision": "fp32", "host": False, "captured": False}
    level = {"kind": "level", "values": "haar", "inputs": "f32", "out": "f32", "precision": "fp32", "update": True, "pyramid": False, "slices": 0, "k": 0}
    return [
        # the smallest call: a 12-qubit circuit in two halves, every qubit active, double precision throughout
        {**step, "name": "step_12q", "widths": "7,7", "cuts": "2", "zoom": "0,0", "active": "5,7", "inputs": "f64", "out": "f64", "k": 16},
        # one recursion of a 30-qubit circuit into 2^20 bins, kept in a CUDA graph as a search loop keeps it
        {**step, **line, "name": "step_30q", "captured": True, "k": 1024},
        # the same recursion as its user sees it whose QPU results arrive in pinned host memory
        {**step, **line, "name": "step_30q_host", "host": True, "k": 1024},
        # a 40-qubit grid's recursion: new outputs attributed, 2^22 bins in double precision on the tensor cores, best 1024
        {**level, **grid, "name": "level_40q", "precision": "split_bf16", "out": "f64", "k": 1024},
        # few, wide subcircuits: attribution and merge of 335 MB of outputs into 2^24 bins
        {**level, "name": "level_wide", "widths": "20,22", "cuts": "2", "zoom": "0,0", "active": "10,14"},
        # a dense join of two halves over four cut wires, on the tensor cores and in plain FP32
        {**level, **join, "name": "join_tensor", "precision": "split_bf16", "update": False},
        {**level, **join, "name": "join_fp32", "update": False},
        # one recursion level of many zoomed bins over a few resident circuits
        {"kind": "batch", "name": "batch_256", "shape": 4, "circuits": 4, "queries": 256, "a_min": 10, "a_max": 20, "pyramid": False, "update": False},
        # the same with the outputs of a new run and the marginals kept, as a program does that asks many queries of one run
        {"kind": "batch", "name": "batch_64_pyramid", "shape": 9, "circuits": 2, "queries": 64, "a_min": 10, "a_max": 20, "pyramid": True, "update": True},
        # the best bins of a large distribution (2^26 bins)
        {"kind": "top", "name": "top_64m", "n": 1 << 26, "dtype": "f32", "values": "narrow", "k": 1024, "threshold": False},
        # one recursion of a 1000-qubit search: new roles, their plan, the bins, the best of them, the plan released
        {"kind": "search", "name": "search_1000q", "values": "bv", "blocks": 59, "width": 18, "cut": 1, "fixed": 120, "bins": 20, "k": 16},
        # a server's burst: zoom queries on large resident circuits, planned, batched and returned to the host
        {"kind": "serve", "name": "serve_48", "shape": 6, "circuits": 3, "queries": 48, "a_min": 12, "a_max": 20, "pyramid": False},
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "level", "level", "level", "join", "batch", "top", "top", "search", "serve"])
    if kind == "step":
        while True:
            c = _draw_chain(rng, rng.randint(2, 6), 3, 13, 20, 8)
            if 6 <= sum(_ints(c["active"])) <= 21 and _chain_flops(c, _ints(c["active"])) < 2e9:
                break
        precision = rng.choice(["fp32", "fp32", "split_bf16"])
        return {"kind": kind, **c, "values": rng.choice(["haar", "haar", "bv"]), "inputs": rng.choice(["f32", "f32", "f64"]),
                "out": rng.choice(["f32", "f32", "f64"]), "precision": precision, "host": rng.random() < 0.2, "captured": rng.random() < 0.3,
                "k": min(_log(rng, 1, 4096), 1 << sum(_ints(c["active"])))}
    if kind == "level":
        while True:
            c = _draw_chain(rng, rng.randint(2, 5), 3, 22, rng.choice([18, 22, 26]), 30)
            if 8 <= sum(_ints(c["active"])) <= 22 and sum(1 << w for w in _sizes(c)) <= 1 << 26 and _chain_flops(c, _ints(c["active"])) < 2e9:
                break
        k = rng.choice([0, _log(rng, 1, 4096)])
        return {"kind": kind, **c, "values": rng.choice(["haar", "haar", "bv"]), "inputs": rng.choice(["f32", "f32", "f64"]), "out": rng.choice(["f32", "f64"]),
                "precision": rng.choice(["fp32", "split_bf16"]), "update": rng.random() < 0.7, "pyramid": rng.random() < 0.2,
                "slices": 1 if rng.random() < 0.2 else 0, "k": min(k, 1 << sum(_ints(c["active"])))}
    if kind == "join":
        cut, w0, w1 = rng.randint(2, 4), rng.randint(13, 16), rng.randint(13, 16)
        a0, a1 = rng.randint(7, min(12, w0 - cut)), rng.randint(7, 12)
        return {"kind": "level", "widths": "%d,%d" % (w0, w1), "cuts": str(cut), "zoom": "0,0", "active": "%d,%d" % (a0, a1), "values": "haar",
                "inputs": "f32", "out": rng.choice(["f32", "f32", "f64"]), "precision": rng.choice(["fp32", "split_bf16"]), "update": False, "pyramid": False,
                "slices": 0, "k": 0}
    if kind in ("batch", "serve"):
        a = rng.randint(8, 18)
        n = _log(rng, 8, 256 if kind == "batch" else 48)
        c = {"kind": kind, "shape": rng.randrange(1 << 20), "circuits": rng.randint(1, 4 if kind == "batch" else 3), "queries": n, "a_min": a,
             "a_max": rng.randint(a, 20), "pyramid": rng.random() < 0.3}
        return {**c, "update": rng.random() < 0.3} if kind == "batch" else c
    if kind == "top":
        return {"kind": kind, "n": _log(rng, 1000, 1 << 26), "dtype": rng.choice(["f32", "f64"]), "values": rng.choice(["narrow", "thomas", "peaked"]),
                "k": _log(rng, 1, 4096), "threshold": rng.random() < 0.3}
    blocks, width = _log(rng, 6, 59), rng.randint(8, 18)
    return {"kind": "search", "values": rng.choice(["bv", "haar"]) if width <= 14 else "bv", "blocks": blocks, "width": width, "cut": 1,
            "fixed": rng.randint(0, blocks * (width - 1) // 2), "bins": rng.randint(8, 20), "k": _log(rng, 1, 256)}


# ---- shapes ------------------------------------------------------------------------------------

def _ints(text):
    return [int(v) for v in text.split(",") if v]


def _text(values):
    return ",".join(str(v) for v in values)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _links(c):
    """(incoming, outgoing) cut wires of every block."""
    cuts = _ints(c["cuts"])
    return list(zip([0] + cuts, cuts + [0]))


def _data(c):
    return [w - o for w, (_, o) in zip(_ints(c["widths"]), _links(c))]


def _sizes(c):
    """log2 of the values in every block's variant outputs."""
    return [w + 2 * (i + o) for w, (i, o) in zip(_ints(c["widths"]), _links(c))]


def _draw_chain(rng, blocks, most_cuts, most_width, most_log, most_merged):
    while True:
        cuts = [rng.randint(1, most_cuts) for _ in range(blocks - 1)]
        links = list(zip([0] + cuts, cuts + [0]))
        widths = []
        for i, o in links:
            lo, hi = max(i + o + 1, 4), min(most_width, most_log - 2 * (i + o))
            widths.append(rng.randint(max(lo, hi - 6), hi) if lo <= hi else 0)
        if 0 in widths:
            continue
        zoom, active = [], []
        for w, (_, o) in zip(widths, links):
            n = w - o
            z = rng.choice([0, rng.randint(0, n // 3)])
            lo = max(0, n - z - most_merged)
            zoom.append(z)
            active.append(rng.randint(lo, max(lo, min(n - z, max(lo, 14 if blocks == 2 else 8)))))
        if sum(active) <= MOST_BINS:
            return {"widths": _text(widths), "cuts": _text(cuts), "zoom": _text(zoom), "active": _text(active)}


def _graph(c):
    """(n_qubits, edge_up, edge_down, n_data, data_qubit) of a chain."""
    up, down = [], []
    for b, h in enumerate(_ints(c["cuts"])):
        up += [b] * h
        down += [b + 1] * h
    n = _data(c)
    return sum(n), up, down, n, list(range(sum(n)))


def _roles(c, zoom, active, bits):
    """Roles of a query: per block the lowest `zoom` data qubits fixed (to `bits`), the next `active` kept, the rest merged."""
    roles = []
    for n, z, a in zip(_data(c), zoom, active):
        roles += [ZOOM1 if bits[len(roles) + t] else ZOOM0 for t in range(z)] + [ACTIVE] * a + [MERGED] * (n - z - a)
    return np.array(roles, dtype=np.int8)


def _chain_flops(c, active):
    """Least 2MNK over all ways to contract neighbouring blocks pair by pair."""
    cuts = [0] + _ints(c["cuts"]) + [0]
    nb = len(active)
    best = [[0.0] * nb for _ in range(nb)]
    for span in range(1, nb):
        for i in range(nb - span):
            j = i + span
            best[i][j] = min(best[i][m] + best[m + 1][j] + 2.0 * 2.0 ** (sum(active[i:j + 1]) + 2 * (cuts[i] + cuts[m + 1] + cuts[j + 1])) for m in range(i, j))
    return best[0][nb - 1]


def _many(case):
    """The circuits and queries of a batch or a server: [(chain)], [(circuit, zoom, active)]."""
    rng = random.Random(case["shape"])
    serve = case["kind"] == "serve"
    circuits, queries = [], []
    while len(circuits) < case["circuits"]:
        if serve:      # 16 to 50 blocks of at most 14 wires, 10 to 40 cuts: chains of some blocks each, side by side
            blocks = rng.randint(16, 50)
            cuts = [rng.choice([0, 1, 1]) for _ in range(blocks - 1)]
            for _ in range(2):
                cuts[rng.randrange(blocks - 1)] = rng.randint(1, 2)
            if not 10 <= sum(cuts) <= 40:
                continue
            most_width, most_log, least = 14, 18, 3
        else:          # 5 or 6 blocks of at most 16 wires, 6 to 10 cuts, 60 qubits or more
            blocks = rng.randint(5, 6)
            cuts = [1] * (blocks - 1)
            for _ in range(rng.randint(0, 10 - len(cuts))):
                cuts[rng.randrange(blocks - 1)] += 1
            most_width, most_log, least = 16, 22, 2
        links = list(zip([0] + cuts, cuts + [0]))
        hi = [min(most_width, most_log - 2 * (i + o)) for i, o in links]
        if any(h < i + o + 2 for h, (i, o) in zip(hi, links)):
            continue
        widths = [rng.randint(max(i + o + 2, h - least), h) for h, (i, o) in zip(hi, links)]
        c = {"widths": _text(widths), "cuts": _text(cuts)}
        if sum(_data(c)) >= (200 if serve else 50):
            circuits.append(c)
    for _ in range(case["queries"]):
        ci = rng.randrange(len(circuits))
        n = _data(circuits[ci])
        if serve:
            zoom, hosts = [0] * len(n), rng.sample(range(len(n)), rng.randint(2, 5))
            for b in rng.sample(range(len(n)), rng.randint(1, 3)):
                zoom[b] = rng.randint(0, min(3, n[b]))
        else:
            zoom, hosts = [rng.randint(0, v // 3) for v in n], list(range(len(n)))
        active = [0] * len(n)
        for _ in range(rng.randint(case["a_min"], case["a_max"])):
            free = [b for b in hosts if zoom[b] + active[b] < n[b]] or [b for b in range(len(n)) if zoom[b] + active[b] < n[b]]
            if not free:
                break
            active[rng.choice(free)] += 1
        queries.append((ci, zoom, active))
    return circuits, queries


def _search_chain(case):
    nb = case["blocks"]
    return {"widths": _text([case["width"]] * (nb - 1) + [max(4, case["width"] - 4)]), "cuts": _text([case["cut"]] * (nb - 1))}


def _search_split(case, c):
    """(zoom, active) of every block: the qubits earlier recursions fixed, and Algorithm 2's bins for the rest."""
    zoom, left = [], case["fixed"]
    for b, n in enumerate(_data(c)):
        zoom.append(min(n, left // (case["blocks"] - b)))
        left -= zoom[-1]
    active = [n - z for n, z in zip(_data(c), zoom)]
    while sum(active) > case["bins"]:
        active[max(range(len(active)), key=lambda j: (active[j], -j))] -= 1
    return zoom, active


# ---- inputs ------------------------------------------------------------------------------------

_S = math.sqrt(0.5)
_INIT = [[1, 0], [0, 1], [_S, _S], [_S, 1j * _S]]                                              # |0>, |1>, |+>, |+i>
_BASIS = [[[1, 0], [0, 1]], [[_S, _S], [_S, -_S]], [[_S, -1j * _S], [_S, 1j * _S]], [[1, 0], [0, 1]]]   # I, X, Y, Z: outcome from amplitude


def _haar(kin, kout, n, gen, dtype):
    """Variant outputs [4^k, 2^(n + kout)] of a random isometry from the incoming wires to the data and outgoing ones."""
    ct = torch.complex128 if dtype == torch.float64 else torch.complex64
    amp = torch.randn(1 << kin, 1 << (n + kout), dtype=ct, device="cuda", generator=gen)
    low = np.linalg.cholesky((amp @ amp.mH).to(torch.complex128).cpu().numpy())        # orthonormal rows
    amp = torch.from_numpy(np.linalg.inv(low)).to("cuda", ct) @ amp
    init = torch.ones(1, 1, dtype=torch.complex128, device="cuda")
    for _ in range(kin):
        init = torch.kron(init, torch.tensor(_INIT, dtype=torch.complex128, device="cuda"))
    amp = init.to(ct) @ amp
    basis = torch.tensor(_BASIS, dtype=ct, device="cuda")
    digits, outcomes, given = "ijkl"[:kout], "opqr"[:kout], "abcd"[:kout]
    t = torch.einsum("".join(",%s%s%s" % v for v in zip(digits, outcomes, given)).lstrip(",") + ("," if kout else "") + "s" + given[::-1] + "x->s" + digits + outcomes[::-1] + "x",
                     *([basis] * kout), amp.view([1 << (2 * kin)] + [2] * kout + [1 << n]))
    return (t.real.square() + t.imag.square()).reshape(1 << (2 * (kin + kout)), 1 << (n + kout)).contiguous()


def _bv(kin, kout, n, secret, dtype):
    """Variant outputs of a Bernstein-Vazirani block: data qubits read their secret bit, incoming wires finish here, outgoing ones hold |+>."""
    half = [0.5, 0.5]
    into, away = torch.ones(1, 1, dtype=dtype), torch.ones(1, 1, dtype=dtype)
    for q in reversed(range(kin)):             # the data index is little-endian, the variant index is not
        one = torch.tensor([half, half, [1.0 - secret[q], float(secret[q])], half], dtype=dtype)
        into = torch.einsum("vx,uy->uvxy", into, one).reshape(4 * into.shape[0], 2 * into.shape[1])
    for _ in range(kout):
        away = torch.einsum("vx,uy->vuyx", away, torch.tensor([half, [1.0, 0.0], half, half], dtype=dtype)).reshape(4 * away.shape[0], 2 * away.shape[1])
    p = torch.zeros(1 << (2 * kin), 1 << (2 * kout), 1 << kout, 1 << (n - kin), 1 << kin, dtype=dtype, device="cuda")
    rest = sum(int(s) << t for t, s in enumerate(secret[kin:]))
    p[:, :, :, rest, :] = into.cuda()[:, None, None, :] * away.cuda()[None, :, :, None]
    return p.view(1 << (2 * (kin + kout)), 1 << (n + kout))


def _outputs(c, values, dtype, seed):
    """The variant outputs of every block, on the GPU, and the circuit's secret bits."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    secret = np.random.default_rng(seed).integers(0, 2, sum(_data(c)))
    probs, at = [], 0
    for n, (i, o) in zip(_data(c), _links(c)):
        if values == "bv" and n >= i:
            probs.append(_bv(i, o, n, secret[at:at + n], dtype))
        else:
            probs.append(_haar(i, o, n, gen, dtype))
        at += n
    return probs, secret


def _values(case, seed):
    """A distribution's bins: sums of many states ("narrow"), a deep random circuit's ("thomas"), one with few solutions ("peaked")."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n, dtype = case["n"], torch.float64 if case["dtype"] == "f64" else torch.float32
    if case["values"] == "narrow":
        x = torch.randn(n, dtype=dtype, device="cuda", generator=gen).mul_(0.03).add_(1.0)
    else:
        x = torch.empty(n, dtype=dtype, device="cuda").exponential_(1.0, generator=gen)
        if case["values"] == "peaked":
            x.mul_(torch.rand(n, device="cuda", generator=gen) < 1e-3)
    return x.div_(n)


def _threshold(case):
    return 1.0 / case["n"] if case["threshold"] else -math.inf


_TYPES = {"f32": torch.float32, "f64": torch.float64}


def _zoom_bits(c, seed):
    return np.random.default_rng(seed + 1).integers(0, 2, sum(_data(c)))


class _State:
    """What a program holds between its calls; a server is closed before its context."""

    def __init__(self, **kw):
        self.server = None
        self.__dict__.update(kw)

    def __del__(self):
        if self.server is not None:
            self.server.close()
        if "ctx" in self.__dict__:
            self.ctx.close()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "top":
        # any query's workspace serves: the smallest circuit there is
        ctx = Context()
        c = {"widths": "3,3", "cuts": "1"}
        q, _ = ctx.set_qubit_roles(ctx.load_subcircuit_outputs(*_graph(c), _outputs(c, "haar", torch.float32, seed)[0]), [ACTIVE] * 5)
        return _State(case=case, ctx=ctx, query=q, x=_values(case, seed), top=_top_buffers(case["k"]))
    if kind in ("step", "level"):
        ctx = Context(merge_pyramid=bool(case.get("pyramid")), slice_edges=case.get("slices", 0))
        probs, secret = _outputs(case, case["values"], _TYPES[case["inputs"]], seed)
        if case.get("host"):
            probs = [p.cpu().pin_memory() for p in probs]
        circuit = ctx.load_subcircuit_outputs(*_graph(case), probs)
        roles = _roles(case, _ints(case["zoom"]), _ints(case["active"]), secret if case["values"] == "bv" else _zoom_bits(case, seed))
        query, na = ctx.set_qubit_roles(circuit, roles)
        s = _State(case=case, ctx=ctx, probs=probs, circuit=circuit, query=query, out=torch.zeros(1 << na, dtype=_TYPES[case["out"]], device="cuda"),
                   total=torch.zeros(1, dtype=torch.float64, device="cuda"), top=_top_buffers(max(1, case["k"])), graph=None)
        if case.get("host") and not case["captured"]:
            s.read = [t.cpu().pin_memory() for t in (s.total, *s.top)]
        if case.get("captured"):
            _call(s)
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                _call(s)
            s.graph = graph
        return s
    if kind == "search":
        ctx, c = Context(), _search_chain(case)
        probs, secret = _outputs(c, case["values"], torch.float32, seed)
        circuit = ctx.load_subcircuit_outputs(*_graph(c), probs)
        torch.cuda.synchronize()
        fixed = _roles(c, _search_split(case, c)[0], [0] * case["blocks"], secret)
        return _State(case=case, ctx=ctx, circuit=circuit, graph=_graph(c), zoom=fixed)
    circuits, queries = _many(case)
    ctx = Context(merge_pyramid=case["pyramid"])
    probs = [_outputs(c, "haar", torch.float32, seed + 100 * i)[0] for i, c in enumerate(circuits)]
    ids = [ctx.load_subcircuit_outputs(*_graph(c), p) for c, p in zip(circuits, probs)]
    roles = [_roles(circuits[ci], z, a, _zoom_bits(circuits[ci], seed + j)) for j, (ci, z, a) in enumerate(queries)]
    if kind == "serve":
        torch.cuda.synchronize()
        return _State(case=case, ctx=ctx, ids=ids, circuit=[ci for ci, _, _ in queries], roles=roles, server=Server(ctx))
    qs = [ctx.set_qubit_roles(ids[ci], r)[0] for (ci, _, _), r in zip(queries, roles)]
    sizes = [1 << sum(a) for _, _, a in queries]
    flat = torch.zeros(sum(sizes), dtype=torch.float32, device="cuda")
    totals = torch.zeros(len(qs), dtype=torch.float64, device="cuda")
    return _State(case=case, ctx=ctx, ids=ids, probs=probs, flat=flat, totals=totals, batch=ctx.batch_create(qs, list(flat.split(sizes)), totals))


def _top_buffers(k):
    return (torch.zeros(k, dtype=torch.int64, device="cuda"), torch.zeros(k, dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda"))


# ---- the calls ---------------------------------------------------------------------------------

def _call(s):
    c = s.case
    if c["kind"] == "step":
        s.ctx.reconstruct_select(s.query, s.out, c["k"], probs=s.probs, precision=c["precision"], total_prob=s.total,
                                 bins_out=s.top[0], probs_out=s.top[1], n_found=s.top[2])
        return
    if c["update"]:
        s.ctx.update_subcircuit_outputs(s.circuit, s.probs)
    s.ctx.reconstruct(s.query, s.out, c["precision"], s.total if c["k"] else None)
    if c["k"]:
        s.ctx.top_bins(s.query, s.out, c["k"], -math.inf, *s.top)


def run(s):
    c = s.case
    kind = c["kind"]
    if kind in ("step", "level"):
        if s.graph is not None:
            s.graph.replay()
        else:
            _call(s)
        if "read" in s.__dict__:
            for h, t in zip(s.read, (s.total, *s.top)):
                h.copy_(t, non_blocking=True)
            torch.cuda.current_stream().synchronize()
            return [s.out, *s.read]
        return [s.out, s.total, *s.top] if c["k"] else [s.out]
    if kind == "top":
        return list(s.ctx.top_bins(s.query, s.x, c["k"], _threshold(c), *s.top))
    if kind == "batch":
        if c["update"]:
            for i, p in zip(s.ids, s.probs):
                s.ctx.update_subcircuit_outputs(i, p)
        s.ctx.batch_run(s.batch)
        return [s.flat, s.totals]
    if kind == "search":
        roles = recursion_roles(*s.graph, s.zoom, 1 << c["bins"])
        query, na = s.ctx.set_qubit_roles(s.circuit, roles)
        bins = torch.empty(1 << na, dtype=torch.float32, device="cuda")
        s.ctx.reconstruct(query, bins)
        b, v, n = s.ctx.top_bins(query, bins, min(c["k"], 1 << na), 2.0 ** -c["bins"])
        n = int(n.item())
        b, v = b[:n].cpu(), v[:n].cpu()
        s.ctx.release_query(query)
        return [bins, b, v]
    tickets = [s.server.submit(s.ids[ci], r) for ci, r in zip(s.circuit, s.roles)]
    s.server.drain()
    return [s.server.result(t) for t in tickets]


# ---- the work ----------------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind == "top":
        return {"bytes": case["n"] * (8 if case["dtype"] == "f64" else 4) + 16 * case["k"], "flops": 0}
    if kind in ("step", "level"):
        zoom, active, e = _ints(case["zoom"]), _ints(case["active"]), 8 if case["inputs"] == "f64" else 4
        moved = (8 if case["out"] == "f64" else 4) * 2.0 ** sum(active) + 16 * case["k"]
        for size, z, n, (i, o) in zip(_sizes(case), zoom, _data(case), _links(case)):
            if kind == "step":
                moved += e * 2.0 ** (size - z)                       # the kept states of the new outputs
            else:                                                    # new outputs in and their tensor out, or the kept part of it in
                moved += e * 2.0 ** size + 4.0 * 2.0 ** (size - o) if case["update"] else 4.0 * 2.0 ** (n + 2 * (i + o) - z)
        return {"bytes": moved, "flops": _chain_flops(case, active)}
    if kind == "search":
        c = _search_chain(case)
        zoom, active = _search_split(case, c)
        moved = sum(4.0 * 2.0 ** (n - z + 2 * (i + o)) for n, z, (i, o) in zip(_data(c), zoom, _links(c)))
        return {"bytes": moved + 4.0 * 2.0 ** sum(active), "flops": _chain_flops(c, active)}
    circuits, queries = _many(case)
    moved = flops = 0.0
    for c in circuits:
        tensors = sum(4.0 * 2.0 ** (size - o) for size, (_, o) in zip(_sizes(c), _links(c)))
        moved += tensors + (sum(4.0 * 2.0 ** size for size in _sizes(c)) if case.get("update") else 0)
    for ci, _, active in queries:
        moved += 4.0 * 2.0 ** sum(active)
        flops += _chain_flops(circuits[ci], active)
    return {"bytes": moved, "flops": flops}


# ---- the values in 64 bits ---------------------------------------------------------------------

_D = [[1.0, 1.0, 0.0, 0.0], [-1.0, -1.0, 2.0, 0.0], [-1.0, -1.0, 0.0, 2.0], [1.0, -1.0, 0.0, 0.0]]
_W = [[1.0, 1.0], [1.0, -1.0], [1.0, -1.0], [1.0, -1.0]]


def _attributed(p, kin, kout, n):
    """Eq. 1's tensor [4^k, 2^n] of one block's outputs."""
    t = p.cuda().double()
    d, w = torch.tensor(_D, dtype=torch.float64, device="cuda"), torch.tensor(_W, dtype=torch.float64, device="cuda")
    for q in range(kin):
        t = torch.einsum("es,lsr->ler", d, t.reshape(4 ** q, 4, -1))
    for u in range(kout):      # digit u of the outgoing edges, outcome bit u: the lowest one left
        t = t.reshape(4 ** (kin + u), 4, 4 ** (kout - 1 - u), 2 ** (kout - 1 - u), 2, 1 << n)
        t = torch.einsum("lemhcx,ec->lemhx", t, w)
    return t.reshape(4 ** (kin + kout), 1 << n)


def _bins(c, tensors, roles):
    """All bins of a query from the blocks' tensors, block after block."""
    at, scale, res = 0, 1.0, torch.ones(1, 1, dtype=torch.float64, device="cuda")      # [bins so far, open edges]
    for t, n, (i, o) in zip(tensors, _data(c), _links(c)):
        mine = roles[at:at + n]
        at += n
        for q in reversed(range(n)):       # the highest data qubit first: the front of the remaining index
            if mine[q] == MERGED:
                t = t.reshape(t.shape[0], -1, 2, 1 << q).sum(2)
            elif mine[q] != ACTIVE:
                t = t.reshape(t.shape[0], -1, 2, 1 << q)[:, :, int(mine[q] == ZOOM1)]
            t = t.reshape(t.shape[0], -1)
        a = t.reshape(4 ** i, 4 ** o, -1)
        bins = a.shape[2]
        res = res @ a.reshape(4 ** i, -1)                                              # [bins, (edges out, own bins)]
        res = res.reshape(-1, 4 ** o, bins).permute(2, 0, 1).reshape(-1, 4 ** o)
        scale *= 2.0 ** -i
    return res.reshape(-1) * scale


def _all_attributed(c, probs):
    return [_attributed(p, i, o, n) for p, n, (i, o) in zip(probs, _data(c), _links(c))]


def exact(case, seed):
    kind = case["kind"]
    if kind == "top":
        x = _values(case, seed)
        best = x.topk(min(case["k"], x.numel())).values.double()
        best = best[best >= _threshold(case)]
        return [None, torch.cat([best, best.new_zeros(case["k"] - best.numel())]), None]
    if kind in ("step", "level"):
        probs, secret = _outputs(case, case["values"], _TYPES[case["inputs"]], seed)
        roles = _roles(case, _ints(case["zoom"]), _ints(case["active"]), secret if case["values"] == "bv" else _zoom_bits(case, seed))
        bins = _bins(case, _all_attributed(case, probs), roles)
        return [bins, bins.sum().reshape(1), None, bins.topk(case["k"]).values, None] if case["k"] else [bins]
    if kind == "search":
        c = _search_chain(case)
        probs, secret = _outputs(c, case["values"], torch.float32, seed)
        bins = _bins(c, _all_attributed(c, probs), _roles(c, *_search_split(case, c), secret))
        best = bins.topk(min(case["k"], bins.numel())).values
        return [bins, None, best[best >= 2.0 ** -case["bins"]]]
    circuits, queries = _many(case)
    tensors = [_all_attributed(c, _outputs(c, "haar", torch.float32, seed + 100 * i)[0]) for i, c in enumerate(circuits)]
    found = [_bins(circuits[ci], tensors[ci], _roles(circuits[ci], z, a, _zoom_bits(circuits[ci], seed + j))) for j, (ci, z, a) in enumerate(queries)]
    if kind == "serve":
        return found
    return [torch.cat(found), torch.stack([f.sum() for f in found])]
