"""The workloads this library is timed on: what a serving process has it do, through its Python entry points.

A process keeps one graph with its cached embeddings resident (`Ripple`) and applies batches of updates as they
arrive (`apply_batch`), reading the ids of the vertices whose output changed and the embedding rows after each; now
and then it recomputes everything (`recompute_full`: after loading new features or weights, or as a safety net).  The
listed cases are the graph shapes, models and batch sizes of `paper_2601_12347_b200.inputs.workloads()`; `draw` spreads
sizes, widths, models, batch sizes and the memory the batches arrive in over the ranges between them.

Graphs are R-MAT (a = .57, b = c = .19), generated on the GPU.  A state holds a short stream of batches followed by
their inverses (additions become deletions and back, feature rows return to what they were) in reverse order, so that
the stream can be replayed without end and every batch does its full work each time; a pass applies the next batch.
"""
import math

import numpy as np
import torch

from paper_2601_12347_b200 import inputs as I
from paper_2601_12347_b200 import ripple

_SPARSE = {"vertices": 169_343, "edges": 1_166_243}      # a citation graph's counts
_DENSE = {"vertices": 2_449_029, "edges": 123_718_280}   # a product graph's counts
_ULTRA = {"vertices": 232_965, "edges": 114_900_000}     # a social network's counts: average degree 493

_QUAD = ((0.57, 0.19), (0.19, 0.05))                     # quadrant probabilities [source bit][sink bit]
_MIX = (0.4, 0.4, 0.2)                                   # edge additions, edge deletions, feature replacements
_WSUM = ("gcw",)


def _case(name, graph, model, widths, batch, arrives, vertex_deletions=0):
    c = {"model": model, "layers": len(widths) - 1, "d_in": widths[0], "hidden": widths[1], "d_out": widths[-1],
         "batch": batch, "arrives": arrives, "vertex_deletions": vertex_deletions}
    c.update(graph)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one update at a time, applied the moment it arrives: nothing but latency
        _case("sparse-sage-b1", _SPARSE, "sage", (128, 256, 40), 1, "numpy"),
        # a handful of updates on a graph whose edges carry weights
        _case("sparse-weighted-b10", _SPARSE, "gcw", (128, 256, 40), 10, "numpy"),
        # all five kinds of update, two vertex deletions among them
        _case("sparse-sage-vdel-b100", _SPARSE, "sage", (128, 256, 40), 100, "numpy", 2),
        # three layers: a small batch reaches half of the graph
        _case("sparse-gin3-b100", _SPARSE, "gin", (128, 256, 256, 256), 100, "numpy"),
        _case("sparse-gcn3-b1000", _SPARSE, "gcn", (128, 256, 256, 40), 1000, "pinned"),
        # max aggregation: value-based, pruned propagation
        _case("sparse-max-b1000", _SPARSE, "max", (128, 256, 40), 1000, "pinned"),
        # the large graph: a small batch, the benchmark's batch, and a large one that already sits on the device
        _case("dense-sage-b10", _DENSE, "sage", (100, 256, 47), 10, "pinned"),
        _case("dense-sage-b1000", _DENSE, "sage", (100, 256, 47), 1000, "pinned"),
        # three layers on the large graph: every hop but the first touches most of it
        _case("dense-sage3-b1000", _DENSE, "sage", (100, 256, 256, 47), 1000, "device"),
        # attention layers
        _case("dense-attention-b1000", _DENSE, "gat", (100, 100, 100), 1000, "pinned"),
        # hundreds of in-neighbours per vertex, wide features
        _case("ultra-sage-b100", _ULTRA, "sage", (602, 256, 41), 100, "device"),
        # everything from scratch
        _case("dense-sage-full", _DENSE, "sage", (100, 256, 47), 0, "none"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    top = work(_case("", _DENSE, "sage", (100, 256, 256, 47), 1000, "device"))
    while True:
        n = _log_uniform(rng, 2_000, _DENSE["vertices"])
        e = min(int(n * math.exp(rng.uniform(math.log(4.0), math.log(60.0 if n > 240_000 else 500.0)))),
                _DENSE["edges"], n * n // 40)
        model = rng.choice(("sage", "sage", "sage", "gcn", "gcw", "gin", "max", "gat"))
        layers = rng.choice((2, 2, 3))
        d0 = rng.choice((32, 100, 128, rng.randint(17, 256), 602 if n <= 240_000 else 100))
        hidden = rng.choice((32, 64, 128, 256, rng.randint(24, 256)))
        widths = [d0] + [hidden] * (layers - 1) + [rng.choice((16, 40, 41, 47, rng.randint(5, 120)))]
        if model == "gin":
            widths = [d0] + [hidden] * layers
        if model == "gat":
            widths = [min(d0, 256)] * (layers + 1)
        if rng.random() < 0.12:
            batch, arrives, vdel = 0, "none", 0
        else:
            batch = min(_log_uniform(rng, 1, 10_000), max(1, n // 40), max(1, e // 40))
            arrives = rng.choice(("numpy", "numpy", "pinned", "device"))
            vdel = rng.choice((0, 0, 0, max(1, batch // 50))) if 20 <= batch <= 1000 and n >= 20_000 and e <= 20 * n else 0
        c = _case("", {"vertices": n, "edges": e}, model, widths, batch, arrives, vdel)
        w = work(c)
        # no larger than the largest listed ones, in bytes, in arithmetic and in rows moved along edges
        if w["bytes"] <= top["bytes"] and w["flops"] <= top["flops"] and n * max(widths) <= 2_449_029 * 256:
            return c


# ---- inputs ------------------------------------------------------------------------------------------------------
def _rmat_keys(n, e, gen):
    """e distinct pairs u * n + v (u != v), ascending."""
    scale = max(1, math.ceil(math.log2(n)))
    a, b, c = _QUAD[0][0], _QUAD[0][1], _QUAD[1][0]
    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    got_per_draw = 0.7
    while keys.numel() < e:
        need = int((e - keys.numel()) / max(got_per_draw, 0.02) * 1.04) + 4096
        parts = [keys]
        for lo in range(0, need, 1 << 25):
            m = min(1 << 25, need - lo)
            u = torch.zeros(m, dtype=torch.int32, device="cuda")
            v = torch.zeros(m, dtype=torch.int32, device="cuda")
            for _ in range(scale):
                r = torch.rand(m, device="cuda", generator=gen)
                u.mul_(2).add_(r >= a + b)
                v.mul_(2).add_(((r >= a) & (r < a + b)) | (r >= a + b + c))
            ok = (u < n) & (v < n) & (u != v)
            parts.append(u[ok].to(torch.int64) * n + v[ok])
        before = keys.numel()
        keys = torch.unique(torch.cat(parts))
        got_per_draw = max(keys.numel() - before, 1) / need
    if keys.numel() > e:
        drop = _distinct(keys.numel(), keys.numel() - e, gen)
        keep = torch.ones(keys.numel(), dtype=torch.bool, device="cuda")
        keep[drop] = False
        keys = keys[keep]
    return keys


def _distinct(n, k, gen):
    """k distinct numbers below n, in random order."""
    if k * 4 > n:
        return torch.randperm(n, device="cuda", generator=gen)[:k]
    x = torch.empty(0, dtype=torch.int64, device="cuda")
    while x.numel() < k:
        x = torch.unique(torch.cat([x, torch.randint(n, (2 * (k - x.numel()) + 64,), device="cuda", generator=gen)]))
    return x[torch.randperm(x.numel(), device="cuda", generator=gen)[:k]]


def _model(c):
    w = [c["d_in"]] + [c["hidden"]] * (c["layers"] - 1) + [c["d_out"]]
    kind = c["model"]
    if kind == "sage":
        return I.sage_model(w)
    if kind == "gcn":
        return I.graphconv_model(w, I.AGG_WSUM_GCN)
    if kind == "gcw":
        return I.graphconv_model(w, I.AGG_WSUM_EDGE)
    if kind == "max":
        return I.graphconv_model(w, I.AGG_MAX)
    if kind == "gin":
        return I.gin_model(c["d_in"], c["hidden"], c["layers"])
    return I.gat_model(c["d_in"], c["layers"], d_att=8, slope=0.2)


def _stream(c, keys, perm, feats, weights, gen):
    """A few forward batches, then their inverses in reverse order: host arrays (ups, rows, op_weights)."""
    n, b = c["vertices"], c["batch"]
    count = max(2, min(16, 200 // b))
    total = count * b
    kinds = torch.multinomial(torch.tensor(_MIX, device="cuda"), total, replacement=True, generator=gen)
    gone = torch.empty(0, dtype=torch.int64, device="cuda")
    if c["vertex_deletions"]:
        # deleted vertices: no operation of the stream but the edges that go with them names them
        at = (torch.arange(count, device="cuda")[:, None] * b + torch.arange(c["vertex_deletions"], device="cuda") * 7).flatten()
        kinds[at] = 3
        gone = _distinct(n, at.numel(), gen)
    n_add, n_del, n_feat = (int((kinds == k).sum()) for k in range(3))
    # additions: uniform pairs that are not edges; deletions: uniform over the edges; features: uniform vertices
    cand = torch.randint(n * n, (2 * n_add + 256,), device="cuda", generator=gen)
    pos = torch.searchsorted(keys, cand).clamp_(max=keys.numel() - 1)
    ok = (keys[pos] != cand) & (cand // n != cand % n) & ~torch.isin(cand // n, gone) & ~torch.isin(cand % n, gone)
    cand = torch.unique(cand[ok])
    add = cand[torch.randperm(cand.numel(), device="cuda", generator=gen)[:n_add]]
    live = _distinct(keys.numel(), min(2 * n_del + 64, keys.numel()), gen)
    if gone.numel():
        live = live[~torch.isin(keys[live] // n, gone) & ~torch.isin(keys[live] % n, gone)]
    dele = live[:n_del]
    feat = _distinct(n, min(n_feat + 4 * gone.numel(), n), gen)
    feat = feat[~torch.isin(feat, gone)][:n_feat]
    new_rows = torch.randn(n_feat, c["d_in"], device="cuda", generator=gen)
    ups = torch.zeros(total, 3, dtype=torch.int64, device="cuda")
    ups[:, 0] = kinds
    for k, pairs in ((0, add), (1, keys[dele])):
        ups[kinds == k, 1], ups[kinds == k, 2] = perm[pairs // n], perm[pairs % n]
    fv = perm[feat]
    ups[kinds == 2, 1] = fv
    if gone.numel():
        ups[kinds == 3, 1] = perm[gone]
    opw = torch.empty(total, device="cuda").uniform_(0.1, 1.0, generator=gen)
    undo_w = opw.clone()
    if weights is not None:
        undo_w[kinds == 1] = weights[dele]
    old_rows, lost = feats[fv], feats[perm[gone]] if gone.numel() else None
    lost_edges = None
    if gone.numel():
        touching = torch.isin(keys // n, gone) | torch.isin(keys % n, gone)
        lost_edges = torch.stack([keys[touching] // n, keys[touching] % n], 1)
    host = lambda t: t.cpu().numpy()  # noqa: E731
    U, new_h, old_h, W, UW, G, P = host(ups), host(new_rows), host(old_rows), host(opw), host(undo_w), host(gone), host(perm)
    lost_h = host(lost) if lost is not None else None
    le = host(lost_edges) if lost_edges is not None else None
    rank = np.cumsum(U[:, 0] == 2) - 1
    vrank = np.cumsum(U[:, 0] == 3) - 1
    order = {int(g): i for i, g in enumerate(G)}
    if le is not None:      # an edge between two deleted vertices goes with the one that is deleted first
        who = np.array([min(order.get(int(u), 1 << 30), order.get(int(v), 1 << 30)) for u, v in le])
    forward, inverse = [], []
    for i in range(count):
        s = slice(i * b, (i + 1) * b)
        u = U[s]
        f = np.zeros(b, dtype=I.UPDATE_DTYPE)
        f["op"], f["u"], f["v"] = u[:, 0], u[:, 1], u[:, 2]
        isf = f["op"] == I.OP_SET_FEATURE
        f["v"][isf] = np.arange(int(isf.sum()))
        g = f.copy()
        g["op"] = np.array([I.OP_DEL_EDGE, I.OP_ADD_EDGE, I.OP_SET_FEATURE, I.OP_SET_FEATURE])[f["op"]]
        rows_f, rows_g = new_h[rank[s][isf]], old_h[rank[s][isf]]
        wg = UW[s]
        isd = f["op"] == I.OP_DEL_VERTEX
        if isd.any():       # its feature row and its edges come back
            g["v"][isd] = rows_g.shape[0] + np.arange(int(isd.sum()))
            rows_g = np.concatenate([rows_g, lost_h[vrank[s][isd]]])
            back = le[(who >= vrank[s][isd].min()) & (who <= vrank[s][isd].max())]
            more = np.zeros(back.shape[0], dtype=I.UPDATE_DTYPE)
            more["op"], more["u"], more["v"] = I.OP_ADD_EDGE, P[back[:, 0]], P[back[:, 1]]
            g = np.concatenate([g, more])
            wg = np.concatenate([wg, np.ones(back.shape[0], np.float32)])
        forward.append((f, np.ascontiguousarray(rows_f), W[s].copy()))
        inverse.append((np.ascontiguousarray(g), np.ascontiguousarray(rows_g), np.ascontiguousarray(wg, dtype=np.float32)))
    return forward + inverse[::-1]


def _arrive(batch, how, weighted):
    ups, rows, w = batch
    if how != "numpy":
        ups = torch.from_numpy(np.stack([ups["op"], ups["u"], ups["v"]], axis=1).astype(np.int32))
        rows, w = torch.from_numpy(rows), torch.from_numpy(w)
        ups, rows, w = (t.pin_memory() if how == "pinned" else t.cuda() for t in (ups, rows, w))
    return (ups, rows, w) if weighted else (ups, rows)


def prepare(case, seed):
    """The resident graph with its cached embeddings, and a stream of batches where it receives them."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    n = case["vertices"]
    keys = _rmat_keys(n, case["edges"], gen)
    perm = torch.randperm(n, device="cuda", generator=gen)
    feats = torch.randn(n, case["d_in"], device="cuda", generator=gen)
    weighted = case["model"] in _WSUM
    weights = torch.empty(keys.numel(), device="cuda").uniform_(0.1, 1.0, generator=gen) if weighted else None
    batches = _stream(case, keys, perm, feats, weights, gen) if case["batch"] else []
    order = torch.randperm(keys.numel(), device="cuda", generator=gen)
    perm32 = perm.to(torch.int32)
    src, dst = perm32[keys // n][order], perm32[keys % n][order]
    if weighted:
        weights = weights[order]
    del keys, order
    model = _model(case)
    most = max([b[0].size for b in batches] + [1])
    rp = ripple.Ripple(n, src, dst, feats, model, I.make_weights(model, int(seed) % 65536, zero_bias=False),
                       max_batch=65536 if case["vertex_deletions"] else max(16384, most), edge_weights=weights)
    return {"rp": rp, "batches": [_arrive(b, case["arrives"], weighted) for b in batches], "next": 0,
            "layers": case["layers"], "by_structure": case["model"] != "max"}


def run(state):
    """The next batch of the stream (or everything from scratch), then what a reader takes: the embeddings of every
    layer, the ids whose output changed, the degrees.  The list of ids is as long as the batch makes it, so its length
    stands for it.  (With max aggregation it depends on values, and two correct implementations may differ in a
    vertex on a tie: there it is read, but not compared.)"""
    rp, layers = state["rp"], range(1, state["layers"] + 1)
    if not state["batches"]:
        rp.recompute_full()
        return {"embeddings": [rp.embeddings(l) for l in layers]}
    i = state["next"]
    state["next"] = (i + 1) % len(state["batches"])
    rp.apply_batch(*state["batches"][i])
    changed = rp.affected(state["layers"])
    out = {"embeddings": [rp.embeddings(l) for l in layers], "degrees": rp.degrees()}
    if state["by_structure"]:
        out["changed"] = changed.numel()
    return out


# ---- what a pass cannot do without -------------------------------------------------------------------------------
def _reach(n, e):
    """The generator's own edge probabilities, by popcount class of the ids: class sizes, and for a sender
    probability per class the mean number of senders among a vertex's in-neighbours."""
    s = max(1, math.ceil(math.log2(n)))
    cnt = np.zeros(s + 1)
    ones = 0
    for bit in range(s, -1, -1):          # ids below n, by number of set bits
        if n >> bit & 1:
            for k in range(bit + 1):
                if ones + k <= s:
                    cnt[ones + k] += math.comb(bit, k)
            ones += 1
    share = cnt / np.array([math.comb(s, k) for k in range(s + 1)])
    (a, b), (c, d) = _QUAD
    many = np.zeros((s + 1, s + 1, s + 1))  # [sink class j][ones of the source under j's zeros][ under its ones]
    prob = np.zeros_like(many)
    cls = np.zeros(many.shape, dtype=int)
    for j in range(s + 1):
        for x in range(s - j + 1):
            for y in range(j + 1):
                many[j, x, y] = math.comb(s - j, x) * math.comb(j, y)
                prob[j, x, y] = a ** (s - j - x) * c ** x * b ** (j - y) * d ** y
                cls[j, x, y] = x + y
    many = many * share[cls]
    lo, hi = e * 0.5, e * 1e4
    for _ in range(60):
        mid = math.sqrt(lo * hi)
        got = float((cnt[:, None, None] * many * -np.expm1(-mid * prob)).sum())
        lo, hi = (mid, hi) if got < e else (lo, mid)
    pair = many * -np.expm1(-lo * prob)
    return cnt, lambda p: (pair * p[cls]).sum(axis=(1, 2))


def work(case):
    n, e, L, b = case["vertices"], case["edges"], case["layers"], case["batch"]
    kind = case["model"]
    d = [case["d_in"]] + [case["hidden"]] * (L - 1) + [case["d_out"]]
    self_term, weighted = kind in ("sage", "gin", "gat"), kind in _WSUM
    hidden = case["hidden"]
    byts = flops = 0.0

    def width(l):     # a linear layer that narrows may be applied before the sum
        to = hidden if kind == "gin" else d[l]
        return d[l - 1] if kind in ("max", "gat") else min(d[l - 1], to)

    def matrices(l, senders, rows):
        if kind == "gat":
            return 4.0 * d[l - 1] * senders + 2.0 * d[l] * rows
        if kind == "gin":
            first = 2.0 * d[l - 1] * hidden * (min(senders, rows) if width(l) < d[l - 1] else rows)
            return first + 2.0 * hidden * d[l] * rows
        product = 2.0 * d[l - 1] * d[l]
        nb = product * (min(senders, rows) if width(l) < d[l - 1] else rows)
        return nb + (product * min(senders, rows) if kind == "sage" else 0.0)

    if not b:         # every edge once per layer, every cached row written, the layer before read
        for l in range(1, L + 1):
            byts += e * (8.0 if weighted else 4.0) + 4.0 * n * (d[l - 1] + width(l) + d[l])
            flops += 2.0 * e * width(l) + matrices(l, n, n)
        return {"bytes": byts, "flops": flops}
    cnt, hits = _reach(n, e)
    indeg = hits(np.ones(cnt.size))       # (the generator is symmetric: also the out-degree)
    gone = case["vertex_deletions"]
    add, dele, feat = (m * (b - gone) for m in _MIX)
    edges = dele + gone * 2.0 * e / n
    touched = 1.0 - np.exp(-(add / n + edges * indeg / e))    # end points of changed edges
    p = np.full(cnt.size, min(1.0, (feat + gone) / n))
    byts += 12.0 * b + feat * 8.0 * d[0] + 16.0 * (add + edges)
    for l in range(1, L + 1):
        senders = 1.0 - (1.0 - p) * (1.0 - touched) if kind == "gcn" else p
        nC, msgs = float((cnt * senders).sum()), float((cnt * senders * indeg).sum()) + add + edges
        q = 1.0 - (1.0 - touched) * np.exp(-hits(senders)) * ((1.0 - p) if self_term else 1.0)
        if kind == "max":                 # half of the sinks of a message keep their maximum
            q = 0.5 * q
        rows, w = float((cnt * q).sum()), width(l)
        byts += 4.0 * nC * (d[l - 1] + 2.0 * w) + msgs * (8.0 if weighted else 4.0)
        byts += 4.0 * rows * (2.0 * w + d[l] + (d[l] if kind == "sage" else 0.0) + 1.0)
        flops += 2.0 * msgs * w + matrices(l, nC, rows)
        p = q
    return {"bytes": byts, "flops": flops}


def tolerance(case):
    """Sums of single-precision terms in another order; degrees and counts are whole numbers and equal."""
    return {"rel": 1e-5, "differ": 0.0}
