"""Parity of the CUDA path for attention layers (Sec. 3.4.1, Eq. 3) against the oracle's
hybrid-incremental route: graph, hop sets and counters bit-exact after every batch; embeddings within
1e-4 (1 + |ref|) of the oracle's full recomputation; the cached numerator / denominator rows within
the same bound scaled by sqrt(in-degree) (they are fp32 sums of that many terms)."""
import numpy as np
import pytest

from paper_2601_12347_b200 import inputs as I
from tolerances import TOL

import test_gpu_parity as G

pytestmark = pytest.mark.gpu

env = G.env


def cached_rows(orc, L):
    """[numerator | denominator] per layer, as the library lays them out."""
    return [None] + [np.concatenate([orc.S(l), orc.Den(l)[:, None]], axis=1) for l in range(1, L + 1)]


def check_graph(rp, orc):
    rowptr, col = rp.export_graph()
    orp, ocol = orc.export_csr()
    assert np.array_equal(rowptr, orp) and np.array_equal(col, ocol)


def hub_graph(n, m, seed):
    src, dst = I.er_graph(n, m, seed)
    have = set(zip(src.tolist(), dst.tolist()))
    extra = [(0, int(v)) for v in range(1, 400) if (0, int(v)) not in have]        # a long out-list
    extra += [(int(u), 9) for u in range(100, 700) if (int(u), 9) not in have]      # and a long in-list (3 chunks)
    src = np.concatenate([src, np.array([a for a, _ in extra], dtype=np.int32)])
    dst = np.concatenate([dst, np.array([b for _, b in extra], dtype=np.int32)])
    return src, dst


MODELS = {
    "d18_2l": dict(d=18, n_layers=2, d_att=8, slope=1.0),
    "d18_3l_leaky": dict(d=18, n_layers=3, d_att=8, slope=0.2),
    "d64_2l_leaky": dict(d=64, n_layers=2, d_att=16, slope=0.2),
    "d130_2l": dict(d=130, n_layers=2, d_att=4, slope=0.2),       # the denominator shares the last 16-byte piece of the row
    "d300_2l_relu": dict(d=300, n_layers=2, d_att=8, slope=0.2, act=I.ACT_RELU),
}


@pytest.mark.parametrize("name", list(MODELS.keys()))
def test_small_graphs_every_batch(env, name):
    ripple, Oracle = env
    model = I.gat_model(**MODELS[name])
    L = len(model.layers)
    n = 900
    src, dst = hub_graph(n, 7000, 3)
    X = I.features(n, model.dims[0], 3)
    W = I.make_weights(model, 3)
    rp = ripple.Ripple(n, src, dst, X, model, W, slack=0.05)
    orc = Oracle(n, src, dst, X, model, W)
    G.check_values(rp, orc.full(), L, cached_rows(orc, L))
    stream = I.UpdateStream(n, src, dst, model.dims[0], 3, mix=(0.45, 0.35, 0.18, 0.02))
    for b, bs in enumerate([1, 1, 2, 7, 33, 100, 1, 250, 64, 5] * 2):
        ups, rows = stream.next_batch(bs)
        rp.apply_batch(ups, rows)
        assert orc.apply_incremental(ups, rows) == 0
        check_graph(rp, orc)
        G.check_frontiers(rp, orc, L)
        if b % 3 == 2:
            G.check_values(rp, orc.full(), L, cached_rows(orc, L))
    G.check_values(rp, orc.full(), L, cached_rows(orc, L))
    rp.close()


def test_single_updates_of_each_kind(env):
    ripple, Oracle = env
    model = I.gat_model(20, 2, d_att=8, slope=0.2)
    n, src, dst, X, _, _ = G._small(seed=41)
    X = I.features(n, 20, 41)
    W = I.make_weights(model, 41)
    rp = ripple.Ripple(n, src, dst, X, model, W)
    orc = Oracle(n, src, dst, X, model, W)
    have = set(zip(src.tolist(), dst.tolist()))
    missing = next((a, b) for a in range(n) for b in range(n) if a != b and (a, b) not in have)
    row = I.features(1, 20, 77)
    cases = [
        (G.ups_array([(I.OP_ADD_EDGE, missing[0], missing[1])]), None),
        (G.ups_array([(I.OP_DEL_EDGE, int(src[5]), int(dst[5]))]), None),
        (G.ups_array([(I.OP_SET_FEATURE, int(src[7]), 0)]), row),
        (G.ups_array([(I.OP_DEL_VERTEX, int(dst[11]), 0)]), None),
        (G.ups_array([(I.OP_SET_FEATURE, int(src[9]), 0), (I.OP_DEL_EDGE, int(src[9]), int(dst[9])),
                      (I.OP_ADD_EDGE, int(dst[9]), int(src[9]))]), row),
        (np.zeros(0, dtype=I.UPDATE_DTYPE), None),
    ]
    for ups, rows in cases:
        rp.apply_batch(ups, rows)
        assert orc.apply_incremental(ups, rows) == 0
        check_graph(rp, orc)
        G.check_frontiers(rp, orc, 2)
        G.check_values(rp, orc.full(), 2, cached_rows(orc, 2))
    rp.close()


def test_rows_outside_the_hop_sets_keep_their_bits(env):
    ripple, Oracle = env
    model = I.gat_model(24, 3, d_att=8, slope=0.2)
    n = 3000
    src, dst = I.er_graph(n, 9000, 8)
    X = I.features(n, 24, 8)
    W = I.make_weights(model, 8)
    rp = ripple.Ripple(n, src, dst, X, model, W)
    stream = I.UpdateStream(n, src, dst, 24, 8)
    for _ in range(4):
        before = [rp.embeddings(l).clone() for l in range(4)]
        ups, rows = stream.next_batch(3)
        rp.apply_batch(ups, rows)
        for l in range(4):
            keep = np.setdiff1d(np.arange(n), rp.affected(l).cpu().numpy())
            assert bool((rp.embeddings(l)[keep] == before[l][keep]).all())
    rp.close()


def test_long_stream_stays_within_tolerance_and_budget_gathers_rows_anew(env):
    ripple, Oracle = env
    model = I.gat_model(32, 2, d_att=8, slope=0.2)
    n = 1500
    src, dst = hub_graph(n, 12000, 5)
    X = I.features(n, 32, 5)
    W = I.make_weights(model, 5)
    rebuilt = {}
    for budget in (0.0, 1.5):     # the default, and one so tight that rows come due within the stream
        rp = ripple.Ripple(n, src, dst, X, model, W, rebuild_budget=budget)
        orc = Oracle(n, src, dst, X, model, W)
        stream = I.UpdateStream(n, src, dst, 32, 5)
        total = 0
        for b in range(60):
            ups, rows = stream.next_batch(40)
            rp.apply_batch(ups, rows)
            assert orc.apply_incremental(ups, rows) == 0
            total += sum(rp.stats()["rows_rebuilt"])
            if b % 20 == 19:
                G.check_frontiers(rp, orc, 2)
                G.check_values(rp, orc.full(), 2, cached_rows(orc, 2))
        rebuilt[budget] = total
        rp.close()
    assert rebuilt[1.5] > 0 and rebuilt[1.5] > rebuilt[0.0]


def test_recompute_full_and_device_resident_inputs(env):
    import torch
    ripple, Oracle = env
    model = I.gat_model(16, 2, d_att=4, slope=1.0)
    n, m = 500, 4000
    src, dst = I.er_graph(n, m, 9)
    X = I.features(n, 16, 9)
    W = I.make_weights(model, 9)
    rp = ripple.Ripple(n, torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), torch.from_numpy(X).cuda(), model, W)
    orc = Oracle(n, src, dst, X, model, W)
    stream = I.UpdateStream(n, src, dst, 16, 9)
    for _ in range(6):     # the same size again and again: the launch chain is captured and replayed
        ups, rows = stream.next_batch(50)
        dev_ups = torch.from_numpy(np.stack([ups["op"], ups["u"], ups["v"]], axis=1).astype(np.int32)).cuda()
        rp.apply_batch(dev_ups, torch.from_numpy(rows).cuda())
        assert orc.apply_incremental(ups, rows) == 0
        G.check_frontiers(rp, orc, 2)
    G.check_values(rp, orc.full(), 2, cached_rows(orc, 2))
    rp.recompute_full()
    G.check_values(rp, orc.full(), 2, cached_rows(orc, 2))
    rp.close()


def test_bad_attention_layers_are_refused(env):
    ripple, Oracle = env
    n, src, dst, X, _, _ = G._small(seed=41)
    X = I.features(n, 12, 1)
    model = I.gat_model(12, 2, d_att=4)
    W = I.make_weights(model, 1)
    model.agg = I.AGG_MEAN
    with pytest.raises(Exception):
        ripple.Ripple(n, src, dst, X, model, W)
    model = I.gat_model(12, 2, d_att=4)
    model.layers[1].d_out = 8
    with pytest.raises(Exception):
        ripple.Ripple(n, src, dst, X, model, I.make_weights(I.gat_model(12, 2, d_att=4), 1))


@pytest.mark.parametrize("d", [44, 45, 46, 47, 48, 129, 131, 132])
def test_overflowed_weights_stay_visible(env, d):
    """A logit beyond the range of exp in fp32 gives an infinite weight and an infinite denominator: the rows it reaches are
    NaN whatever the width, in a whole-graph pass and in rows recomputed by a batch, and all others are as ever."""
    ripple, _ = env
    n = 400
    src, dst = I.er_graph(n, 2400, 9)
    model = I.gat_model(d, 1)
    W = I.make_weights(model, 9)
    W[0]["bb"] = np.zeros_like(W[0]["bb"])                    # the source alone decides
    q = W[0]["Wa"].astype(np.float64) @ W[0]["ba"].astype(np.float64)
    X = I.features(n, d, 9)
    huge = (300.0 * q / float(q @ q)).astype(np.float32)     # s_u = 300: exp overflows in fp32
    X[5] = huge
    rp = ripple.Ripple(n, src, dst, X, model, W)
    reached = np.zeros(n, dtype=bool)
    reached[dst[src == 5]] = True
    assert reached.any() and not reached.all()
    H = rp.embeddings(1).cpu().numpy()
    assert np.isnan(H[reached]).all() and np.isfinite(H[~reached]).all()
    ups = np.zeros(1, dtype=I.UPDATE_DTYPE)
    ups["op"], ups["u"], ups["v"] = I.OP_SET_FEATURE, 6, 0
    rp.apply_batch(ups, huge[None])
    reached[dst[src == 6]] = True
    H = rp.embeddings(1).cpu().numpy()
    assert np.isnan(H[reached]).all() and np.isfinite(H[~reached]).all()
    rp.close()


@pytest.mark.parametrize("edges, d", [(0, 18), (2_500_000, 18), (4_900_000, 18), (4_900_000, 130)])   # pieces of 128, 256, 512 entries
def test_rows_gathered_anew_at_the_edges_of_their_pieces(env, edges, d):
    """In-lists around a window (128) and the piece of a recomputation, in a whole-graph pass and in batches whose rounding
    budget is so tight that every row they reach comes due."""
    ripple, Oracle = env
    lengths = (1, 2, 31, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 1600)
    rng = np.random.default_rng(7)
    pool = 3200
    n = pool + len(lengths)
    src = [rng.choice(pool, k, replace=False) for k in lengths]
    dst = [np.full(k, pool + i) for i, k in enumerate(lengths)]
    if edges:       # among the pool: more edges make longer pieces
        a, b = I.er_graph(pool, edges, 5)
        src, dst = src + [a], dst + [b]
    src, dst = np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32)
    model = I.gat_model(d, 1, d_att=8, slope=0.2)
    size = np.float32(np.sqrt(18 / d))     # (logits of order one at either width: the sums' bound knows nothing of the weights' size)
    X = size * I.features(n, d, 5)
    W = I.make_weights(model, 5)
    rp = ripple.Ripple(n, src, dst, X, model, W, rebuild_budget=1e-3)
    orc = Oracle(n, src, dst, X, model, W)
    G.check_values(rp, orc.full(), 1, cached_rows(orc, 1))
    for b in range(2):
        us = np.unique([s[rng.integers(s.size)] for s in np.split(src[:sum(lengths)], np.cumsum(lengths)[:-1])])
        ups = np.zeros(us.size, dtype=I.UPDATE_DTYPE)
        ups["op"], ups["u"], ups["v"] = I.OP_SET_FEATURE, us, np.arange(us.size)
        rows = size * rng.standard_normal((us.size, d)).astype(np.float32)
        rp.apply_batch(ups, rows)
        assert orc.apply_incremental(ups, rows) == 0
        assert rp.stats()["rows_rebuilt"][1] >= len(lengths)
        G.check_frontiers(rp, orc, 1)
        G.check_values(rp, orc.full(), 1, cached_rows(orc, 1))
    rp.close()
