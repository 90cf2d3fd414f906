"""The edges of the kernels' tiles and of the dispatch between their forms, against the oracle: graph, affected sets and
counters exact, embeddings within 1e-4 (1 + |ref|) and cached aggregates within the same bound scaled by sqrt(in-degree)
(GIN stacks: plus GIN_ROW_SLACK of the row's largest entry), as in test_gpu_parity."""
import numpy as np
import pytest

from paper_2601_12347_b200 import inputs as I
from tolerances import GIN_ROW_SLACK

import test_gpu_parity as G

pytestmark = pytest.mark.gpu

env = G.env


def feature_batch(n, ids, dim, seed):
    ups = G.ups_array([(I.OP_SET_FEATURE, int(u), i) for i, u in enumerate(ids)])
    return ups, I.features(len(ids), dim, seed)


def apply_and_check(rp, orc, ups, rows, L, slack=0.0):
    rp.apply_batch(ups, rows)
    assert orc.apply_incremental(ups, rows) == 0
    G.check_graph(rp, orc)
    G.check_frontiers(rp, orc, L)
    G.check_values(rp, orc.full(), L, [None] + [orc.full_S(l) for l in range(1, L + 1)], row_slack=slack)


# Tensor-core form of the layer update: K chunks of 32 (31, 32, 33, and four / five of them: the weights stay in shared
# memory up to 128), column groups of 128, the widths for which it is taken (113 to 256; up to 64 over 256 and more
# entries there is a form in pieces, see test_gpu_narrow_products; others are fp32 sums), row tiles of 128 and the 1024 rows
# from which it is taken (n - 1, n and n + 1 of both), normalised sources, GIN's summed operand.
TC_MODELS = {
    "sage_31_5_47": lambda: I.sage_model([31, 5, 47], I.AGG_MEAN),
    "sage_33_129_256": lambda: I.sage_model([33, 129, 256], I.AGG_SUM),
    "sage_602_41_257": lambda: I.sage_model([602, 41, 257], I.AGG_MEAN),
    "sage_300_128_48": lambda: I.sage_model([300, 128, 48], I.AGG_MEAN),
    "gcn_32_48_128": lambda: I.graphconv_model([32, 48, 128], I.AGG_WSUM_GCN),
    "gcn_129_100_130": lambda: I.graphconv_model([129, 100, 130], I.AGG_WSUM_GCN),
    "gin_33_129": lambda: I.gin_model(33, 129, 2, eps=0.25),
    "gin_128_128": lambda: I.gin_model(128, 128, 2, eps=0.25),
    "gin_100_256": lambda: I.gin_model(100, 256, 2, eps=0.25),
}


@pytest.mark.parametrize("name", list(TC_MODELS.keys()))
def test_row_updates_at_the_edges_of_their_tiles(env, name):
    ripple, Oracle = env
    model = TC_MODELS[name]()
    L = len(model.layers)
    slack = GIN_ROW_SLACK if name.startswith("gin") else 0.0
    for n in (1023, 1024, 1025, 1153):
        src, dst = I.er_graph(n, 4 * n, 3)
        X = I.features(n, model.dims[0], 3)
        W = I.make_weights(model, 3, zero_bias=False)
        rp = ripple.Ripple(n, src, dst, X, model, W, max_batch=2048)
        orc = Oracle(n, src, dst, X, model, W)
        G.check_values(rp, orc.full(), L, row_slack=slack)
        for b in range(2):      # every row changes; then an ordinary batch on the launch geometry of the large one
            apply_and_check(rp, orc, *feature_batch(n, range(n), model.dims[0], 70 + b), L, slack)
        apply_and_check(rp, orc, *feature_batch(n, range(0, n, n // 7), model.dims[0], 80), L, slack)
        rp.recompute_full()
        G.check_values(rp, orc.full(), L, row_slack=slack)
        rp.close()


# A walk that adds into rows of half a gigabyte is made twice, over the lower and the upper half of the ids (330 K rows of
# 256 floats and three messages per row are past the line); the swept hop reads every in-list instead.
@pytest.mark.parametrize("kind", ["sage-push", "sage-pull", "weighted-push", "attention"])
def test_walks_over_rows_that_outgrow_the_cache(env, kind):
    ripple, Oracle = env
    n, hubs, per_hub, d = 330_001, 64, 16_001, 256
    rng = np.random.default_rng(5)
    src = np.repeat(np.arange(hubs, dtype=np.int32) * 5003, per_hub)
    dst = np.concatenate([rng.choice(n, per_hub, replace=False) for _ in range(hubs)]).astype(np.int32)
    keep = src != dst
    src, dst = src[keep], dst[keep]
    kw = {"edge_weights": I.edge_weights(src.size, 5)} if kind == "weighted-push" else {}
    model = {"sage": I.sage_model([d, d], I.AGG_SUM), "weighted": I.graphconv_model([d, d], I.AGG_WSUM_EDGE),
             "attention": I.gat_model(d, 1, d_att=8, slope=0.2)}[kind.split("-")[0]]
    X = I.features(n, d, 5)
    W = I.make_weights(model, 5)
    mode = ripple.SCATTER_PULL if kind == "sage-pull" else ripple.SCATTER_PUSH
    rp = ripple.Ripple(n, src, dst, X, model, W, scatter_mode=ripple.SCATTER_AUTO if kind == "attention" else mode, **kw)
    orc = Oracle(n, src, dst, X, model, W, **kw)
    ups, rows = feature_batch(n, np.arange(hubs) * 5003, d, 6)
    rp.apply_batch(ups, rows)
    assert orc.apply_incremental(ups, rows) == 0
    G.check_frontiers(rp, orc, 1)
    assert rp.stats()["active_edges"][1] >= 2 * n
    G.check_values(rp, orc.full(), 1)
    rp.close()


# How a batch reaches the device: one block up to 4 updates, up to 512 updates and 32 KB staged by one block, more by a grid;
# host batches of up to 64 KB packed into the staging area, larger ones read where they lie if they are pinned and packed
# if not.  (Batches beyond the staging area: test_gpu_batch_memory.py.)
@pytest.mark.parametrize("mem", ["host", "pinned", "device"])
@pytest.mark.parametrize("d", [8, 602])
def test_batches_at_the_edges_of_the_staging_forms(env, mem, d):
    import torch
    ripple, Oracle = env
    model = I.sage_model([d, 24, 10], I.AGG_MEAN)
    n = 1500
    src, dst = I.er_graph(n, 6000, 11)
    X = I.features(n, d, 11)
    W = I.make_weights(model, 11, zero_bias=False)
    rp = ripple.Ripple(n, src, dst, X, model, W)
    orc = Oracle(n, src, dst, X, model, W)
    stream = I.UpdateStream(n, src, dst, d, 11)
    for b, bs in enumerate([1, 4, 5, 13, 14, 26, 28, 511, 512, 513, 700, 512]):
        if b % 2:
            ups, rows = feature_batch(n, (np.arange(bs) * 7 + b) % n, d, 300 + b)
        else:
            ups, rows = stream.next_batch(bs)
        a, r = ups, rows
        if mem != "host":
            a = torch.from_numpy(np.stack([ups["op"], ups["u"], ups["v"]], axis=1).astype(np.int32))
            r = torch.from_numpy(rows)
            a, r = (a.cuda(), r.cuda()) if mem == "device" else (a.pin_memory(), r.pin_memory())
        rp.apply_batch(a, r)
        assert orc.apply_incremental(ups, rows) == 0
        G.check_graph(rp, orc)
        G.check_frontiers(rp, orc, 2)
        G.check_values(rp, orc.full(), 2)
    rp.close()


# The default arithmetic is fp32 sums outside the lines of the tensor-core forms, tf32-split products from 113 columns on, and
# up to 64 columns over 256 and more entries products of three bf16 parts, which have to be as exact as fp32 sums: a layer's product
# over rows without in-neighbours, against fp64, on both sides of the lines.  u = 2^-24.  A sequential fp32 sum of K terms of
# random sign: one rounding per term, 0.58 u / x rms for a partial sum of mantissa x (0.41 u over a binade), and partial sums
# that grow like sqrt(k): 0.41 u sqrt(K / 2).  The tensor core truncates one addition per eight terms (0.31 u each, by measurement
# at K = 32 to 602) and its operands' remainders are rounded (2.2 u).  Half as much again is allowed of either.
@pytest.mark.parametrize("rows", [600, 1022, 1024, 4000])
@pytest.mark.parametrize("K", [32, 100, 256, 602])
def test_products_are_as_exact_as_their_arithmetic(env, K, rows):
    ripple, _ = env
    for d in (24, 48, 96, 112, 113, 128, 256, 257):
        model = I.sage_model([K, d], I.AGG_MEAN)
        X, W = I.features(rows, K, d), I.make_weights(model, 3, zero_bias=False)
        rp = ripple.Ripple(rows, np.array([0], dtype=np.int32), np.array([1], dtype=np.int32), X, model, W)
        got = rp.embeddings(1).cpu().numpy().astype(np.float64)[2:]
        rp.close()
        ref = X.astype(np.float64)[2:] @ W[0]["Wa"].astype(np.float64) + W[0]["ba"]
        tensor = 113 <= d <= 256 and rows >= 1024
        bound = 1.5 * 2.0 ** -24 * (2.2 + 0.31 * K / 8 if tensor else 0.41 * np.sqrt(K / 2))
        err = float(np.linalg.norm(got - ref) / np.linalg.norm(ref))
        assert err <= bound, (d, err, bound)


@pytest.mark.parametrize("K", [8, 256, 260, 516, 602])
@pytest.mark.parametrize("items", [1, 2, "all", "one row more"])
def test_few_row_products_at_the_edge_of_the_device(env, K, items):
    """The form of small batches for few rows takes items of 16 rows and 32 columns, 256 entries of K at a time, while all items
    fit on the device at once (four per SM): one row group, two, all that fit (100 columns: four column groups), one row
    beyond."""
    import torch
    ripple, Oracle = env
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    rows = {1: 16, 2: 17, "all": 16 * sm, "one row more": 16 * sm + 1}[items]
    n = rows + 50
    ring = np.arange(1, n, dtype=np.int32)
    src = np.concatenate([np.zeros(rows, dtype=np.int32), ring, ring])      # vertex 0 reaches `rows` sinks
    dst = np.concatenate([1 + np.arange(rows, dtype=np.int32), 1 + ring % (n - 1), 1 + (ring + 6) % (n - 1)])
    model = I.graphconv_model([K, 100], I.AGG_MEAN)
    X = I.features(n, K, 3)
    W = I.make_weights(model, 3, zero_bias=False)
    rp = ripple.Ripple(n, src, dst, X, model, W, pre_transform=False)
    orc = Oracle(n, src, dst, X, model, W)
    for b in range(3):
        apply_and_check(rp, orc, *feature_batch(n, [0], K, 90 + b), 1)
        assert rp.stats()["affected"][1] == rows
    rp.close()
