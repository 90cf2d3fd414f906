"""The kernels that sum rows over in-lists (whole-graph sums, rebuilding hops, the sweep) at the sizes where their cuts lie:
list lengths around a window (128), the smallest piece (64) and the longest list a tile takes, rows of every number of
groups per warp and of several pieces per lane, ids beyond the exact filter, tiles of 8 and of 32 sinks."""
import numpy as np
import pytest

from paper_2601_12347_b200 import inputs as I
from tolerances import GIN_ROW_SLACK

import test_gpu_parity as G

pytestmark = pytest.mark.gpu

LENGTHS = (0, 1, 2, 7, 8, 9, 31, 63, 64, 65, 96, 127, 128, 129, 200, 255, 256, 257, 300, 511, 513, 1025, 2100)


env = G.env


def lists_of_every_length(n, seed):
    """Sinks spread over the ids, each length several times, neighbours drawn without repetition."""
    rng = np.random.default_rng(seed)
    lens = np.array(LENGTHS * 3)
    sinks = rng.choice(n, lens.size, replace=False)
    sinks[:8] = np.arange(8) + 3 * 32          # eight of them in one tile
    src, dst = [], []
    for v, k in zip(np.unique(sinks), lens):
        u = rng.choice(n - 1, k, replace=False)
        u[u >= v] += 1
        src.append(u)
        dst.append(np.full(k, v))
    return np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32)


def feature_batch(rng, n, d, count):
    vs = rng.choice(n, count, replace=False)
    ups = np.zeros(count, dtype=I.UPDATE_DTYPE)
    ups["op"], ups["u"], ups["v"] = I.OP_SET_FEATURE, vs, np.arange(count)
    return ups, rng.standard_normal((count, d)).astype(np.float32)


# widths: 1, 3, 5, 6, 10, 11, 12, 16, 25, 32, 33, 65 and 129 pieces of 16 bytes per row
@pytest.mark.parametrize("d", [4, 12, 18, 24, 40, 44, 47, 64, 100, 128, 132, 260, 516])
@pytest.mark.parametrize("agg", ["mean", "gcn", "weighted"])
def test_sums_over_lists_of_every_length(env, d, agg):
    ripple, Oracle = env
    n = 3000
    src, dst = lists_of_every_length(n, d)
    kw = {"edge_weights": I.edge_weights(src.size, 5)} if agg == "weighted" else {}
    model = {"mean": I.sage_model([d, d, 8]), "gcn": I.graphconv_model([d, d, 8], I.AGG_WSUM_GCN),
             "weighted": I.graphconv_model([d, d, 8], I.AGG_WSUM_EDGE)}[agg]
    X = I.features(n, d, d)
    W = I.make_weights(model, d)
    # rows that thousands of terms cancel into: the slack that the parity tests give unnormalised sums
    slack = GIN_ROW_SLACK if agg == "weighted" else 0.0
    for mode in (ripple.SCATTER_PULL, ripple.SCATTER_REGATHER):
        rp = ripple.Ripple(n, src, dst, X, model, W, scatter_mode=mode, pre_transform=False, **kw)
        orc = Oracle(n, src, dst, X, model, W, **kw)
        G.check_values(rp, orc.full(), 2, row_slack=slack)
        for count in (9, 2500):     # senders that the filter holds, and too many for it
            rng = np.random.default_rng(count)
            vs = rng.choice(n, count, replace=False)
            ups = np.zeros(count, dtype=I.UPDATE_DTYPE)
            ups["op"], ups["u"], ups["v"] = I.OP_SET_FEATURE, vs, np.arange(count)
            rows = rng.standard_normal((count, d)).astype(np.float32)
            rp.apply_batch(ups, rows)
            assert orc.apply_incremental(ups, rows) == 0
            G.check_frontiers(rp, orc, 2)
            G.check_values(rp, orc.full(), 2, row_slack=slack)
        rp.close()


@pytest.mark.parametrize("n", [303_104, 524_288, 524_289, 600_001])   # tiles of 32 from the first; the filter hashes from the third
def test_sweep_on_graphs_beyond_the_exact_filter(env, n):
    ripple, Oracle = env
    d = 12
    src, dst = lists_of_every_length(n, n % 1000)
    model = I.sage_model([d, d, 8])
    X = I.features(n, d, 3)
    W = I.make_weights(model, 3)
    rp = ripple.Ripple(n, src, dst, X, model, W, scatter_mode=ripple.SCATTER_PULL, pre_transform=False)
    orc = Oracle(n, src, dst, X, model, W)
    rng = np.random.default_rng(1)
    for count in (5, 60):
        vs = rng.choice(src, count, replace=False)
        vs = np.unique(vs)
        ups = np.zeros(vs.size, dtype=I.UPDATE_DTYPE)
        ups["op"], ups["u"], ups["v"] = I.OP_SET_FEATURE, vs, np.arange(vs.size)
        rows = rng.standard_normal((vs.size, d)).astype(np.float32)
        rp.apply_batch(ups, rows)
        assert orc.apply_incremental(ups, rows) == 0
        G.check_frontiers(rp, orc, 2)
    G.check_values(rp, orc.full(), 2)
    rp.close()


def test_swept_and_pushed_hops_agree_where_the_device_chooses(env):
    """Batches of 2100 feature updates (F), whose second hop carries nearly all edges from 18 K senders and is swept, and of 2100
    edges deleted (D) and added (A), whose second hop carries a tenth and is pushed.  After an F both forms are in the chain:
    D and A replay the chain captured for F and push on it.  After a D or an A the sweep is not in the chain, and F pushes
    once.  900 feature updates (f) lie on the other side of the line, near enough to keep both.  PUSH pushes throughout."""
    ripple, _ = env
    n = 20_000
    src, dst = I.er_graph(n, 400_000, 4)
    model = I.sage_model([64, 200, 196])
    X = I.features(n, 64, 4)
    W = I.make_weights(model, 4)
    rps = [ripple.Ripple(n, src, dst, X, model, W, scatter_mode=m, regather_threshold=-1.0) for m in (ripple.SCATTER_AUTO, ripple.SCATTER_PUSH)]
    rng = np.random.default_rng(2)
    edges = np.zeros(2100, dtype=I.UPDATE_DTYPE)
    at = rng.choice(src.size, edges.size, replace=False)
    edges["u"], edges["v"] = src[at], dst[at]
    before = "F"      # (nothing known: both forms)
    for kind in "FFFFDFFAFFDFfF":
        if kind in "DA":
            ups, rows = edges.copy(), None
            ups["op"] = I.OP_DEL_EDGE if kind == "D" else I.OP_ADD_EDGE
        else:
            ups, rows = feature_batch(rng, n, 64, 2100 if kind == "F" else 900)
        for rp in rps:
            rp.apply_batch(ups, rows)
        assert list(rps[0].stats()["scatter_pull"][1:3]) == [0, 1 if kind == "F" and before in "Ff" else 0], before + kind
        before = kind
        assert list(rps[1].stats()["scatter_pull"][1:3]) == [0, 0]
        for l in range(3):
            assert np.array_equal(rps[0].affected(l).cpu().numpy(), rps[1].affected(l).cpu().numpy())
            a, c = (rp.embeddings(l).cpu().numpy() for rp in rps)
            assert np.max(np.abs(a - c) / (1 + np.abs(c))) <= 1e-4
    for rp in rps:
        rp.close()


@pytest.mark.parametrize("min_width", [None, "0", "257"])
def test_a_hop_is_swept_for_what_it_carries_not_for_the_batch_before(env, monkeypatch, min_width):
    """Batches of 6000 and of one update in turn: hop 2 carries 1.5 M wide messages in the one, 2500 in the other, and is swept
    in the one and pushed in the other; never swept where the least width excludes it."""
    ripple, _ = env
    if min_width is not None:
        monkeypatch.setenv("RIPPLE_GATHER_MIN_WIDTH", min_width)
    n, d = 30_000, 32
    src, dst = I.er_graph(n, 1_500_000, 8)
    model = I.sage_model([d, 256, 256])
    X = I.features(n, d, 8)
    W = I.make_weights(model, 8)
    rps = [ripple.Ripple(n, src, dst, X, model, W, scatter_mode=m, regather_threshold=-1.0) for m in (ripple.SCATTER_AUTO, ripple.SCATTER_PUSH)]
    rng = np.random.default_rng(8)
    for count in (6000, 6000, 1, 6000, 1, 1, 6000):
        ups, rows = feature_batch(rng, n, d, count)
        for rp in rps:
            rp.apply_batch(ups, rows)
        st = rps[0].stats()
        assert st["active_edges"][2] > (1 << 20) if count > 1 else st["active_edges"][2] < 10_000
        assert list(st["scatter_pull"][1:3]) == [0, 1 if count > 1 and min_width is None else 0]
        assert list(rps[1].stats()["scatter_pull"][1:3]) == [0, 0]
        for l in range(3):
            assert np.array_equal(rps[0].affected(l).cpu().numpy(), rps[1].affected(l).cpu().numpy())
            a, c = (rp.embeddings(l).cpu().numpy() for rp in rps)
            assert np.max(np.abs(a - c) / (1 + np.abs(c))) <= 1e-4
    for rp in rps:
        rp.close()


@pytest.mark.parametrize("agg", ["mean", "gcn", "weighted"])
@pytest.mark.parametrize("n", [3000, 310_000, 600_001])     # tiles of 8 and of 32; ids that the filter holds and hashes
def test_sweeps_of_the_frontiers_lists_and_of_all(env, n, agg):
    """SCATTER_PULL: a hop that carries less than an eighth of the edges reads the lists of its frontier, marked beforehand;
    with the hub among its senders (a third of the edges) all lists.  Feature updates, and edges that come and go."""
    ripple, Oracle = env
    d = 12
    src, dst = lists_of_every_length(n, n % 1000)
    have = set(zip(src.tolist(), dst.tolist()))
    hub = n - 7
    extra = [v for v in range(0, min(n, src.size // 2 + 200)) if v != hub and (hub, v) not in have]
    src = np.concatenate([src, np.full(len(extra), hub, dtype=np.int32)])
    dst = np.concatenate([dst, np.array(extra, dtype=np.int32)])
    kw = {"edge_weights": I.edge_weights(src.size, 5)} if agg == "weighted" else {}
    model = {"mean": I.sage_model([d, d, d, 8]), "gcn": I.graphconv_model([d, d, d, 8], I.AGG_WSUM_GCN),
             "weighted": I.graphconv_model([d, d, d, 8], I.AGG_WSUM_EDGE)}[agg]
    X = I.features(n, d, 3)
    W = I.make_weights(model, 3)
    rp = ripple.Ripple(n, src, dst, X, model, W, scatter_mode=ripple.SCATTER_PULL, pre_transform=False, **kw)
    orc = Oracle(n, src, dst, X, model, W, **kw)
    stream = I.UpdateStream(n, src, dst, d, 4)
    rng = np.random.default_rng(n)
    few = many = 0
    for b in range(7):
        if b in (2, 5):
            ups = np.zeros(2, dtype=I.UPDATE_DTYPE)
            ups["op"], ups["u"], ups["v"] = I.OP_SET_FEATURE, [hub, int(src[5])], [0, 1]
            rows = rng.standard_normal((2, d)).astype(np.float32)
        elif b in (0, 4):
            vs = np.unique(rng.choice(src, 12 if b else 1))
            ups = np.zeros(vs.size, dtype=I.UPDATE_DTYPE)
            ups["op"], ups["u"], ups["v"] = I.OP_SET_FEATURE, vs, np.arange(vs.size)
            rows = rng.standard_normal((vs.size, d)).astype(np.float32)
        else:
            ups, rows = stream.next_batch(30)
        rp.apply_batch(ups, rows)
        assert orc.apply_incremental(ups, rows) == 0
        G.check_frontiers(rp, orc, 3)
        st = rp.stats()
        assert list(st["scatter_pull"][1:4]) == [1, 1, 1]
        share = np.array(st["active_edges"][1:4]) * 8 >= st["num_edges"]
        few, many = few + int((~share).sum()), many + int(share.sum())
    assert few >= 3 and many >= 2, (few, many)
    G.check_values(rp, orc.full(), 3, row_slack=GIN_ROW_SLACK if agg == "weighted" else 0.0)
    rp.close()
