"""A batch that is rejected late, when its row moves are planned (the overflow pool is exhausted), after its operations have
been resolved and its feature updates marked, leaves nothing behind: what follows is what the oracle computes without it."""
import numpy as np
import pytest

from paper_2601_12347_b200 import inputs as I

import test_gpu_parity as G

pytestmark = pytest.mark.gpu

env = G.env

N, D, HUB = 900, 20, 5

MODELS = {
    "sage": lambda: I.sage_model([D, 24, 16, 10], I.AGG_MEAN),
    "sage_equal": lambda: I.sage_model([D, D, D], I.AGG_SUM),
    "gcn": lambda: I.graphconv_model([D, 24, 16, 10], I.AGG_WSUM_GCN),
    "max": lambda: I.graphconv_model([D, 24, 10], I.AGG_MAX),
    "gat": lambda: I.gat_model(D, 2, d_att=8, slope=0.2),
}


def _problem(name):
    model = MODELS[name]()
    src, dst = I.er_graph(N, 4000, 5)
    return model, src, dst, I.features(N, D, 5), I.make_weights(model, 5, zero_bias=False)


def _new_sinks(rp, u):
    rowptr, col = rp.export_graph()
    have = set(col[rowptr[u]:rowptr[u + 1]].tolist())
    return [v for v in range(N) if v != u and v not in have]


@pytest.mark.parametrize("size", [4, 100, 700])
@pytest.mark.parametrize("name", list(MODELS.keys()))
def test_what_follows_a_rejected_batch(env, name, size):
    ripple, Oracle = env
    model, src, dst, X, W = _problem(name)
    L = len(model.layers)
    rp = ripple.Ripple(N, src, dst, X, model, W, slack=0.001, pool_edges=4)
    orc = Oracle(N, src, dst, X, model, W)
    for again in range(4):       # from the third time on a captured chain may be replayed
        if size == 4:            # the row is filled to its capacity first, so that one more edge is too many
            for v in _new_sinks(rp, HUB):
                one = G.ups_array([(I.OP_ADD_EDGE, HUB, v)])
                try:
                    rp.apply_batch(one)
                except ripple.RippleError as e:
                    assert e.status == ripple.ERR_CAPACITY
                    break
                assert orc.apply_incremental(one) == 0
            n_feat, sinks = 3, [v]
        else:
            n_feat, sinks = size // 5, _new_sinks(rp, HUB)[:size - size // 5]
        ups = G.ups_array([(I.OP_SET_FEATURE, HUB + i, i) for i in range(n_feat)] + [(I.OP_ADD_EDGE, HUB, v) for v in sinks])
        with pytest.raises(ripple.RippleError) as ei:
            rp.apply_batch(ups, I.features(n_feat, D, 77))
        assert ei.value.status == ripple.ERR_CAPACITY
        # edges out of a vertex whose feature row the rejected batch named, and other feature rows
        rowptr, col = rp.export_graph()
        u = next(x for x in range(HUB + 1, HUB + n_feat) if rowptr[x + 1] > rowptr[x])
        ids = np.random.default_rng(again).permutation(N)[:12]
        ok = G.ups_array([(I.OP_SET_FEATURE, int(v), i) for i, v in enumerate(ids)] + [(I.OP_DEL_EDGE, u, int(col[rowptr[u]]))])
        new = I.features(12, D, 90 + again)
        rp.apply_batch(ok, new)
        assert orc.apply_incremental(ok, new) == 0
        G.check_graph(rp, orc)
        if name != "max":        # (value-based frontiers may differ on ties)
            G.check_frontiers(rp, orc, L)
        G.check_values(rp, orc.full(), L)
    rp.close()


def test_what_follows_a_batch_that_a_worker_rejects(env):
    ripple, Oracle = env
    from paper_2601_12347_b200.partitioned import Cluster
    model, src, dst, X, W = _problem("sage")
    cl = Cluster(1, np.zeros(N, dtype=np.int32), src, dst, X, model, W, slack=0.001, pool_edges=4)
    orc = Oracle(N, src, dst, X, model, W)
    ids = cl.router.global_ids(0, cl.workers[0].n)           # local to global; the worker takes local ids
    local = {int(g): i for i, g in enumerate(ids) if g >= 0}
    have = set(dst[src == HUB].tolist())
    sinks = [v for v in range(N) if v != HUB and v not in have][:80]
    ups = G.ups_array([(I.OP_SET_FEATURE, local[HUB + 1 + i], i) for i in range(20)] +
                      [(I.OP_ADD_EDGE, local[HUB], local[v]) for v in sinks])
    with pytest.raises(ripple.RippleError) as ei:
        cl.workers[0].begin(ups, I.features(20, D, 77), np.zeros(ups.size, dtype=np.uint8))
    assert ei.value.status == ripple.ERR_CAPACITY
    gone = [i for i in range(src.size) if HUB + 1 <= src[i] <= HUB + 20][:10]
    ok = G.ups_array([(I.OP_DEL_EDGE, int(src[i]), int(dst[i])) for i in gone] + [(I.OP_SET_FEATURE, HUB + 300, 0)])
    new = I.features(1, D, 91)
    cl.apply_batch(ok, new)
    assert orc.apply_incremental(ok, new) == 0
    full = orc.full()
    for l in range(4):
        assert np.max(np.abs(cl.embeddings(l, N) - full[l]) / (1 + np.abs(full[l]))) <= 1e-4, l
    cl.close()
