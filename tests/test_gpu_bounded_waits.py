"""Every call that can meet a bounded wait that gave up says so (RIPPLE_ERR_TIMEOUT), not only the batch: the layer-wise
recomputation, the growth of the vertex set and the phases of a partitioned execution.  The wait is made to run out by the
diagnostic environment switch: the tensor-core update never signals its first finished tile, its epilogue gives up after some
milliseconds and the device goes on answering."""
import numpy as np
import pytest

from paper_2601_12347_b200 import inputs as I

import test_gpu_parity as G

pytestmark = pytest.mark.gpu

env = G.env

N = 5000


def _problem():
    model = I.sage_model([24, 256, 256, 12], I.AGG_MEAN)
    src, dst = I.er_graph(N, 25000, 3)
    X = I.features(N, 24, 3)
    W = I.make_weights(model, 3, zero_bias=False)
    return model, src, dst, X, W


def _expect_timeout(ripple, monkeypatch, call):
    monkeypatch.setenv("RIPPLE_DEBUG_TC_WITHHOLD", "1")
    with pytest.raises(ripple.RippleError) as ei:
        call()
    assert ei.value.status == ripple.ERR_TIMEOUT and "wait gave up" in str(ei.value)
    monkeypatch.delenv("RIPPLE_DEBUG_TC_WITHHOLD")


@pytest.mark.parametrize("call", ["create", "recompute", "reserve"])
def test_whole_graph_calls_report_a_timeout(env, monkeypatch, call):
    ripple, Oracle = env
    model, src, dst, X, W = _problem()
    if call == "create":
        _expect_timeout(ripple, monkeypatch, lambda: ripple.Ripple(N, src, dst, X, model, W))
    else:
        rp = ripple.Ripple(N, src, dst, X, model, W)
        _expect_timeout(ripple, monkeypatch, rp.recompute_full if call == "recompute" else lambda: rp.reserve_vertices(N + 2000))
        rp.close()
    rp = ripple.Ripple(N, src, dst, X, model, W)
    rp.recompute_full()
    G.check_values(rp, Oracle(N, src, dst, X, model, W).full(), 3)
    rp.close()


@pytest.mark.parametrize("call", ["recompute", "batch"])
def test_workers_report_a_timeout(env, monkeypatch, call):
    ripple, Oracle = env
    from paper_2601_12347_b200.partitioned import Cluster
    model, src, dst, X, W = _problem()
    owner = np.random.default_rng(0).integers(0, 2, size=N).astype(np.int32)
    cl = Cluster(2, owner, src, dst, X, model, W)
    ups, rows = I.UpdateStream(N, src, dst, 24, 3).next_batch(1500)
    _expect_timeout(ripple, monkeypatch, cl.recompute_full if call == "recompute" else lambda: cl.apply_batch(ups, rows))
    cl.close()
