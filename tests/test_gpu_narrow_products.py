"""Products of at most 64 columns over 256 and more entries: the tensor-core form that sums pieces of 16 entries apart, at
the edges of its rule (255 / 256 entries, 64 / 65 columns, 1023 / 1024 rows), of its pieces and chunks and of its tiles; two
problems over the same rows side by side and single ones; and its error, which is no larger than that of fp32 sums."""
import numpy as np
import pytest

from paper_2601_12347_b200 import inputs as I

import test_gpu_kernel_edges as E
import test_gpu_parity as G

pytestmark = pytest.mark.gpu

env = G.env

MODELS = {
    "sage_20_256_40": lambda: I.sage_model([20, 256, 40]),
    "sage_20_255_47": lambda: I.sage_model([20, 255, 47]),
    "sage_20_257_5": lambda: I.sage_model([20, 257, 5]),
    "sage_272_64": lambda: I.sage_model([272, 64]),
    "sage_300_65": lambda: I.sage_model([300, 65]),
    "sage_602_33_33": lambda: I.sage_model([602, 33, 33]),
    "gcn_20_260_48": lambda: I.graphconv_model([20, 260, 48], I.AGG_WSUM_GCN),
    "max_20_256_40": lambda: I.graphconv_model([20, 256, 40], I.AGG_MAX),
}


@pytest.mark.parametrize("name", list(MODELS))
def test_narrow_products_at_their_edges(env, name):
    ripple, Oracle = env
    model = MODELS[name]()
    L = len(model.layers)
    for n in (1023, 1024, 1025, 1153, 20_000):
        src, dst = I.er_graph(n, 4 * n, 3)
        X = I.features(n, model.dims[0], 3)
        W = I.make_weights(model, 3, zero_bias=False)
        rp = ripple.Ripple(n, src, dst, X, model, W, max_batch=20_480)
        orc = Oracle(n, src, dst, X, model, W)
        G.check_values(rp, orc.full(), L)
        for b in range(2):      # every row changes; then an ordinary batch on the launch geometry of the large one
            ups, rows = E.feature_batch(n, range(n), model.dims[0], 70 + b)
            rp.apply_batch(ups, rows)
            assert orc.apply_incremental(ups, rows) == 0
            G.check_values(rp, orc.full(), L)
        ups, rows = E.feature_batch(n, range(0, n, max(1, n // 300)), model.dims[0], 80)
        rp.apply_batch(ups, rows)
        assert orc.apply_incremental(ups, rows) == 0
        G.check_values(rp, orc.full(), L)
        rp.close()


@pytest.mark.parametrize("K", [256, 602])
@pytest.mark.parametrize("cols", [5, 47, 64])
def test_no_less_exact_than_fp32_sums(env, K, cols):
    """Self products of rows as a rectifier leaves them, against fp64: the pieces' error within that of the fp32 form (2-norm;
    measured 1.7e-7 to 2.2e-7 against 1.8e-7 to 3.3e-7; a tenth for the luck of 4096 rows)."""
    ripple, _ = env
    n = 4096
    model = I.sage_model([K, cols])
    W = I.make_weights(model, 3)
    W[0]["Wb"] = np.zeros_like(W[0]["Wb"])
    X = np.maximum(np.random.default_rng(K + cols).standard_normal((n, K)), 0).astype(np.float32)
    ref = X.astype(np.float64) @ W[0]["Wa"].astype(np.float64)
    if model.layers[0].act:
        ref = np.maximum(ref, 0)
    src = np.arange(n, dtype=np.int32)
    err = []
    for mode in (ripple.GEMM_FP32, ripple.GEMM_AUTO):
        rp = ripple.Ripple(n, src, (src + 1) % n, X, model, W, gemm_mode=mode)
        got = rp.embeddings(1).cpu().numpy().astype(np.float64)
        err.append(np.linalg.norm(got - ref) / np.linalg.norm(ref))
        rp.close()
    assert err[1] <= 1.1 * err[0], err
