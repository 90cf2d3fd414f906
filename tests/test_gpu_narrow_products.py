"""Products of at most 64 columns over 256 and more entries: the tensor-core form that sums chunks of 32 entries apart, at
the edges of its rule (255 / 256 entries, 64 / 65 columns, 1023 / 1024 rows), of its chunks and of its tiles; two
problems over the same rows side by side and single ones; its error, which is no larger than that of fp32 sums, dense rows
or sparse ones; and entries that have no parts."""
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


def self_product(ripple, X, W, model, mode):
    n = X.shape[0]
    src = np.arange(n, dtype=np.int32)
    rp = ripple.Ripple(n, src, (src + 1) % n, X, model, W, gemm_mode=mode)
    got = rp.embeddings(1).cpu().numpy()
    rp.close()
    return got


@pytest.mark.parametrize("K", [256, 602])
@pytest.mark.parametrize("entries", [1, 2, 3, 4, 8, 16, 64])
@pytest.mark.parametrize("near", [False, True])
def test_sparse_rows_keep_the_bits_of_fp32(env, K, entries, near):
    """Rows with a few entries that are not zero, scattered or side by side (across the middle of a chunk among them): a sum
    of few terms has almost no rounding to hide behind, so operands held in fewer than 24 bits show (22 bits: 1.4e-7 where the
    fp32 sum has 2.5e-8).  Both errors are at least that of one rounding and equal for one entry; a fiftieth for the luck of
    the draw."""
    ripple, _ = env
    n, cols = 2048, 47
    model = I.sage_model([K, cols])
    W = I.make_weights(model, 5)
    W[0]["Wb"] = np.zeros_like(W[0]["Wb"])
    rng = np.random.default_rng(K + entries)
    X = np.zeros((n, K), dtype=np.float32)
    for i in range(n):
        at = 32 * rng.integers(0, K // 32) + 16 - entries // 2 if near else 0
        ids = np.arange(at, at + entries) % K if near else rng.choice(K, entries, replace=False)
        X[i, ids] = rng.standard_normal(entries)
    ref = X.astype(np.float64) @ W[0]["Wa"].astype(np.float64)
    err = [np.linalg.norm(self_product(ripple, X, W, model, m) - ref) / np.linalg.norm(ref) for m in (ripple.GEMM_FP32, ripple.GEMM_AUTO)]
    assert err[1] <= 1.02 * err[0], err


def test_entries_without_parts(env):
    """Infinite entries, NaN, and entries next to the largest: infinite, NaN and finite results where the fp32 sum has them."""
    ripple, _ = env
    n, K, cols = 2048, 300, 40
    model = I.sage_model([K, cols])
    W = I.make_weights(model, 6)
    W[0]["Wb"] = np.zeros_like(W[0]["Wb"])
    W[0]["Wa"][::3] = np.round(W[0]["Wa"][::3] * 64) / 64     # (weights with no second part, some of them zero)
    rng = np.random.default_rng(1)
    X = rng.standard_normal((n, K)).astype(np.float32)
    at = rng.integers(0, K, n)
    big = np.finfo(np.float32).max
    for i in range(n):
        X[i, at[i]] = (np.inf, -np.inf, np.nan, big, -big, 1.0)[i % 6]
    X[6::12, 7] = -np.inf                                     # two infinite entries
    a, b = (self_product(ripple, X, W, model, m) for m in (ripple.GEMM_FP32, ripple.GEMM_AUTO))
    assert np.array_equal(np.isnan(a), np.isnan(b)) and np.isnan(a).any()
    assert np.array_equal(np.isposinf(a), np.isposinf(b)) and np.isposinf(a).any()
    assert np.array_equal(np.isneginf(a), np.isneginf(b)) and np.isneginf(a).any()
    f = np.isfinite(a)
    scale = 1.0 + np.abs(a[f].astype(np.float64))
    assert np.max(np.abs(a[f].astype(np.float64) - b[f]) / scale) <= 1e-5
