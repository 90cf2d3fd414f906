"""Where a batch may lie: memory that kernels cannot read as it is (registered only in part, odd addresses) is copied, and
every memory space brings the weights of its operations along.  Against the oracle, as in test_gpu_parity."""
import mmap

import numpy as np
import pytest

from paper_2601_12347_b200 import inputs as I

from tolerances import GIN_ROW_SLACK

import test_gpu_parity as G

pytestmark = pytest.mark.gpu

env = G.env

N, D = 1500, 64


def _pair(env, weighted=False, **kw):
    ripple, Oracle = env
    model = I.graphconv_model([D, 24, 10], I.AGG_WSUM_EDGE) if weighted else I.sage_model([D, 24, 10], I.AGG_MEAN)
    src, dst = I.er_graph(N, 6000, 11)
    more = {"edge_weights": I.edge_weights(src.size, 11)} if weighted else {}
    X = I.features(N, D, 11)
    W = I.make_weights(model, 11, zero_bias=False)
    return ripple.Ripple(N, src, dst, X, model, W, **more, **kw), Oracle(N, src, dst, X, model, W, **more), src, dst


def _feature_batch(count, seed):
    ups = G.ups_array([(I.OP_SET_FEATURE, int(u), i) for i, u in enumerate(np.random.default_rng(seed).permutation(N)[:count])])
    return ups, I.features(count, D, seed)


def _check(rp, orc, ups, rows, **kw):
    assert orc.apply_incremental(ups, rows, **kw) == 0
    G.check_graph(rp, orc)
    G.check_frontiers(rp, orc, 2)
    G.check_values(rp, orc.full(), 2)


def _raw(ups):
    return np.stack([ups["op"], ups["u"], ups["v"]], axis=1).astype(np.int32)


@pytest.mark.parametrize("part", ["first page", "all but the last page"])
def test_rows_registered_in_part_are_copied(env, part):
    import torch
    rp, orc, *_ = _pair(env)
    page = mmap.PAGESIZE
    ups, rows = _feature_batch(700, 5)                       # 180 KB of rows: past the size that is packed without a look
    buf = mmap.mmap(-1, (rows.nbytes // page + 1) * page)
    mine = np.frombuffer(buf, dtype=np.float32, count=rows.size).reshape(rows.shape)
    mine[:] = rows
    pinned = torch.from_numpy(_raw(ups)).pin_memory()
    size = page if part == "first page" else rows.nbytes // page * page
    rt = torch.cuda.cudart()
    assert int(rt.cudaHostRegister(mine.ctypes.data, size, 0)) == 0
    try:
        rp.apply_batch(pinned, torch.from_numpy(mine))
    finally:
        rt.cudaHostUnregister(mine.ctypes.data)
    _check(rp, orc, ups, rows)
    rp.close()


@pytest.mark.parametrize("mem", ["pinned", "device"])
@pytest.mark.parametrize("count", [3, 100, 700])
def test_odd_addresses_are_copied(env, mem, count):
    import torch
    ripple, _ = env
    rp, orc, *_ = _pair(env)
    ups, rows = _feature_batch(count, 6)
    kept = []

    def odd(a):      # the same bytes, one byte past an allocation's start
        t = torch.empty(a.nbytes + 16, dtype=torch.uint8, pin_memory=mem == "pinned", device="cuda" if mem == "device" else "cpu")
        t[1:1 + a.nbytes] = torch.from_numpy(np.frombuffer(a.tobytes(), dtype=np.uint8).copy())
        kept.append(t)
        return t.data_ptr() + 1
    pu, pr = odd(_raw(ups)), odd(rows)
    torch.cuda.synchronize()
    assert rp.lib.ripple_apply_batch(rp.h, pu, count, pr, count, ripple.MEM_DEVICE if mem == "device" else ripple.MEM_HOST) == ripple.OK
    _check(rp, orc, ups, rows)
    rp.close()


# Rows as a slice from the second of a tensor with an odd width (in bounds, on a 4-byte boundary only), and batches larger
# than the staging area, copied ahead of a chain that is replayed for a batch of the same geometry read in place.
@pytest.mark.parametrize("mem", ["host", "pinned", "device"])
def test_rows_off_the_wide_alignment_and_batches_beyond_the_staging_area(env, mem):
    import torch
    ripple, Oracle = env
    d = 603
    model = I.sage_model([d, 24, 10], I.AGG_MEAN)
    src, dst = I.er_graph(N, 6000, 11)
    X, W = I.features(N, d, 11), I.make_weights(model, 11, zero_bias=False)
    rp, orc = ripple.Ripple(N, src, dst, X, model, W), Oracle(N, src, dst, X, model, W)
    for b, count in enumerate([600, 1000, 600, 1000, 600]):  # 1.4 and 2.4 MB of rows; the area holds 1.3
        ids = np.random.default_rng(b).permutation(N)[:count]
        ups = G.ups_array([(I.OP_SET_FEATURE, int(u), i) for i, u in enumerate(ids)])
        all_rows = I.features(count + 1, d, 40 + b)
        rows = all_rows[1:]
        if mem == "host":
            rp.apply_batch(ups, rows)
        else:
            a, r = torch.from_numpy(_raw(ups)), torch.from_numpy(all_rows)
            a, r = (a.cuda(), r.cuda()) if mem == "device" else (a.pin_memory(), r.pin_memory())
            torch.cuda.synchronize()
            rp.apply_batch(a, r[1:])
        _check(rp, orc, ups, np.ascontiguousarray(rows))
    rp.close()


@pytest.mark.parametrize("mem", ["host", "pinned", "device"])
def test_operation_weights_arrive_from_every_memory_space(env, mem):
    import torch
    rp, orc, src, dst = _pair(env, weighted=True)
    stream = I.UpdateStream(N, src, dst, D, 11)
    for b, count in enumerate([3, 100, 700, 3, 100, 700, 4000]):
        ups, rows = stream.next_batch(count)
        w = I.edge_weights(count, 20 + b)
        if mem == "host":
            rp.apply_batch(ups, rows, w)
        else:
            t = [torch.from_numpy(x) for x in (_raw(ups), rows, w)]
            t = [x.cuda() if mem == "device" else x.pin_memory() for x in t]
            torch.cuda.synchronize()
            rp.apply_batch(*t)
        _check(rp, orc, ups, rows, op_weights=w)
        assert np.array_equal(rp.export_graph_weighted()[2], orc.export_weights())
    rp.close()


def test_more_launch_geometries_than_captured_chains_are_kept(env):
    """Sizes and memory spaces mixed on one context: twenty and more geometries go round, so chains are captured while a
    batch is in flight, replayed, given up and captured again."""
    import torch
    rp, orc, src, dst = _pair(env, weighted=True)
    stream = I.UpdateStream(N, src, dst, D, 12)
    rng = np.random.default_rng(4)
    sizes = [1, 3, 5, 12, 17, 33, 65, 128, 129, 300, 600, 1025]
    todo = [(s, m) for s in sizes for m in ("host", "pinned", "device")]
    for rnd in range(4):
        order = rng.permutation(len(todo)) if rnd < 3 else np.repeat(rng.permutation(len(todo))[:8], 3)
        for k in order:
            count, mem = todo[k]
            ups, rows = stream.next_batch(count)
            w = I.edge_weights(count, 900 + rnd) if count % 2 else None
            a = [_raw(ups), rows] + ([w] if w is not None else [])
            t = [torch.from_numpy(x) for x in a]
            if mem == "host":
                rp.apply_batch(ups, *a[1:])
            else:
                t = [x.cuda() if mem == "device" else x.pin_memory() for x in t]
                torch.cuda.synchronize()
                rp.apply_batch(*t)
            assert orc.apply_incremental(ups, rows, op_weights=w) == 0
            G.check_frontiers(rp, orc, 2)
        G.check_graph(rp, orc)
        assert np.array_equal(rp.export_graph_weighted()[2], orc.export_weights())
        G.check_values(rp, orc.full(), 2, row_slack=GIN_ROW_SLACK)
    rp.close()
