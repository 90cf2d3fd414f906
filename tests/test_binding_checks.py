"""What the Python binding hands to the library, without a device: an array whose shape, type or memory space is not the one
that the library reads never reaches it."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2601_12347_b200 import inputs as I
from paper_2601_12347_b200 import ripple

D0 = 6


class _Lib:
    """Notes the calls instead of making them."""

    def __init__(self):
        self.calls = []

    def ripple_apply_batch(self, h, uptr, n, fptr, nr, mem):
        self.calls.append((n, nr, mem))
        return ripple.OK

    def ripple_apply_batch_weighted(self, h, uptr, n, fptr, nr, wptr, mem):
        self.calls.append((n, nr, mem, wptr is not None))
        return ripple.OK


class _Cuda:
    """Stands for a tensor in device memory."""
    is_cuda = True

    def __init__(self, t):
        self._t = t

    def __getattr__(self, name):
        return getattr(self._t, name)

    def contiguous(self):
        return self


@pytest.fixture
def rp():
    r = ripple.Ripple.__new__(ripple.Ripple)
    r.lib, r.h, r.dims, r.n = _Lib(), ctypes.c_void_p(None), [D0, 4], 100
    return r


def _ups(n):
    return np.array([(I.OP_SET_FEATURE, i, i) for i in range(n)], dtype=ripple.UPDATE_DTYPE)


def _tups(n):
    return torch.tensor([[I.OP_SET_FEATURE, i, i] for i in range(n)], dtype=torch.int32)


@pytest.mark.parametrize("wrap", [lambda t: t, _Cuda], ids=["host", "device"])
def test_tensors_of_the_wrong_shape_or_type_are_refused(rp, wrap):
    rows, w = torch.zeros(3, D0), torch.ones(3)
    for bad in [dict(feat_rows=torch.zeros(3, D0 - 1)), dict(feat_rows=torch.zeros(3, D0 + 1)), dict(feat_rows=torch.zeros(3 * D0)),
                dict(feat_rows=torch.zeros(3, D0, dtype=torch.float64)), dict(feat_rows=torch.zeros(3, D0, dtype=torch.float16)),
                dict(ups=_tups(3).to(torch.int64)), dict(ups=_tups(3).to(torch.int16)), dict(ups=_tups(3)[:, :2]),
                dict(ups=_tups(3).flatten()), dict(op_weights=torch.ones(3, dtype=torch.float64)), dict(op_weights=torch.ones(3, 2))]:
        args = dict(ups=_tups(3), feat_rows=rows, op_weights=w)
        args.update(bad)
        with pytest.raises((TypeError, ValueError)):
            rp.apply_batch(*(wrap(args[k]) for k in ("ups", "feat_rows", "op_weights")))
    assert rp.lib.calls == []
    rp.apply_batch(wrap(_tups(3)), wrap(rows), wrap(w))
    rp.apply_batch(wrap(_tups(3)), wrap(rows))
    rp.apply_batch(wrap(torch.zeros(0, 3, dtype=torch.int32)), None)
    mem = ripple.MEM_DEVICE if wrap is _Cuda else ripple.MEM_HOST
    assert rp.lib.calls == [(3, 3, mem, True), (3, 3, mem), (0, 0, mem)]


def test_arrays_of_the_wrong_shape_are_refused(rp):
    for rows in (np.zeros((3, D0 - 1), np.float32), np.zeros((3, D0 + 1), np.float32), np.zeros(3 * D0, np.float32)):
        with pytest.raises(ValueError):
            rp.apply_batch(_ups(3), rows)
    with pytest.raises((AssertionError, ValueError)):
        rp.apply_batch(_ups(3), np.zeros((3, D0), np.float32), np.ones(2, np.float32))
    assert rp.lib.calls == []
    rp.apply_batch(_ups(3), np.zeros((3, D0)), np.ones(3))          # other types of host arrays are converted
    rp.apply_batch(_ups(3), np.zeros((6, D0), np.float32)[::2])
    rp.apply_batch(_ups(0), np.zeros((0, D0), np.float32))
    assert [c[:2] for c in rp.lib.calls] == [(3, 3), (3, 3), (0, 0)]


def test_device_arrays_beside_host_operations_are_refused(rp):
    for ups in (_ups(3), _tups(3)):
        with pytest.raises(ValueError):
            rp.apply_batch(ups, _Cuda(torch.zeros(3, D0)))
        with pytest.raises(ValueError):
            rp.apply_batch(ups, torch.zeros(3, D0), _Cuda(torch.ones(3)))
    assert rp.lib.calls == []


def test_strided_host_tensors_are_made_contiguous(rp):
    seen = []
    rp.lib.ripple_apply_batch = lambda h, uptr, n, fptr, nr, mem: seen.append(
        np.ctypeslib.as_array(ctypes.cast(fptr, ctypes.POINTER(ctypes.c_float)), (nr, D0)).copy()) or ripple.OK
    wide = torch.arange(3 * 2 * D0, dtype=torch.float32).reshape(3, 2 * D0)
    rp.apply_batch(_tups(3), wide[:, ::2])
    assert np.array_equal(seen[0], wide[:, ::2].numpy())
