"""Tensors over the library's buffers are wrapped once and handed out again: on the context's device, as ordinary tensors,
whatever device or mode was current at the first call."""
import ctypes
import types

import pytest
import torch

from paper_2601_12347_b200 import inputs as I
from paper_2601_12347_b200 import ripple

import test_gpu_parity as G

env = G.env


def test_a_buffer_is_wrapped_on_its_context_s_device():
    asked = []

    def as_tensor(arr, device):
        asked.append(torch.device(device))
        return torch.zeros(3)
    r = ripple.Ripple.__new__(ripple.Ripple)
    r._torch = types.SimpleNamespace(as_tensor=as_tensor, inference_mode=torch.inference_mode, Tensor=torch.Tensor)
    r._device, r._views, r._handle, r.h, r.n, r.dims = torch.device("cuda", 1), {}, None, ctypes.c_void_p(None), 3, [2, 2]
    ok = lambda *a: ripple.OK  # noqa: E731
    r.lib = types.SimpleNamespace(ripple_get_embeddings=ok, ripple_get_aggregate=ok, ripple_get_affected=ok, ripple_get_degrees=ok)
    r.embeddings(1), r.aggregate(1), r.affected(1), r.degrees()
    assert asked == [torch.device("cuda", 1)] * 5
    with pytest.raises(TypeError):       # though 1.0 == 1
        r.embeddings(1.0)


def test_a_first_call_in_inference_mode_leaves_ordinary_tensors():
    r = ripple.Ripple.__new__(ripple.Ripple)
    r._torch, r._device, r._views = torch, torch.device("cpu"), {}
    with torch.inference_mode():
        r._view("x", lambda: [1.0, 2.0])
    t = r._view("x", lambda: None)
    assert not t.is_inference()
    w = torch.ones(2, requires_grad=True)
    (t * w).sum().backward()
    assert w.grad.tolist() == [1.0, 2.0]


@pytest.mark.gpu
def test_views_read_in_inference_mode_serve_training_too(env):
    ripple_, _ = env
    model = I.sage_model([18, 36, 10], I.AGG_MEAN)
    src, dst = I.er_graph(300, 2000, 3)
    rp = ripple_.Ripple(300, src, dst, I.features(300, 18, 3), model, I.make_weights(model, 3))
    with torch.inference_mode():
        rp.embeddings(2), rp.affected(2), rp.degrees()
    w = torch.ones(10, 1, device="cuda", requires_grad=True)
    (rp.embeddings(2) @ w).sum().backward()
    assert torch.allclose(w.grad[:, 0], rp.embeddings(2).sum(0), rtol=1e-4)
    assert not rp.affected(2).is_inference() and not rp.degrees()[0].is_inference()
    rp.close()


@pytest.mark.gpu
def test_buffers_are_wrapped_when_they_are_allocated(env, monkeypatch):
    ripple_, _ = env
    model = I.sage_model([18, 36, 10], I.AGG_MEAN)
    src, dst = I.er_graph(300, 2000, 3)
    rp = ripple_.Ripple(300, src, dst, I.features(300, 18, 3), model, I.make_weights(model, 3))
    old = rp.embeddings(1)
    for n in (300, 400):
        if n == 400:
            rp.reserve_vertices(n)
        with monkeypatch.context() as m:
            m.setattr(torch, "as_tensor", None)
            assert [rp.embeddings(l).shape for l in range(3)] == [(n, 18), (n, 36), (n, 10)]
            assert rp.degrees()[0].shape == (n,) and rp.affected(0).numel() == 0
    assert rp.embeddings(1).data_ptr() != old.data_ptr()
    rp.close()
