"""Gradients of the jump network at the edges of the backward kernels' tiles
(128 pixels x 2 rows of the weight-gradient kernel, 32 x 8 cells of the end
layers), against the FP64 oracle with the bounds derived in test_gpu_net."""
import numpy as np
import pytest

from oracle import net as onet
from paper_2105_09671_gb300 import _lib as L

from test_gpu_net import C_GRAD, TOL_GRAD, TOL_OUT, _elementwise_ratio, _flat, _params, _rel, _shape_args, _unflat

pytestmark = pytest.mark.gpu

SHAPES = [(2, (3, 7, 127)), (2, (2, 8, 128)), (2, (1, 9, 129)), (2, (2, 33, 33)), (2, (1, 16, 32)), (2, (5, 1, 1)),
          (3, (1, 3, 7, 129)), (3, (2, 2, 9, 33)), (3, (1, 1, 8, 32))]


@pytest.mark.parametrize("ndim,shape", SHAPES)
def test_gradients_at_tile_edges(ndim, shape):
    import torch
    params = _params(ndim, seed=11)
    rng = np.random.default_rng(13)
    phi = rng.uniform(-1, 1, size=shape).astype(np.float32).astype(np.float64)
    target = (phi + 0.1 * rng.uniform(-1, 1, size=shape)).astype(np.float32).astype(np.float64)
    scale = 0.1
    loss_ref, grads_ref = onet.loss_and_grads(params, phi, target, scale, ndim)
    h = L.ac_net_create(ndim, torch.cuda.current_stream().cuda_stream)
    try:
        L.ac_net_set_params(h, _flat(params))
        d_phi = torch.tensor(phi, dtype=torch.float32, device="cuda")
        d_tgt = torch.tensor(target, dtype=torch.float32, device="cuda")
        b, nx, ny, nz = _shape_args(ndim, shape)
        if nz == 1 and ndim == 3:  # the binding sizes the gradient by nz; ask the library for 3D
            g = np.empty(L.ac_net_param_count(3), dtype=np.float32)
            import ctypes
            loss = ctypes.c_double()
            L.check(L.lib().ac_net_loss_grads(ctypes.c_void_p(h), ctypes.c_void_p(d_phi.data_ptr()),
                                              ctypes.c_void_p(d_tgt.data_ptr()), b, nx, ny, nz, scale,
                                              ctypes.byref(loss), g.ctypes.data_as(ctypes.c_void_p)))
            loss = loss.value
        else:
            loss, g = L.ac_net_loss_grads(h, d_phi.data_ptr(), d_tgt.data_ptr(), b, nx, ny, nz, scale,
                                          want_grads=True)
    finally:
        L.ac_net_destroy(h)
    assert loss == pytest.approx(loss_ref, rel=TOL_OUT)
    for li, ((gw, gb), (rw, rb)) in enumerate(zip(_unflat(g.astype(np.float64), params), grads_ref)):
        for got, ref in ((gw, rw), (gb, rb)):
            assert _rel(got, ref) <= TOL_GRAD, f"layer {li}"
            assert _elementwise_ratio(got, ref) <= C_GRAD, f"layer {li}"


@pytest.mark.parametrize("ndim,shape", [(2, (2, 9, 40)), (3, (1, 5, 6, 33))])
@pytest.mark.parametrize("bias", [-30.0, -1e10, -1e13, -1e18, 1e10, 1e13, 1e18])
@pytest.mark.parametrize("layer", [0, 2, 4])
def test_saturated_units_pass_no_gradient_or_all_of_it(ndim, shape, bias, layer):
    # pre-activations at which gelu' is 0 or 1 exactly (FP32): with negative ones the
    # layers before get gradient 0; with positive ones and the next layer's weights 0
    # (and the loss finite) it is 0 as well, and every gradient is finite
    import torch
    params = [(w.copy(), b.copy()) for w, b in _params(ndim, seed=11)]
    params[layer][1][:] = bias
    if bias > 0:
        params[layer + 1][0][:] = 0.0
    rng = np.random.default_rng(13)
    phi = rng.uniform(-1, 1, size=shape)
    h = L.ac_net_create(ndim, torch.cuda.current_stream().cuda_stream)
    try:
        L.ac_net_set_params(h, _flat(params))
        d_phi = torch.tensor(phi, dtype=torch.float32, device="cuda")
        d_tgt = d_phi + 0.1
        b, nx, ny, nz = _shape_args(ndim, shape)
        loss, g = L.ac_net_loss_grads(h, d_phi.data_ptr(), d_tgt.data_ptr(), b, nx, ny, nz, 0.1, want_grads=True)
    finally:
        L.ac_net_destroy(h)
    assert np.isfinite(loss)
    for li, (gw, gb) in enumerate(_unflat(g.astype(np.float64), params)):
        if li <= layer:
            assert np.max(np.abs(gw)) == 0.0 and np.max(np.abs(gb)) == 0.0, f"layer {li}"
        elif bias < 0:
            assert np.isfinite(gw).all() and np.isfinite(gb).all(), f"layer {li}"


def test_buffers_are_cleared_in_the_order_of_the_networks_stream():
    # a network on a non-blocking stream, the legacy stream busy: the zero ghost
    # ring of its gradients must not wait for that stream
    import torch
    params = _params(2, seed=11)
    rng = np.random.default_rng(13)
    phi = rng.uniform(-1, 1, size=(4, 70, 150)).astype(np.float32)
    d_phi = torch.tensor(phi, device="cuda")
    d_tgt = d_phi + 0.1
    big = torch.rand((8192, 8192), device="cuda")
    grads = []
    for busy in (False, True):
        stream = torch.cuda.Stream()
        h = L.ac_net_create(2, stream.cuda_stream)
        try:
            L.ac_net_set_params(h, _flat(params))
            torch.cuda.synchronize()
            if busy:
                for _ in range(20):
                    big @ big
            _, g = L.ac_net_loss_grads(h, d_phi.data_ptr(), d_tgt.data_ptr(), 4, 150, 70, 1, 0.1, want_grads=True)
            grads.append(g.astype(np.float64))
        finally:
            L.ac_net_destroy(h)
    assert _rel(grads[1], grads[0]) <= 1e-5  # (FP32 sums in another order)
