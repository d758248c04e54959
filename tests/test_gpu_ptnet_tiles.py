"""The network's tiled kernels: several fields per launch (tiles of different fields side by side), more
tiles than thread blocks of a weight gradient and fewer, unequal extents, each layer and its adjoint."""
import numpy as np
import pytest
import torch

from oracle.dirac import WilsonClover
from oracle.ptnet import PTNet, init_weights
from paper_0706_2298_gb300 import dwsolve as dw
from paper_0706_2298_gb300 import synth

from .gpu_util import from_packed, rel, to_packed

pytestmark = pytest.mark.gpu

# Sums of 576 products (a layer) in FP32 chains of 64: 64 roundings of 6e-8 each at most per chain, three
# layers one after the other.
TOL = 3 * 64 * 6e-8


def _flat(W):
    return np.concatenate([w.reshape(-1) for w in W])


@pytest.mark.parametrize("L,bs,nf,antiperiodic", [
    ((4, 4, 4, 4), (2, 2, 2, 2), 1, True),
    ((4, 4, 8, 4), (2, 2, 4, 2), 5, False),
    ((8, 4, 8, 8), (4, 2, 4, 4), 3, True),
])
def test_network_and_gradient(L, bs, nf, antiperiodic):
    U = synth.random_gauge(L, 61)
    ctx = dw.dw_create(L, 0.0, 1.0, U, bs, antiperiodic)
    P = PTNet(WilsonClover(L, U.numpy(), 0.0, 1.0, antiperiodic))
    W = [w.astype(np.complex64).astype(np.complex128) for w in init_weights(16, seed=5, scale=0.5)]
    wd = torch.from_numpy(_flat(W).astype(np.complex64).view(np.float32).copy()).cuda()
    x = synth.complex_gaussian((nf, ctx.V, 4, 3), 62).numpy()
    y = synth.complex_gaussian((nf, ctx.V, 4, 3), 63).numpy()
    xd, yd, out = to_packed(ctx, dw.DW_F32, x), to_packed(ctx, dw.DW_F32, y), ctx.empty_field(dw.DW_F32, nf)
    dw.ptnet_forward(ctx, wd, nf, xd, out)
    got = from_packed(ctx, dw.DW_F32, out, nf).reshape(nf, ctx.V, 4, 3)
    for f in range(nf):
        assert rel(got[f], P.forward(W, x[f])) <= TOL
    g = torch.empty_like(wd)
    loss = dw.ptnet_loss_grad(ctx, wd, nf, xd, yd, g)
    loss_o, G = P.loss_and_grad(W, list(x), list(y))
    assert abs(loss - loss_o) <= TOL * loss_o
    gd, at = g.cpu().numpy().view(np.complex64).astype(np.complex128), 0
    for w in G:
        assert rel(gd[at:at + w.size], w.reshape(-1)) <= TOL
        at += w.size


@pytest.mark.parametrize("adjoint", [0, 1])
def test_layer16(adjoint):
    L = (4, 8, 4, 8)
    U = synth.random_gauge(L, 64)
    ctx = dw.dw_create(L, 0.0, 1.0, U, (2, 4, 2, 4))
    P = PTNet(WilsonClover(L, U.numpy(), 0.0, 1.0))
    w = init_weights(16, seed=6, scale=0.6)[1]
    h = synth.complex_gaussian((16, ctx.V, 4, 3), 65).numpy()
    hx, hy = to_packed(ctx, dw.DW_F32, h), ctx.empty_field(dw.DW_F32, 16)
    dw.ptnet_layer16(ctx, torch.from_numpy(w.astype(np.complex64).view(np.float32).copy()).cuda(), adjoint, 0, hx, hy)
    ref = (P.layer_adjoint if adjoint else P.layer)(w, h.reshape((16,) + L + (4, 3))).reshape(16, ctx.V, 4, 3)
    assert rel(from_packed(ctx, dw.DW_F32, hy, 16), ref) <= TOL
