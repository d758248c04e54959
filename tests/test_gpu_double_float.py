"""The double-float D (DW_F64X) with its run-time directions: every direction and wrap on small unequal
lattices, several fields per call, and calls interleaved on two streams (scratch of the context's pool)."""
import pytest
import torch

from oracle.dirac import WilsonClover
from paper_0706_2298_gb300 import dwsolve as dw
from paper_0706_2298_gb300 import synth

from .gpu_util import from_packed, rel, to_packed

pytestmark = pytest.mark.gpu

# a component is a sum of about 100 terms with 2^-48 relative error each: 100 x 3.6e-15 at most
TOL = 1e-13


@pytest.mark.parametrize("L,bs,nrhs,antiperiodic", [
    ((4, 4, 4, 4), (2, 2, 2, 2), 1, True),
    ((4, 4, 8, 4), (2, 2, 4, 2), 3, False),
    ((8, 4, 4, 16), (4, 2, 2, 4), 2, True),
])
def test_dirac_f64x(L, bs, nrhs, antiperiodic):
    U = synth.random_gauge(L, 71)
    ctx = dw.dw_create(L, -0.1, 1.3, U, bs, antiperiodic)
    D = WilsonClover(L, U.numpy(), -0.1, 1.3, antiperiodic)
    psi = synth.gaussian_source(L, 72, nrhs).reshape(nrhs, ctx.V, 4, 3)
    x = to_packed(ctx, dw.DW_F64, psi)
    y = ctx.empty_field(dw.DW_F64, nrhs)
    dw.dw_apply(ctx, dw.DW_F64X, dw.DW_OP_FULL, nrhs, x, y)
    got = from_packed(ctx, dw.DW_F64, y, nrhs).reshape(nrhs, ctx.V, 4, 3)
    for r in range(nrhs):
        assert rel(got[r], D.apply(psi[r].numpy())) <= TOL


def test_two_streams():
    L = (8, 8, 8, 8)
    U = synth.random_gauge(L, 73)
    ctx = dw.dw_create(L, -0.1, 1.0, U, (4, 4, 4, 4))
    x = [to_packed(ctx, dw.DW_F64, synth.gaussian_source(L, 74 + k)) for k in range(2)]
    ref, y = [torch.empty_like(v) for v in x], [torch.empty_like(v) for v in x]
    for k in range(2):
        dw.dw_apply(ctx, dw.DW_F64X, dw.DW_OP_FULL, 1, x[k], ref[k])
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    for _ in range(20):
        for k in range(2):
            dw.dw_apply(ctx, dw.DW_F64X, dw.DW_OP_FULL, 1, x[k], y[k], stream=streams[k])
    torch.cuda.synchronize()
    for k in range(2):
        assert torch.equal(ref[k], y[k])
