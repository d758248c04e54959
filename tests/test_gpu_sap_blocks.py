"""The staged Schwarz kernel over block shapes: 32 to 256 sites, unequal extents, extents of 2 (every
site on the boundary) up to 32, several right-hand sides split over CTAs, few MR steps."""
import pytest

from oracle.dirac import WilsonClover
from oracle.sap import SchwarzOracle
from paper_0706_2298_gb300 import dwsolve as dw
from paper_0706_2298_gb300 import synth

from .gpu_util import from_packed, rel, to_packed

pytestmark = pytest.mark.gpu

# A cycle applies the block operator about 2 x 12 times one after the other; with FP32 rounding (6e-8) in
# each application and a condition number of the blocks below 10 the error stays below 24 x 6e-8 x 10
# per cycle.
TOL = 1.5e-5


@pytest.mark.parametrize("L,bs,nrhs,ncy,nmr,antiperiodic", [
    ((8, 8, 8, 8), (4, 4, 4, 4), 1, 2, 4, True),
    ((8, 8, 8, 8), (4, 4, 4, 4), 5, 1, 1, True),
    ((16, 8, 8, 4), (8, 4, 4, 2), 2, 2, 4, False),
    ((64, 4, 4, 4), (32, 2, 2, 2), 1, 1, 3, True),
    ((4, 8, 8, 8), (2, 4, 4, 4), 3, 2, 4, True),
    ((32, 4, 4, 4), (16, 2, 2, 2), 1, 2, 3, True),
    ((8, 4, 8, 8), (4, 2, 4, 2), 2, 2, 4, True),
    ((4, 4, 8, 4), (2, 2, 4, 2), 2, 2, 4, False),
    ((8, 8, 8, 8), (4, 4, 4, 4), 2, 1, 0, True),
])
def test_block_shapes(L, bs, nrhs, ncy, nmr, antiperiodic):
    U = synth.random_gauge(L, 31)
    ctx = dw.dw_create(L, -0.1, 1.2, U, bs, antiperiodic)
    sap = SchwarzOracle(WilsonClover(L, U.numpy(), -0.1, 1.2, antiperiodic), bs)
    rho = synth.gaussian_source(L, 32, nrhs).reshape(nrhs, ctx.V, 4, 3)
    xi = ctx.empty_field(dw.DW_F32, nrhs)
    dw.sap_precondition(ctx, dw.DW_F32, ncy, nmr, nrhs, to_packed(ctx, dw.DW_F32, rho), xi)
    got = from_packed(ctx, dw.DW_F32, xi, nrhs).reshape(nrhs, ctx.V, 4, 3)
    for r in range(nrhs):
        assert rel(got[r], sap.apply(rho[r].numpy(), ncy, nmr)) <= TOL
