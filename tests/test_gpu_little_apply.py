"""The little operator on full vectors against its definition, restriction x D x prolongation: compiled and generic
numbers of basis vectors, odd ones, and rows that fill their last warp or not."""
import pytest
import torch

from paper_0706_2298_gb300 import dwsolve as dw
from paper_0706_2298_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ns", [1, 7, 12, 20, 32])
def test_little_apply_definition(Ns):
    L, bs = (8, 8, 8, 4), (4, 4, 4, 2)
    ctx = dw.dw_create(L, -0.1, 1.3, synth.random_gauge(L, 71), (4, 4, 4, 2))
    d = dw.deflation_build(ctx, bs, Ns, 1, 2, 4, synth.start_fields(L, Ns, 72).cuda())
    v = torch.view_as_real(synth.complex_gaussian((d.Nb * Ns,), 73)).to(torch.float64).contiguous().cuda()
    w, ref = torch.empty_like(v), torch.empty_like(v)
    dw.little_apply(d, v, w)
    psi, dpsi = ctx.empty_field(dw.DW_F64), ctx.empty_field(dw.DW_F64)
    dw.dfl_prolong(d, dw.DW_F64, v, psi)
    dw.dw_apply(ctx, dw.DW_F64, dw.DW_OP_FULL, 1, psi, dpsi)
    dw.dfl_restrict(d, dw.DW_F64, dpsi, ref)
    # FP64 sums of at most 256 x 12 (restriction) and 9 x 32 terms: a few 1e-15
    assert float((w - ref).norm() / ref.norm()) <= 1e-13
