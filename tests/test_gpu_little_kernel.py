"""The FP32 little solver's kernel for compiled Ns against the generic cooperative kernel (the one that is
pinned on dense solves): every compiled Ns, thread blocks without rows (16 little blocks), and more than 16
block rows per thread block with slices too large for shared memory."""
import pytest
import torch

from paper_0706_2298_gb300 import dwsolve as dw
from paper_0706_2298_gb300 import synth

pytestmark = pytest.mark.gpu

# both solutions have a relative residual of 1e-5; the even-odd deflated systems of these random
# subspaces are well conditioned (below 10), so the solutions differ by less than 2 x 1e-5 x 10 / 2
TOL, SOL = 1e-5, 1e-4


@pytest.mark.parametrize("L,bs,Ns", [
    ((8, 8, 8, 8), (4, 4, 4, 4), 12),
    ((8, 8, 8, 8), (4, 4, 4, 4), 16),
    ((8, 8, 8, 8), (4, 4, 4, 4), 24),
    ((8, 8, 8, 8), (4, 4, 4, 4), 32),
    ((16, 8, 8, 8), (2, 2, 2, 2), 8),
    ((24, 16, 16, 16), (2, 2, 2, 2), 20),
])
def test_against_generic_kernel(L, bs, Ns, monkeypatch):
    ctx = dw.dw_create(L, 0.0, 1.0, synth.random_gauge(L, 41, device="cuda"), bs)
    start = synth.start_fields(L, Ns, 42).cuda()
    out = []
    for flag in (None, "0"):
        if flag:
            monkeypatch.setenv("DW_COOP_RING", flag)
        d = dw.deflation_build(ctx, bs, Ns, 1, 2, 4, start)
        w = synth.complex_gaussian((d.Nb * Ns,), 43)
        wt = torch.view_as_real(w).to(torch.float32).contiguous().cuda()
        vt = torch.empty_like(wt)
        rc, it, rr = dw.little_dirac_solve(d, dw.DW_F32, wt, vt, TOL, 500)
        assert rc == dw.DW_OK and rr <= TOL
        out.append((vt.double(), it))
    assert float((out[0][0] - out[1][0]).norm() / out[1][0].norm()) <= SOL
    assert abs(out[0][1] - out[1][1]) <= 2
