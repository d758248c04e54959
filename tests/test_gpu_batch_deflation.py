"""Batched deflated solves against one solve per right-hand side: batches that fill, split and leave over the
right-hand-side groups of the batched restriction and prolongation, each compiled group of basis vectors, little
blocks smaller than a thread group, and more than one launch of the multi right-hand-side little solver."""
import pytest
import torch

from paper_0706_2298_gb300 import dwsolve as dw
from paper_0706_2298_gb300 import synth

from .gpu_util import rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,bs,Ns,nrhs", [
    ((8, 8, 8, 8), (4, 4, 4, 4), 8, 2),
    ((8, 8, 8, 8), (4, 4, 4, 4), 20, 2),
    ((8, 8, 8, 8), (4, 4, 4, 4), 20, 5),
    ((8, 8, 8, 8), (4, 4, 4, 4), 20, 13),
    ((16, 8, 8, 8), (4, 4, 4, 4), 16, 7),
    ((8, 8, 8, 8), (4, 4, 4, 4), 24, 3),
    ((8, 8, 8, 8), (4, 4, 4, 4), 32, 4),
    ((8, 8, 4, 4), (2, 2, 2, 2), 8, 6),
    ((8, 4, 4, 8), (4, 2, 2, 4), 12, 3),
])
def test_batch_against_single(L, bs, Ns, nrhs, monkeypatch):
    ctx = dw.dw_create(L, -0.2, 1.0, synth.random_gauge(L, 61), (4, 4, 4, 4) if min(L) > 4 else (2, 2, 2, 2))
    d = dw.deflation_build(ctx, bs, Ns, 3, 4, 4, synth.start_fields(L, Ns, 62).cuda(), basis_prec=dw.DW_BF16,
                           iter_prec=dw.DW_F32)
    eta = synth.gaussian_source(L, 63, nrhs=nrhs).cuda()
    p = dw.sol_params(tol=1e-10, nkv=16, mixed=1)
    out = []
    for flag in (None, "0"):
        if flag:
            monkeypatch.setenv("DW_BATCH", flag)
        psi = torch.empty_like(eta)
        rc, infos = dw.gcr_solve(ctx, d, p, nrhs, eta, psi)
        assert rc == dw.DW_OK
        out.append((psi.cpu().numpy(), [i.iterations for i in infos]))
    # both solve to 1e-10: they agree to the conditioning of D (below 100 here) times the tolerance, and rounding
    # of the FP32 preconditioner moves the step that meets it by one at most per restart (a wrong coarse
    # solution would leave the low modes in and cost more)
    assert rel(out[0][0], out[1][0]) <= 1e-8
    assert max(abs(a - b) for a, b in zip(*(o[1] for o in out))) <= 3
