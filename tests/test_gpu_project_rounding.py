"""Rounding of the FP32 restriction and prolongation with the BF16 basis: the distance from FP64 sums of the same
numbers against that of plain FP32 sums, in which each product and sum is rounded by itself: the products of a site one
after the other, the sites of a block pairwise; the basis vectors one after the other.  Chains of fused
multiply-adds over all terms are 10% (restriction) and 26% (prolongation) further from FP64, by the count of roundings and
the sizes of the sums they happen at."""
import numpy as np
import pytest
import torch

from oracle.sap import Blocking
from paper_0706_2298_gb300 import dwsolve as dw
from paper_0706_2298_gb300 import synth

from .gpu_util import from_packed, rel, to_packed

pytestmark = pytest.mark.gpu

BOUND = 1.05      # the errors of 10240 or more numbers each: 1% by chance


def product(ar, ai, br, bi):
    """(a b) with every operation rounded by itself."""
    return ar * br - ai * bi, ar * bi + ai * br


def parts(z, dtype):
    return z.real.astype(dtype), z.imag.astype(dtype)


def restriction(phi, psi, dtype):
    """phi[Ns, Nb, sites, 12], psi[Nb, sites, 12]"""
    pr, pi = parts(psi, dtype)
    fr, fi = parts(phi, dtype)
    re, im = np.zeros(phi.shape[:3], dtype), np.zeros(phi.shape[:3], dtype)
    for j in range(12):
        x, y = product(fr[..., j], -fi[..., j], pr[..., j], pi[..., j])
        re, im = re + x, im + y
    while re.shape[-1] > 1:
        re, im = re[..., ::2] + re[..., 1::2], im[..., ::2] + im[..., 1::2]
    return (re[..., 0].astype(np.float64) + 1j * im[..., 0]).T


def prolongation(phi, c, dtype):
    """phi as above, c[Nb, Ns]"""
    cr, ci = parts(c, dtype)
    re, im = np.zeros(phi.shape[1:], dtype), np.zeros(phi.shape[1:], dtype)
    for k in range(phi.shape[0]):
        x, y = product(cr[:, k, None, None], ci[:, k, None, None], *parts(phi[k], dtype))
        re, im = re + x, im + y
    return re.astype(np.float64) + 1j * im


@pytest.mark.parametrize("L,bs,Ns", [
    ((16, 16, 16, 16), (4, 4, 4, 4), 20),          # 128 threads per block of the prolongation
    ((24, 16, 16, 16), (4, 4, 4, 4), 8),           # 256
])
def test_error_against_plain_single_precision(L, bs, Ns):
    ctx = dw.dw_create(L, 0.0, 1.0, synth.random_gauge(L, 71, device="cuda"), bs)
    d = dw.deflation_build(ctx, bs, Ns, 1, 2, 4, synth.start_fields(L, Ns, 72).cuda())
    basis = torch.empty((Ns, ctx.V, 4, 3), dtype=torch.complex128, device="cuda")
    dw.dfl_basis_export(d, basis)
    blocks = Blocking(L, bs)
    phi = basis.cpu().numpy().reshape(Ns, ctx.V, 12)[:, blocks.sites]
    psi = synth.gaussian_source(L, 73).to(torch.complex64).to(torch.complex128)
    c = torch.empty((d.Nb * Ns, 2), dtype=torch.float32, device="cuda")
    dw.dfl_restrict(d, dw.DW_F32, to_packed(ctx, dw.DW_F32, psi), c)
    got = c.double().cpu().numpy().reshape(d.Nb, Ns, 2)
    x = psi.numpy().reshape(ctx.V, 12)[blocks.sites]
    want = restriction(phi, x, np.float64)
    assert rel(got[..., 0] + 1j * got[..., 1], want) <= BOUND * rel(restriction(phi, x, np.float32), want)

    c = torch.randn((d.Nb, Ns, 2), generator=torch.Generator().manual_seed(74))
    out = ctx.empty_field(dw.DW_F32)
    dw.dfl_prolong(d, dw.DW_F32, c.cuda(), out)
    got = from_packed(ctx, dw.DW_F32, out).reshape(ctx.V, 12)[blocks.sites]
    z = c.double().numpy()[..., 0] + 1j * c.double().numpy()[..., 1]
    want = prolongation(phi, z, np.float64)
    assert rel(got, want) <= BOUND * rel(prolongation(phi, z, np.float32), want)


@pytest.mark.parametrize("Ns,nrhs", [(3, 2), (5, 2), (5, 6), (6, 4), (7, 5), (13, 3)])
def test_batch_with_remaining_vectors(Ns, nrhs, monkeypatch):
    """The batched prolongation takes four basis vectors at a time, those that remain one by one.  (Without them
    the coarse corrections miss a mode and the solver does not reach 1e-10 in a similar number of steps.)"""
    L = (8, 8, 8, 8)
    ctx = dw.dw_create(L, -0.1, 1.0, synth.random_gauge(L, 75), (4, 4, 4, 4))
    d = dw.deflation_build(ctx, (4, 4, 4, 4), Ns, 3, 4, 4, synth.start_fields(L, Ns, 76).cuda())
    eta = synth.gaussian_source(L, 77, nrhs=nrhs).cuda()
    p = dw.sol_params(tol=1e-10, nkv=16, mixed=1)
    out = []
    for flag in ("1", "0"):
        monkeypatch.setenv("DW_BATCH", flag)
        psi = torch.empty_like(eta)
        rc, infos = dw.gcr_solve(ctx, d, p, nrhs, eta, psi)
        assert rc == dw.DW_OK
        out.append((psi.cpu().numpy(), max(i.iterations for i in infos)))
    assert rel(out[0][0], out[1][0]) <= 1e-8       # the tolerance times the condition of D (below 100)
    assert out[0][1] <= 1.5 * out[1][1]
