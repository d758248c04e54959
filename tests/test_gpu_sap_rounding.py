"""Rounding of the FP32 Schwarz procedure: its distance from the FP64 oracle against that of a plain FP32
restatement (the oracle's steps on complex64 arrays, in which the hops have a sum of their own and each product and sum
is rounded by itself).  An order of summation that rounds at the size of the clover term in every addition is
half as far again from FP64."""
import numpy as np
import pytest

import oracle.dirac as od
from oracle.dirac import WilsonClover
from oracle.sap import SchwarzOracle
from paper_0706_2298_gb300 import dwsolve as dw
from paper_0706_2298_gb300 import synth

from .gpu_util import from_packed, rel, to_packed

pytestmark = pytest.mark.gpu


class Single(WilsonClover):
    """An operator's matrices, and its arithmetic, in complex64."""

    def __init__(self, D):
        self.__dict__.update(D.__dict__)
        self.C, self._Cinv = D.C.astype(np.complex64), D.Cinv.astype(np.complex64)
        self.Uf = [u.astype(np.complex64) for u in D.Uf]

    def _grid(self, psi):
        return psi.reshape((-1,) + self.L + (4, 3)), psi.ndim == 3, psi.shape


def plain_single(D, bs, rho, ncy, nmr, monkeypatch):
    monkeypatch.setattr(od, "GAMMA", [g.astype(np.complex64) for g in od.GAMMA])
    monkeypatch.setattr(od, "_I4", od._I4.astype(np.complex64))
    sap = SchwarzOracle(Single(D), bs)
    per_site = sap.blk.per_site
    sap.blk.per_site = lambda v: per_site(v).astype(np.complex64)
    out = sap.apply(rho.astype(np.complex64), ncy, nmr)
    assert out.dtype == np.complex64
    monkeypatch.undo()
    return out


# 10%: the two errors are those of about 1e5 differently rounded numbers each, through operators of the same condition
@pytest.mark.parametrize("bs,ncy,nmr,staged", [
    ((4, 4, 4, 4), 4, 4, "1"),          # 256 sites: tensor memory, two warp quadruples
    ((4, 4, 4, 2), 2, 4, "1"),          # 128 sites: tensor memory
    ((4, 4, 2, 2), 2, 4, "1"),          # 64 sites: shared memory
    ((4, 2, 2, 2), 2, 3, "1"),          # 32 sites: both parities in one warp
    ((4, 4, 4, 4), 2, 4, "0"),          # the generic kernel
])
def test_error_against_plain_single_precision(bs, ncy, nmr, staged, monkeypatch):
    L = (8, 8, 8, 8)
    U = synth.random_gauge(L, 31)
    D = WilsonClover(L, U.numpy(), 0.0, 1.0)
    rho = synth.gaussian_source(L, 32).numpy()
    want = SchwarzOracle(D, bs).apply(rho, ncy, nmr)
    plain = rel(plain_single(D, bs, rho, ncy, nmr, monkeypatch), want)
    monkeypatch.setenv("DW_SAP_STAGED", staged)
    ctx = dw.dw_create(L, 0.0, 1.0, U, bs)
    xi = ctx.empty_field(dw.DW_F32)
    dw.sap_precondition(ctx, dw.DW_F32, ncy, nmr, 1, to_packed(ctx, dw.DW_F32, rho), xi)
    assert rel(from_packed(ctx, dw.DW_F32, xi), want) <= 1.1 * plain
