"""The FP32 little solver's kernel where its thread blocks own unequal numbers of little-block rows, so that they reach
the grid barriers of a step at different times: every vector that another thread block gathers has to be final by
then.  Solves of a right-hand side of size 1e12 and of size 1 alternate, so that whatever a solve leaves in the workspace
is wrong by twelve orders of magnitude for the next one.  And right-hand sides so small that the squares of FP32
vectors underflow: a step whose vector vanishes is not used."""
import pytest
import torch

from paper_0706_2298_gb300 import dwsolve as dw
from paper_0706_2298_gb300 import synth

pytestmark = pytest.mark.gpu


def solve(d, w, tol):
    v = torch.full_like(w, float("nan"))
    rc, it, rr = dw.little_dirac_solve(d, dw.DW_F32, w, v, tol, 500)
    return rc, it, rr, v


# even block rows per thread block (152 of them), the last one's in brackets; slices of the vectors in shared memory or not
@pytest.mark.parametrize("L,Ns", [
    ((16, 12, 16, 16), 20),       # 11 (7), in shared memory
    ((20, 16, 16, 16), 8),        # 17 (10), in shared memory
    ((20, 16, 16, 16), 24),       # 17 (10), not in shared memory
    ((24, 16, 16, 16), 20),       # 21 (6), not in shared memory, two chunks of rows
])
def test_unequal_rows(L, Ns, monkeypatch):
    ctx = dw.dw_create(L, 0.0, 1.0, synth.random_gauge(L, 51, device="cuda"), (2, 2, 2, 2))
    start = synth.start_fields(L, Ns, 52).cuda()
    tol = 1e-6
    d = dw.deflation_build(ctx, (2, 2, 2, 2), Ns, 1, 2, 4, start)
    w = torch.view_as_real(synth.complex_gaussian((3, d.Nb * Ns), 53)).to(torch.float32).contiguous().cuda()
    monkeypatch.setenv("DW_COOP_RING", "0")
    ref = dw.deflation_build(ctx, (2, 2, 2, 2), Ns, 1, 2, 4, start)      # the generic kernel
    want = [solve(ref, x, tol) for x in w]
    monkeypatch.delenv("DW_COOP_RING")
    for n in range(24):
        x = w[n % 3]
        big = solve(d, 1e12 * x, tol)
        rc, it, rr, v = solve(d, x, tol)
        assert rc == dw.DW_OK and big[0] == dw.DW_OK
        assert bool(torch.isfinite(v).all()) and bool(torch.isfinite(big[3]).all())
        assert abs(it - want[n % 3][1]) <= 1 and abs(big[1] - want[n % 3][1]) <= 1
        # residuals of 1e-6 each and a condition number below 10
        assert float((v - want[n % 3][3]).norm() / v.norm()) <= 2e-5


@pytest.mark.parametrize("size", [1e-16, 1e-18, 1e-19, 1e-20, 1e-21, 1e-22, 3e-23, 1e-23, 1e-30])
def test_vanishing_right_hand_side(size):
    L, Ns = (8, 8, 8, 8), 8
    ctx = dw.dw_create(L, 0.0, 1.0, synth.random_gauge(L, 54), (4, 4, 4, 4))
    d = dw.deflation_build(ctx, (4, 4, 4, 4), Ns, 1, 2, 4, synth.start_fields(L, Ns, 55).cuda())
    w = torch.view_as_real(synth.complex_gaussian((d.Nb * Ns,), 56)).to(torch.float32).contiguous().cuda()
    one = solve(d, w, 1e-4)
    assert one[0] == dw.DW_OK
    rc, it, rr, v = solve(d, size * w, 1e-4)
    assert bool(torch.isfinite(v).all())
    if size >= 1e-16:             # squares down to 1e-4 of the right-hand side are normal numbers: the same solution
        assert rc == dw.DW_OK and abs(it - one[1]) <= 1
        assert float((v.double() / size - one[3].double()).norm() / one[3].double().norm()) <= 2e-3
