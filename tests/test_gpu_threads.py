"""Several threads, each on a stream of its own, making their first double-float calls on one context at once."""
import threading

import pytest
import torch

from paper_0706_2298_gb300 import dwsolve as dw
from paper_0706_2298_gb300 import synth

from .gpu_util import to_packed

pytestmark = pytest.mark.gpu


def test_first_double_float_calls_from_threads():
    L, n = (8, 8, 8, 8), 8
    U = synth.random_gauge(L, 81)
    x = synth.gaussian_source(L, 82)
    for _ in range(4):
        ctx = dw.dw_create(L, 0.0, 1.0, U, (4, 4, 4, 4))
        # a mixed solve makes the double-float links, but takes no scratch memory
        eta = x.cuda()
        dw.gcr_solve(ctx, None, dw.sol_params(tol=1e-1, nmx=4, mixed=1), 1, eta, torch.empty_like(eta))
        f = to_packed(ctx, dw.DW_F64, x)
        out = [torch.empty_like(f) for _ in range(n)]
        streams = [torch.cuda.Stream() for _ in range(n)]
        torch.cuda.synchronize()
        start, errors = threading.Barrier(n), []

        def call(i):
            try:
                start.wait()
                for _ in range(5):
                    dw.dw_apply(ctx, dw.DW_F64X, dw.DW_OP_FULL, 1, f, out[i], stream=streams[i].cuda_stream)
                streams[i].synchronize()
            except Exception as e:
                errors.append(e)

        ts = [threading.Thread(target=call, args=(i,)) for i in range(n)]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
        assert not errors
        want = torch.empty_like(f)
        dw.dw_apply(ctx, dw.DW_F64X, dw.DW_OP_FULL, 1, f, want)
        torch.cuda.synchronize()
        assert all(torch.equal(o, want) for o in out)
