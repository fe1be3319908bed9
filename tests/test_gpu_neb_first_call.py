"""The first call of a model with nebular emission allocates nothing beyond the
workspace its stream has: the memory in use stays as it was, and it can be the
call that a CUDA graph captures.  Under a memory budget or a precision mask the
grid keeps no table beside the template; the results are the same bit for bit."""
import numpy as np
import pytest

import synth
from tests import cases

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_first_nebular_call():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_30145_gb300 import build
    build.build()
    import dataclasses

    from paper_2609_30145_gb300 import Context, _ffi
    w = synth.shrink(synth.WORKLOADS["phot_107x12x6000_b1024"], n_age=20, n_feh=4, n_lam=1500, n_sfh=10)
    orc = cases.oracle_for(w)
    th32, _ = cases.theta_pair(w, 200, seed=97)
    theta = torch.from_numpy(th32).cuda()
    got, loaded = [], []
    for budget, mask in ((0, 0), (1 << 30, 0), (0, _ffi.GRID_COPY_FP32)):
        ctx = Context(0, hbm_budget_bytes=budget)
        ctx._grid_ids = {id(orc.grid): (ctx.load_grid(orc.grid, precision_mask=mask), orc.grid)}
        loaded.append(ctx.memory_used())
        plain = cases.gpu_model_for(ctx, orc, dataclasses.replace(w, use_nebular=0))
        neb = cases.gpu_model_for(ctx, orc, w)
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            plain.loglike(theta, "fp32")
            plain.loglike_grad(theta, "fp32")
            neb_lnl = torch.empty(200, dtype=torch.float64, device="cuda")
            st = torch.empty(200, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        used = ctx.memory_used()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):   # its first call
            neb.loglike(theta, "fp32", out=neb_lnl, status=st)
        neb_lnl.zero_()
        graph.replay()
        torch.cuda.synchronize()
        captured = neb_lnl.cpu().numpy()
        with torch.cuda.stream(stream):
            direct = neb.loglike(theta, "fp32")[0]
            phot = neb.forward(theta, "fp32")[0]
        torch.cuda.synchronize()
        assert ctx.memory_used() == used
        assert np.array_equal(direct.cpu().numpy(), captured)
        got.append((captured, phot.cpu().numpy()))
        ctx.close()
    assert loaded[0] - loaded[1] == 16 * 7 * 12 * 1500   # the table of a cell's four corners
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert np.array_equal(a, b)
