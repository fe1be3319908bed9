"""Uncalibrated spectra of far more pixels than the window has nodes need no
shared memory per pixel: forward spectra and lnL of 60001 pixels on a grid of 300
nodes against the FP64 oracle, with and without the spectral noise floor, in
launches of 512 threads per row (3 rows) and of 128, which must agree bit for
bit."""
import numpy as np
import pytest

import synth
from tests import cases

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N_PIX = 60001


@pytest.mark.parametrize("kind", ["specphot_afe_107x12x5x6000_b2048", "specphot_afe_floor_107x12x5x6000_b2048"])
def test_sixty_thousand_pixels(kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_30145_gb300 import build
    build.build()
    from paper_2609_30145_gb300 import Context
    ctx = Context(0)
    w = synth.shrink(synth.WORKLOADS[kind], n_age=16, n_feh=3, n_lam=300, n_sfh=6, n_pix=N_PIX)
    orc = cases.oracle_for(w, lsf_r=np.geomspace(20.0, 500.0, N_PIX))
    model = cases.gpu_model_for(ctx, orc, w)
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    th32, th64 = cases.theta_pair(w, 4 * sm + 5, seed=41, orc=orc)
    theta = torch.from_numpy(th32).cuda()
    lnl, spec = model.loglike(theta, "fp32")[0], model.forward(theta, "fp32")[1]
    assert torch.equal(model.loglike(theta[:3], "fp32")[0], lnl[:3])
    assert torch.equal(model.forward(theta[:3], "fp32")[1], spec[:3])
    ref = orc.eval(th64[:3])
    assert not ref["status"].any()
    scale = np.abs(ref["spec"]).max(axis=1, keepdims=True)
    # the FP32 flux and lnL tolerances of the parity tests
    assert np.max(np.abs(spec[:3].cpu().numpy() - ref["spec"]) / np.maximum(np.abs(ref["spec"]), 1e-6 * scale)) < 2e-5
    assert np.max(np.abs(lnl[:3].cpu().numpy() - ref["lnl"]) / cases.lnl_scale(orc, ref)) < 1e-5
    ctx.close()
