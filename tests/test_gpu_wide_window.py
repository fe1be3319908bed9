"""The widest window a spectrum can have: 19190 nodes take all of a CTA's shared
memory but for what the kernel declares, so that the bands' extents and data
are read from the model.  Spectrum, photometry and lnL against the FP64 oracle;
the same model on a grid of 19100 nodes, whose bands fit."""
import numpy as np
import pytest

import synth
from tests import cases

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_lam", [19190, 19100])
def test_widest_window(n_lam):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_30145_gb300 import build
    build.build()
    from paper_2609_30145_gb300 import Context
    ctx = Context(0)
    w = synth.shrink(synth.WORKLOADS["specphot_afe_107x12x5x6000_b2048"], n_age=16, n_feh=3, n_lam=n_lam, n_sfh=6,
                     n_pix=400)
    w.grid_kw["lam_um"] = (0.4, 2.0)   # the bands and pixels (0.6 to 5.3 um) span more than the grid
    orc = cases.oracle_for(w, with_data=False)
    th32, _ = cases.theta_pair(w, 40, seed=43)
    th32[:, cases.z_column(w.n_sfh, w.zmode)] = np.linspace(0.7, 1.4, 40).astype(np.float32)
    th64 = th32.astype(np.float64)
    true = orc.eval(th64[20:21])
    ph, sp = true["phot"][0], true["spec"][0]
    orc.set_data(phot_d=1.03 * ph, phot_sigma=0.05 * (np.abs(ph) + np.median(np.abs(ph))), spec_d=0.98 * sp,
                 spec_sigma=0.05 * (np.abs(sp) + np.median(np.abs(sp))))
    model = cases.gpu_model_for(ctx, orc, w)
    theta = torch.from_numpy(th32).cuda()
    lnl = model.loglike(theta, "fp32")[0].cpu().numpy()
    phot, spec = (x.cpu().numpy() for x in model.forward(theta, "fp32"))
    ref = orc.eval(th64)
    assert not ref["status"].any()
    for got, want in ((phot, ref["phot"]), (spec, ref["spec"])):   # the FP32 tolerances of the parity tests
        floor = 1e-6 * np.abs(want).max(axis=1, keepdims=True)
        assert np.max(np.abs(got - want) / np.maximum(np.abs(want), floor)) < 2e-5
    assert np.max(np.abs(lnl - ref["lnl"]) / cases.lnl_scale(orc, ref)) < 1e-5
    ctx.close()
