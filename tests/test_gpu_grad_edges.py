"""Edges of the adjoint's kernels: odd numbers of pixels (two per thread), pixel
ranges in order with linearly interpolated and Gaussian rows side by side, grids
on which many or few filter samples share a bracket (the warps' shuffled sums),
and launches whose dW tiles go to clusters of 8, 4, 2 or 1 CTAs, which must give a
row the same bits."""
import dataclasses

import numpy as np
import pytest

import synth
from tests import cases
from tests.test_gpu_grad import GRAD_TOL, check_grad, gpu_grad

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_30145_gb300 import build
    build.build()
    from paper_2609_30145_gb300 import Context
    c = Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n_pix", [2, 63, 64, 129, 515])
def test_pixel_pairs_in_order(ctx, n_pix):
    """Resolution rising with wavelength from R = 40 to 30000, no stellar
    dispersion: the pixels' ranges stay in order and pass from Gaussian rows to
    linear ones."""
    w = synth.shrink(synth.WORKLOADS["specphot_afe_107x12x5x6000_b2048"], n_age=20, n_feh=4, n_lam=1500,
                     n_sfh=10, n_pix=n_pix, batch=40)
    orc = cases.oracle_for(w, lsf_r=np.geomspace(40.0, 30000.0, n_pix), sigma_gal_kms=0.0)
    model = cases.gpu_model_for(ctx, orc, w)
    th32, th64 = cases.theta_pair(w, w.batch, seed=91)
    lnl, g, st = gpu_grad(model, th32, "fp32")
    ref = orc.grad(th64)
    assert np.array_equal(st, ref["status"])
    kinks = {int(r): model.offsets["zred"] for r in np.nonzero(cases.kink_rows(orc, th64))[0]}
    check_grad(g, ref["grad"], st, GRAD_TOL["mixed_lsf"], skip=kinks)
    model.close()


@pytest.mark.parametrize("n_lam", [150, 700, 6000])
def test_samples_per_bracket(ctx, n_lam):
    """From tens of samples in a bracket to several nodes between samples."""
    w = dataclasses.replace(synth.shrink(synth.WORKLOADS["phot_107x12x6000_b1024"], n_age=20, n_feh=4, n_lam=n_lam,
                                         n_sfh=10), batch=40)
    orc = cases.oracle_for(w)
    model = cases.gpu_model_for(ctx, orc, w)
    th32, th64 = cases.theta_pair(w, w.batch, seed=92)
    lnl, g, st = gpu_grad(model, th32, "fp32")
    ref = orc.grad(th64)
    assert np.array_equal(st, ref["status"])
    check_grad(g, ref["grad"], st, GRAD_TOL["phot"])
    model.close()


@pytest.mark.parametrize("name", ["phot_107x12x6000_b1024", "specphot_afe_107x12x5x6000_b2048"])
def test_a_row_keeps_its_bits_whatever_the_cluster(ctx, name):
    w = synth.shrink(synth.WORKLOADS[name], n_age=40, n_lam=3000, n_sfh=12)
    orc = cases.oracle_for(w)
    model = cases.gpu_model_for(ctx, orc, w)
    theta = torch.from_numpy(cases.theta_pair(w, 3000, seed=93)[0]).cuda()

    def grad(rows):
        lnl, g, st = model.loglike_grad(theta[rows].contiguous(), "fp32")
        return torch.cat([lnl[:, None], g.double()], 1).cpu().numpy()

    alone = np.concatenate([grad(slice(i, i + 1)) for i in (0, 31, 63)])
    for n in (64, 65, 300, 700, 1500, 3000):
        assert np.array_equal(grad(slice(0, n))[[0, 31, 63]], alone), n
    model.close()
