"""K-tile-masked calls (one [Fe/H] per row, FP32) whose windows and masks start
empty because the call before emptied them: a sequence of calls of different
sizes, with the redshift sampled or fixed, self-ordered (up to 128 rows) or not,
with gradients and an unmasked model in between, must give each row the lnL it
has alone, bit for bit, and the oracle's on sampled rows."""
import dataclasses

import numpy as np
import pytest

import synth
from tests import cases

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


@pytest.mark.parametrize("z_fixed", [False, True])
def test_masks_and_windows_start_empty(ctx, z_fixed):
    w = dataclasses.replace(synth.shrink(synth.WORKLOADS["specphot_afe_107x12x5x6000_b2048"], n_age=40, n_lam=1500,
                                         n_sfh=12, n_pix=200))
    orc = cases.oracle_for(w)
    z = 2.0
    model = cases.gpu_model_for(ctx, orc, w, fixed={"zred": z} if z_fixed else None)
    other = cases.gpu_model_for(ctx, orc, dataclasses.replace(w, zmode=0))   # a [Fe/H] per bin: no masks
    th32, _ = cases.theta_pair(w, 700, seed=3)
    zc = cases.z_column(w.n_sfh, w.zmode)
    if z_fixed:
        th32[:, zc] = z
    full = th32.astype(np.float64)
    mine = np.delete(th32, zc, axis=1) if z_fixed else th32
    theta = torch.from_numpy(np.ascontiguousarray(mine)).cuda()
    oth = torch.from_numpy(cases.theta_pair(dataclasses.replace(w, zmode=0), 90, seed=5)[0]).cuda()

    def lnl(rows):
        return model.loglike(theta[rows].contiguous(), "fp32")[0].cpu().numpy()

    def lnl_and_grad(rows):   # the adjoint sums its lnL in its own order
        l, g, _ = model.loglike_grad(theta[rows].contiguous(), "fp32")
        return np.column_stack([l.cpu().numpy(), g.cpu().numpy()])

    alone = np.concatenate([lnl(slice(i, i + 1)) for i in range(0, 700, 50)])
    alone_g = np.concatenate([lnl_and_grad(slice(i, i + 1)) for i in range(0, 700, 50)])
    for n in (700, 64, 128, 129, 1, 700, 300):
        got = lnl(slice(0, n))
        k = (n + 49) // 50
        assert np.array_equal(got[::50], alone[:k]), n
        if n in (128, 129):
            assert np.array_equal(lnl_and_grad(slice(0, n))[::50], alone_g[:k]), n
        other.loglike(oth, "fp32")
        lnl(slice(400, 460))
    ref = orc.eval(full[::50])
    scale = cases.lnl_scale(orc, ref)
    ok = ref["status"] == 0
    assert np.max(np.abs(alone - ref["lnl"])[ok] / scale[ok]) < 1e-5   # the FP32 lnL tolerance of the parity tests
    model.close()
    other.close()
