"""The forward epilogue's two ways to a filter sample's bracket against the FP64
oracle: without a walk where the index table's cells are wide against the
place's rounding and every sample lies inside the grid, by a walk elsewhere.
Axes: even in ln(lambda), uneven by up to a factor of seven, and one with two
nodes 2e-5 apart (its cells are too fine for the first way); with redshifts
that keep every sample inside the grid and with ones that take some below it.
Bands of 2 to 200 samples, among them lengths that are no multiple of a warp."""
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


def _grid(w, kind):
    g = synth.make_grid(**dict(w.grid_kw, n_lam=1400), seed=1)
    n = g.lam_aa.size
    if kind == "even":
        keep = np.arange(0, n, 2)
    else:   # runs of every node, every third and every seventh
        keep = np.concatenate([np.arange(0, 300), np.arange(300, 900, 3), np.arange(900, n, 7)])
    g.lam_aa, g.flux = g.lam_aa[keep], np.ascontiguousarray(g.flux[..., keep])
    if kind == "close":
        k = keep.size // 2
        g.lam_aa = np.insert(g.lam_aa, k + 1, g.lam_aa[k] * (1 + 2e-5))
        g.flux = np.insert(g.flux, k + 1, g.flux[..., k], axis=-1)
    return g


@pytest.mark.parametrize("rows", [40, 700])
@pytest.mark.parametrize("inside", [True, False])
@pytest.mark.parametrize("kind", ["even", "uneven", "close"])
def test_photometry_on_other_axes(ctx, kind, inside, rows):
    w = synth.WORKLOADS["tiny_phot_16x4x512"]
    filt = synth.make_filters_gauss(7, 0.6, 4.5, 0.2, 200)
    filt = [(x[::s], t[::s]) for (x, t), s in zip(filt, (1, 2, 3, 7, 13, 1, 50))]
    filt.append((np.array([2.0e4, 2.1e4]), np.array([1.0, 1.0])))
    orc = cases.oracle_for(w, grid=_grid(w, kind), filters=synth.pack_filters(filt))
    model = cases.gpu_model_for(ctx, orc, w)
    th32, th64 = cases.theta_pair(w, rows, seed=23)
    zc = model.offsets["zred"]
    # the grid starts at 0.1 um and the bands at 0.45 um: below z = 3.4 every sample lies inside
    z = np.linspace(0.5, 3.0, rows) if inside else np.linspace(5.0, 8.0, rows)
    th32[:, zc] = z.astype(np.float32)
    th64 = th32.astype(np.float64)
    phot, _ = model.forward(torch.from_numpy(th32).cuda(), "fp32")
    torch.cuda.synchronize()
    sel = np.unique(np.linspace(0, rows - 1, 40).astype(int))
    ref = orc.eval(th64[sel])["phot"]
    floor = 1e-6 * np.abs(ref).max(axis=1, keepdims=True)
    err = cases.rel_err(phot.cpu().numpy()[sel], ref, floor)
    assert err.max() < 2e-5, (kind, inside, rows, float(err.max()))   # the FP32 flux tolerance of the parity tests
    model.close()
