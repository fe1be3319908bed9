"""The adjoint's filter samples on the forward's axes (test_gpu_sample_brackets):
even in ln(lambda), uneven by up to a factor of seven, and one with two nodes
2e-5 apart, so that brackets come from the index table alone or by a walk; with
redshifts that keep every sample inside the grid and with ones that take some
below it.  Every column of the gradient, d lnL / dz among them, against the
oracle's analytic gradient."""
import numpy as np
import pytest

import synth
from tests import cases
from tests.test_gpu_grad import GRAD_TOL, check_grad, gpu_grad
from tests.test_gpu_sample_brackets import _grid

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


@pytest.mark.parametrize("inside", [True, False])
@pytest.mark.parametrize("kind", ["even", "uneven", "close"])
def test_gradient_on_other_axes(ctx, kind, inside):
    w = synth.WORKLOADS["tiny_phot_16x4x512"]
    filt = synth.make_filters_gauss(7, 0.6, 4.5, 0.2, 200)
    filt = [(x[::s], t[::s]) for (x, t), s in zip(filt, (1, 2, 3, 7, 13, 1, 50))]
    filt.append((np.array([2.0e4, 2.1e4]), np.array([1.0, 1.0])))
    orc = cases.oracle_for(w, grid=_grid(w, kind), filters=synth.pack_filters(filt))
    model = cases.gpu_model_for(ctx, orc, w)
    th32, _ = cases.theta_pair(w, 40, seed=29)
    z = np.linspace(0.5, 3.0, 40) if inside else np.linspace(5.0, 8.0, 40)
    th32[:, model.offsets["zred"]] = z.astype(np.float32)
    lnl, g, st = gpu_grad(model, th32, "fp32")
    ref = orc.grad(th32.astype(np.float64))
    assert np.array_equal(st, ref["status"])
    check_grad(g, ref["grad"], st, GRAD_TOL["tiny"])   # the tolerance of this workload on its own grid
    model.close()
