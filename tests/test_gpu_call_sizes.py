"""Calls of different row counts on one stream.  The per-tile node windows that the
contraction reads are left empty by the call before, whatever its number of
128-row tiles: every row of every call must have, bit for bit, the lnL,
photometry and gradient that it has in a context of its own.  Grids of 512
wavelengths (every column of a row of Y is a node) and 1500, with windows that
reach the grid's red end, the redshift sampled (rows ordered by the
preparation kernel) and fixed (rows in the caller's order)."""
import numpy as np
import pytest

import synth
from tests import cases

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES = (64, 300, 1024, 64, 300, 1000, 100, 300, 129, 700, 1, 1024)


@pytest.fixture(scope="module")
def contexts():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_30145_gb300 import build
    build.build()
    from paper_2609_30145_gb300 import Context
    made = [Context(0), Context(0)]
    yield made
    for c in made:
        c.close()


@pytest.mark.parametrize("z_fixed", [False, True])
@pytest.mark.parametrize("n_lam", [512, 1500])
@pytest.mark.parametrize("call", ["fp32", "bf16", "fp8", "forward", "grad"])
def test_sizes_in_turn(contexts, call, n_lam, z_fixed):
    w = synth.shrink(synth.WORKLOADS["phot_107x12x6000_b1024"], n_age=20, n_feh=4, n_lam=n_lam, n_sfh=10)
    orc = cases.oracle_for(w)
    zc, z = cases.z_column(w.n_sfh, w.zmode), 0.05
    th32, _ = cases.theta_pair(w, 1024, seed=61)
    th32[:, zc] = np.random.default_rng(62).uniform(0.01, 0.3, 1024).astype(np.float32)
    fixed = {"zred": z} if z_fixed else None
    theta = torch.from_numpy(np.ascontiguousarray(np.delete(th32, zc, axis=1) if z_fixed else th32)).cuda()

    def result(model, rows):
        if call == "forward":
            return [model.forward(rows, "fp32")[0]]
        if call == "grad":
            return list(model.loglike_grad(rows, "fp32"))
        return list(model.loglike(rows, call))

    one, many = (cases.gpu_model_for(c, orc, w, fixed=fixed) for c in contexts)
    alone = [x.cpu().numpy() for x in result(one, theta)]
    assert np.isfinite(alone[0]).all()
    for i, n in enumerate(SIZES):
        got = result(many, theta[:n])
        for a, b in zip(got, alone):
            assert np.array_equal(a.cpu().numpy(), b[:n]), (i, n)
    one.close()
    many.close()
