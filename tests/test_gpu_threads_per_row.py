"""The forward epilogue's instances of 128, 256 and 512 threads per row, chosen by
the launch's rows: a row's photometry, spectrum, lnL and status are the same bit
for bit whichever instance computed them, so a batch large enough for the
narrow instance is compared with its own leading rows evaluated in smaller
calls, at the sizes on both sides of each instance's limit."""
import pytest

import synth
from tests import cases

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SPEC = "specphot_afe_107x12x5x6000_b2048"


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


def _small(name, n_pix=None):
    return synth.shrink(synth.WORKLOADS[name], n_age=24, n_feh=4, n_lam=900, n_sfh=9, n_pix=n_pix)


def _case(kind):
    """(workload, oracle with data, rows -> FP32 parameter rows)"""
    if kind == "lines":
        w = _small("specphot_lines_107x12x6000_b1024", 333)
        orc = cases.lines_case(w)
        return w, orc, lambda n: cases.lines_theta_pair(w, orc, n, seed=11)[0]
    w = {"tiny": synth.WORKLOADS["tiny_phot_16x4x512"], "phot": _small("phot_107x12x6000_b1024"),
         "calib": _small(SPEC, 257), "sgal": _small("specphot_afe_sgal_107x12x5x6000_b2048", 130),
         "floor": _small("specphot_afe_floor_107x12x5x6000_b2048", 100),
         "dense": _small(SPEC, 2001)}[kind]   # more pixels than twice the row's nodes
    orc = cases.calib_case(w, [0.2] + [0.1] * 12) if kind == "calib" else cases.oracle_for(w)
    return w, orc, lambda n: cases.theta_pair(w, n, seed=11, orc=orc)[0]


@pytest.mark.parametrize("kind", ["tiny", "phot", "calib", "sgal", "floor", "lines", "dense"])
def test_rows_do_not_depend_on_the_threads_per_row(ctx, kind):
    w, orc, rows = _case(kind)
    model = cases.gpu_model_for(ctx, orc, w)
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    theta = torch.from_numpy(rows(4 * sm + 60)).cuda()

    def call(n):
        lnl, st = model.loglike(theta[:n], "fp32")
        phot, spec = model.forward(theta[:n], "fp32")
        return [x for x in (lnl, st, phot, spec) if x is not None]

    whole = call(theta.shape[0])
    assert bool((whole[1] == 0).any())
    for n in (1, 37, 2 * sm, 2 * sm + 1, 4 * sm, 4 * sm + 1):
        for a, b in zip(call(n), whole):
            assert torch.equal(a.view(torch.uint8), b[:n].contiguous().view(torch.uint8)), (kind, n)
    model.close()
