"""What a workspace's buffers start from is set in the order of the call's own
stream: calls on a stream that does not wait for the default one, each larger
than the one before (so that the workspace is made anew), while the default
stream is busy for 0 to about 100 us.  Rows with K-tile masks and rows without
must have the lnL that they have on the default stream, bit for bit."""
import numpy as np
import pytest

import synth
from tests import cases

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


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


@pytest.mark.parametrize("name", ["specphot_afe_107x12x5x6000_b2048", "phot_107x12x6000_b1024"])
def test_first_call_of_a_size_beside_a_busy_default_stream(contexts, name):
    w = synth.shrink(synth.WORKLOADS[name], n_age=30, n_feh=6, n_lam=1024, n_sfh=10, n_pix=150)
    orc = cases.oracle_for(w)
    one, many = (cases.gpu_model_for(c, orc, w) for c in contexts)
    theta = torch.from_numpy(cases.theta_pair(w, 700, seed=71)[0]).cuda()
    alone = one.loglike(theta, "fp32")[0].cpu().numpy()
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    for i in range(50):
        n = 20 + 13 * i
        rows = theta[:n].clone()
        torch.cuda.synchronize()
        torch.cuda._sleep(4000 * i)
        with torch.cuda.stream(stream):
            lnl = many.loglike(rows, "fp32")[0]
        torch.cuda.synchronize()
        assert np.array_equal(lnl.cpu().numpy(), alone[:n]), (i, n)
    one.close()
    many.close()
