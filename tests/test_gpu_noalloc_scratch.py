"""The scratch that a row takes in sed_loglike_noalloc, which sets the largest
accepted batch: its place in the order, its scalars (248 bytes), its weights and
its two rows of nodes.  Refused calls state what they would need and launch
nothing."""
import re

import pytest

import synth
from tests import cases

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROW_SCALARS = 248
SCRATCH = 32 * 1024 * 1024


def test_largest_batch():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_30145_gb300 import Context
    from paper_2609_30145_gb300.api import SedError
    w = synth.WORKLOADS["tiny_phot_16x4x512"]
    orc = cases.oracle_for(w)
    ctx = Context(0)
    model = cases.gpu_model_for(ctx, orc, w)
    n = 128 * 256   # every part is a whole number of 256-byte units
    theta = torch.from_numpy(cases.theta_pair(w, n, seed=95)[0]).cuda()
    need = {}
    for prec in ("fp32", "fp32_simt"):
        with pytest.raises(SedError) as e:
            model.loglike_noalloc(theta, prec)
        need[prec] = int(re.search(r"need (\d+) bytes", str(e.value)).group(1))
    weights = need["fp32"] - need["fp32_simt"]   # two parts of the weights against one
    windows = 2 * 4 * n // 128
    assert need["fp32_simt"] == 256 + windows + weights + n * (4 + ROW_SCALARS + 2 * 4 * 512)
    per_row = need["fp32"] / n
    lnl = model.loglike(theta[:8000], "fp32")[0]
    most = int((SCRATCH - 256 * 12) / per_row)
    assert torch.equal(model.loglike_noalloc(theta[:most], "fp32")[0], lnl[:most])
    ctx.close()
