"""A call whose workspace does not fit the context's memory budget is refused, and
the next, smaller call on the stream works: it has the results of a context
without a budget."""
import numpy as np
import pytest

import synth
from tests import cases

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("call", ["loglike", "loglike_grad"])
@pytest.mark.parametrize("first", [0, 200])
def test_smaller_call_after_a_refused_one(call, first):
    """first: rows of a call made before the refused one (0: the refused one is the stream's first)"""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2609_30145_gb300 import Context
    from paper_2609_30145_gb300.api import SedError
    w = synth.WORKLOADS["tiny_phot_16x4x512"]
    orc = cases.oracle_for(w)
    theta = torch.from_numpy(cases.theta_pair(w, 100000, seed=81)[0]).cuda()
    free, tight = Context(0), Context(0, hbm_budget_bytes=64 << 20)
    one, two = (cases.gpu_model_for(c, orc, w) for c in (free, tight))
    ref = [x.cpu().numpy() for x in getattr(one, call)(theta[:300])]
    if first:
        getattr(two, call)(theta[:first])
    held = []
    for _ in range(2):
        with pytest.raises(SedError):
            getattr(two, call)(theta)
        held.append(tight.memory_used())
    assert held[0] == held[1]
    for n in (300, 64, 300):
        got = getattr(two, call)(theta[:n])
        for a, b in zip(got, ref):
            assert np.array_equal(a.cpu().numpy(), b[:n]), n
    free.close()
    tight.close()
