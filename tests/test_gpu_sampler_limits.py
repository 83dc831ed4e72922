"""The plain sampler at the limits of its configuration against the oracle's linear merge: guided
samples that all coincide, that lie beyond every stratum, and that are NaN (an infinite interval)."""
import numpy as np
import pytest

from gpu_common import Problem
from helpers import CUBE

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("guide_half", [0.0, 1e-30, 1e30, 2.5e38, float("inf")])
@pytest.mark.parametrize("n_strat,n_guided", [(48, 16), (1, 40), (33, 1)])
def test_merge_is_the_oracles(guide_half, n_strat, n_guided):
    w = CUBE.with_(name="limits", rays=200, n_strat=n_strat, n_guided=n_guided, n_smooth=0, guide_half=guide_half)
    p = Problem(w)
    b = p.gpu_sample(3, 5)
    bt, _ = p.oracle_sample(3, 5)
    t = b.t.cpu().numpy()
    np.testing.assert_array_equal(np.isnan(t), np.isnan(bt["t"]))
    num = ~np.isnan(t)
    assert np.array_equal(t[num].view(np.uint32), bt["t"][num].view(np.uint32))
    assert np.array_equal(b.cls.cpu().numpy(), bt["cls"])
    assert list(b.counts.cpu().numpy()[:3]) == list(bt["counts"][:3])
