"""Sources beyond the range of a squared distance in FP64 (marked gpu): the kernel is 0 there, so points that a
caller has put at infinity, or 1e160 away, add nothing to the others' sums."""
import numpy as np
import pytest

from paper_2006_03515_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("far", [1e100, 1e160, float("inf")])
def test_distant_sources_add_nothing(kf, far):
    import torch
    pts, h = W.uniform_grid(8, 0.4)
    n = len(pts)
    I = np.random.default_rng(5).random(n)
    a, b = kf.absorption(152.0)
    all_pts = np.concatenate([pts, [[far, 0.0, 0.0], [0.0, -far, 0.0]]])
    dp, dI = torch.as_tensor(all_pts, device="cuda"), torch.as_tensor(np.concatenate([I, [1.0, 0.0]]), device="cuda")
    got = kf.direct_noalloc(dp, h, dI, a, b)[:n]
    zero = dI.clone()
    zero[n:] = 0.0
    near = all_pts.copy()
    near[n:] = [[9.0, 0.0, 0.0], [0.0, 9.0, 0.0]]
    want = kf.direct_noalloc(torch.as_tensor(near, device="cuda"), h, zero, a, b)[:n]
    assert torch.equal(got, want)
