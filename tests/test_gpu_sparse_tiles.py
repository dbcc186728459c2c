"""Tensor-core translations of trees with fewer V-list slots than tiles (marked gpu): small distant
clusters, whose deep levels have boxes without a V list, so that most tiles of the launch have no slot.

The mixed form against the FP64 form of the same points, to the mixed form's target of 1e-6, after the device
memory that the plan's work space comes from has held NaN."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("clusters,width", [
    (((0.1, 300), (0.9, 100)), 0.01),                 # one tile of 2 slots, six without
    (((0.1, 300), (0.9, 300)), 0.001),                # deeper chains of single boxes
    (((0.05, 100), (0.5, 80), (0.95, 120)), 0.002),
    (((0.1, 70), (0.9, 70)), 1e-4),
])
def test_small_distant_clusters(kf, clusters, width):
    import torch
    rng = np.random.Generator(np.random.PCG64(3))
    pts = np.concatenate([c + width * (rng.random((n, 3)) - 0.5) for c, n in clusters])
    h = torch.full((len(pts),), width / 20, dtype=torch.float64, device="cuda")
    dp = torch.as_tensor(pts, device="cuda")
    I = torch.as_tensor(rng.random(len(pts)) + 0.1, device="cuda")
    a, b = kf.absorption(152.0)
    s64 = kf.Plan(dp, h, 64, 6, a, b, precision="fp64").eval(I)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    dirt = [torch.full((1 << 18,), float("nan"), device="cuda") for _ in range(256)]
    torch.cuda.synchronize()
    del dirt
    torch.cuda.empty_cache()
    p = kf.Plan(dp, h, 64, 6, a, b, precision="mixed")
    assert p.info()["m2l_tensor"]
    s = [p.eval(I) for _ in range(2)]
    p.check()
    assert float(torch.linalg.norm(s[0] - s64) / torch.linalg.norm(s64)) <= 1e-6
    assert torch.equal(s[0], s[1])
