"""kifmm_direct_noalloc over its range of sizes and pressures (marked gpu): fewer points than a warp's
lanes, groups of targets that are not full, shares of sources that are empty, and both cluster
sizes, against the oracle's direct sum in FP64. Its terms carry a few roundings each (the bar is 2e-14,
some ninety units of FP64 rounding, on the relative 2-norm); the result may take the source's place."""
import numpy as np
import pytest

from oracle import direct as D
from paper_2006_03515_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p_o2,mode", [
    (1, 152.0, "cell_exact"), (2, 152.0, "paper_gl2"), (31, 1.52, "cell_exact"), (33, 152.0, "cell_exact"),
    (257, 15.2, "cell_exact"), (1000, 1.52, "paper_gl2"), (4097, 152.0, "cell_exact"),
    (9000, 1.52, "cell_exact"),
])
def test_direct_matches_oracle(kf, n, p_o2, mode):
    import torch
    side = int(np.ceil(n ** (1 / 3)))
    pts, h = W.uniform_grid(side, 0.7)
    pts = np.ascontiguousarray(pts[:n])
    I = np.random.default_rng(n).random(n) * 1e22
    a, b = kf.absorption(p_o2)
    ref = D.direct_sum(pts, np.full(n, h), I, a, b, 1.0, mode=mode)
    dp, dI = torch.as_tensor(pts, device="cuda"), torch.as_tensor(I, device="cuda")
    got = kf.direct_noalloc(dp, h, dI, a, b, self_mode=mode).cpu().numpy()
    assert np.linalg.norm(got - ref) <= 2e-14 * np.linalg.norm(ref)
    assert np.array_equal(kf.direct_noalloc(dp, h, dI, a, b, S=dI, self_mode=mode).cpu().numpy(), got)


def test_one_block_per_target_group(kf):
    """Above 1216 groups of targets a group takes one block: against a plan of one leaf."""
    import torch
    pts, h = W.uniform_grid(34, 1.0)   # 39304 points, 1229 groups
    I = torch.as_tensor(np.random.default_rng(1).random(len(pts)), device="cuda")
    a, b = kf.absorption(152.0)
    dp = torch.as_tensor(pts, device="cuda")
    got = kf.direct_noalloc(dp, h, I, a, b)
    few = kf.direct_noalloc(dp[:4096].contiguous(), h, I[:4096].contiguous(), a, b)
    rest = kf.direct_noalloc(dp, h, torch.cat([torch.zeros_like(I[:4096]), I[4096:]]), a, b)
    assert float(torch.linalg.norm(got[:4096] - few - rest[:4096]) / torch.linalg.norm(got[:4096])) <= 2e-14
