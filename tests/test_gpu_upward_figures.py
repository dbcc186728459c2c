"""The plan's figures of the upward pass (marked gpu): a plan whose exact slices run on the tensor cores at any
level reports the flop that they execute there, also where only the lattice's leaves take them."""
import pytest

from paper_2006_03515_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m0,levels", [(6, 2), (8, 1)])
def test_tensor_levels_have_flops(kf, monkeypatch, m0, levels):
    import torch
    monkeypatch.setenv("KIFMM_OZ_MIN", "0")
    pts, h, _ = W.config_uniform(32)
    a, b = kf.absorption(152.0)
    p = kf.Plan(torch.as_tensor(pts, device="cuda"), float(h[0]), 64, m0, a, b, precision="mixed")
    i = p.info()
    assert i["upward_tensor_levels"] == levels
    # 512 leaves of 64 points: a product of two FP16 slices is 2 rank 64 flop a leaf
    assert i["upward_mma_flops"] >= 2 * i["pinv_rank_min"] * 64 * 512
    monkeypatch.setenv("KIFMM_UPWARD", "fp64")
    p = kf.Plan(torch.as_tensor(pts, device="cuda"), float(h[0]), 64, m0, a, b, precision="mixed")
    assert p.info()["upward_tensor_levels"] == 0 and p.info()["upward_mma_flops"] == 0
