"""M2L of the FP64 form by Fourier transforms (marked gpu): against the dense products in the rank
basis (KIFMM_M2L=simt) for every surface order that takes the transforms and one beyond, on a uniform
grid, on a cloud with W and X lists, and with a comparison kernel.

Bar: the densities cancel by up to 1e3 before they reach the check surface, and a value passes about
sixty additions and products of rounding 1.1e-16, with random signs: 1e3 x 1.1e-16 x sqrt(60) = 9e-13;
5e-12 allows for the levels' sum."""
import numpy as np
import pytest

from paper_2006_03515_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _pair(kf, monkeypatch, pts, h, I, leaf, m0, **kw):
    import torch
    a, b = kf.absorption(152.0)
    dp, dI = torch.as_tensor(pts, device="cuda"), torch.as_tensor(I, device="cuda")
    s = kf.Plan(dp, h, leaf, m0, a, b, precision="fp64", **kw).eval(dI)
    monkeypatch.setenv("KIFMM_M2L", "simt")
    ref = kf.Plan(dp, h, leaf, m0, a, b, precision="fp64", **kw).eval(dI)
    assert float(torch.linalg.norm(s - ref) / torch.linalg.norm(ref)) <= 5e-12


@pytest.mark.parametrize("m0", [3, 4, 5, 6, 7, 8, 9])
def test_uniform(kf, monkeypatch, m0):
    pts, h, I = W.config_uniform(16)
    _pair(kf, monkeypatch, pts, float(h[0]), I, 8, m0)


@pytest.mark.parametrize("kernel", ["zheleznyak", "helmholtz3"])
def test_cloud_with_w_and_x_lists(kf, monkeypatch, kernel):
    import torch
    rng = np.random.Generator(np.random.PCG64(11))
    pts = np.concatenate([0.1 * rng.random((4000, 3)) + 0.3, rng.random((3000, 3))])
    h = torch.full((len(pts),), 0.01, dtype=torch.float64, device="cuda")
    _pair(kf, monkeypatch, pts, h, rng.random(len(pts)) + 0.1, 16, 6, kernel=kernel)
