"""The tensor-core translation launches' split over the SMs (marked gpu): tiles cut between CTAs,
whole tiles and tiles without a slot, at every coefficient count that a surface order gives.

The mixed form (its M2L, L2L, near field and local expansion go through that launch) against the
FP64 form of the same plan, to the mixed form's target of 1e-6; two evaluations agree bit for bit,
since the pieces of a cut tile are added in slot order."""
import numpy as np
import pytest

from paper_2006_03515_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _check(kf, pts, h, I, leaf, m0, **kw):
    import torch
    a, b = kf.absorption(152.0)
    dp, dI = torch.as_tensor(pts, device="cuda"), torch.as_tensor(I, device="cuda")
    s64 = kf.Plan(dp, h, leaf, m0, a, b, precision="fp64", **kw).eval(dI)
    p = kf.Plan(dp, h, leaf, m0, a, b, precision="mixed", **kw)
    s = [p.eval(dI) for _ in range(2)]
    p.check()
    assert float(torch.linalg.norm(s[0] - s64) / torch.linalg.norm(s64)) <= 1e-6
    assert torch.equal(s[0], s[1])


@pytest.mark.parametrize("n,leaf,m0", [
    (8, 8, 4),      # one level of 64 boxes: one tile, its slots cut over several CTAs
    (16, 8, 3), (16, 8, 5), (16, 8, 7), (16, 8, 8),   # 5 tiles, each R of the surface orders
    (24, 64, 6),    # tiles that hold two octants
    (40, 64, 6),    # partly filled last tiles, leaves of a full lattice
    (64, 64, 6),    # more tiles than a fraction of the SMs, fewer than all
])
def test_uniform(kf, n, leaf, m0):
    pts, h, I = W.config_uniform(n)
    _check(kf, pts, float(h[0]), I, leaf, m0, pad_lattice=n % 8 != 0)


def test_boxes_without_v_lists(kf):
    """Two distant dense clusters: boxes of the deep levels whose neighbourhoods are empty."""
    import torch
    rng = np.random.Generator(np.random.PCG64(7))
    pts = np.concatenate([0.02 * rng.random((3000, 3)), 0.98 + 0.02 * rng.random((500, 3)), rng.random((200, 3))])
    h = torch.full((len(pts),), 1e-3, dtype=torch.float64, device="cuda")
    _check(kf, pts, h, rng.random(len(pts)) + 0.1, 32, 6)


@pytest.mark.parametrize("p", [4, 7, 8])
def test_chebyshev(kf, p):
    pts, h, I = W.config_uniform(32)
    _check(kf, pts, float(h[0]), I, 64, p, repr="cheb")
