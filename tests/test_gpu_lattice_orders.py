"""The leaves' sliced upward operator on a lattice at surface orders whose own operator does not fit the
slice kernel (marked gpu): the mixed form's upward coefficients against the FP64 form's to 1e-8 of each
box's largest (their common bar), and the field to the mixed form's 1e-6."""
import numpy as np
import pytest

from paper_2006_03515_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m0,p_o2", [(40, 8, 152.0), (48, 8, 1.52), (44, 7, 15.2)])
def test_leaf_coefficients(kf, monkeypatch, n, m0, p_o2):
    import torch
    monkeypatch.setenv("KIFMM_OZ_MIN", "0")   # (small grids take the slices too)
    pts, h, I = W.config_uniform(n)
    a, b = kf.absorption(p_o2)
    dp, dI = torch.as_tensor(pts, device="cuda"), torch.as_tensor(I, device="cuda")
    out = []
    for prec in ("fp64", "mixed"):
        p = kf.Plan(dp, float(h[0]), 64, m0, a, b, precision=prec, pad_lattice=True)
        s = p.eval(dI)
        p.check()
        t = p.tree()
        out.append((s, p.upward()[t["leaf"] == 1], p.info()))
    assert out[1][2]["lattice_far"] and out[1][2]["upward_tensor_levels"] >= 1
    assert float(torch.linalg.norm(out[1][0] - out[0][0]) / torch.linalg.norm(out[0][0])) <= 1e-6
    c64, c = out[0][1], out[1][1]
    r = min(c64.shape[1], c.shape[1])
    scale = np.abs(c64).max(axis=1)
    on = scale > 0
    assert np.all(np.abs(c[on, :r] - c64[on, :r]).max(axis=1) <= 1e-8 * scale[on])
