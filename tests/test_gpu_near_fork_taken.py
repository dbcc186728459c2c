"""Which plans off the lattice run their pair sums on the second stream (marked gpu): those of 1024 leaves or more,
seen by the eighth phase time that a forked plan reports, with the same bits as on one stream on both sides of
the line."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,forked", [(28700, False), (28850, True), (40000, True)])   # 1009, 1044, 3900 leaves
def test_fork_from_1024_leaves(kf, monkeypatch, n, forked):
    import torch
    pts = torch.as_tensor(np.random.default_rng(17).random((n, 3)), device="cuda")
    I = torch.rand(n, device="cuda", dtype=torch.float64, generator=torch.Generator("cuda").manual_seed(1))
    a, b = kf.absorption(150.0)
    monkeypatch.setenv("KIFMM_TIMING", "1")
    out = []
    for mode in (None, "same"):
        if mode:
            monkeypatch.setenv("KIFMM_NEAR_STREAM", mode)
        p = kf.Plan(pts, 0.01, 64, 4, a, b, precision="mixed")
        assert (p.info()["n_leaves"] >= 1024) == forked and not p.info()["near_tensor"]
        out.append(p.eval(I).clone())
        p.check()
        assert len(p.phase_times()) == (8 if forked and mode is None else 7)
        p.close()
    assert torch.equal(*out)
