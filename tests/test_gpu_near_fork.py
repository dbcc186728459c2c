"""The generic pair sums on the plan's second stream (marked gpu): grids off the lattice with leaves enough
to fork them (and one just below) give bit for bit what the plan's own stream gives, in both output types,
again after another field, and in a captured batch on two lanes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(28, 24, 20), (44, 40, 36), (60, 52, 48), (72, 60, 52)])
def test_same_bits_as_on_one_stream(kf, monkeypatch, dims):
    import torch
    h = 1.0 / max(dims)
    pts = (np.stack(np.meshgrid(*(np.arange(d) for d in dims[::-1]), indexing="ij"), -1)[..., ::-1].reshape(-1, 3) + 0.5) * h
    dp = torch.as_tensor(np.ascontiguousarray(pts), device="cuda")
    I = [1e20 * torch.rand(pts.shape[0], device="cuda", generator=torch.Generator("cuda").manual_seed(k)) for k in (1, 2)]
    a, b = kf.absorption(150.0)

    def plan(stream=None):
        return kf.Plan(dp, h, 64, 4, a, b, precision="mixed", stream=stream)
    monkeypatch.setenv("KIFMM_NEAR_STREAM", "same")
    p = plan()
    ref = [p.eval(x).clone() for x in I] + [p.eval(I[0].double()).clone()]
    p.close()
    monkeypatch.delenv("KIFMM_NEAR_STREAM")
    p = plan()
    out = [p.eval(x).clone() for x in I] + [p.eval(I[0].double()).clone()]
    p.close()
    for x, y in zip(ref, out):
        assert torch.equal(x, y)
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    plans = [plan(st) for _ in I]
    S = [torch.empty_like(x) for x in I]
    kf.eval_batch(plans, I, S, C=[1.0, 1.0], capture=True, lanes=2)
    torch.cuda.synchronize()
    for x, y in zip(ref, S):
        assert torch.equal(x, y)
    for p in plans:
        p.close()
