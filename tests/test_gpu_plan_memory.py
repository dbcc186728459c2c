"""FP64 plans where device memory runs out (marked gpu): the transforms of the M2L need more of it than the
dense products, so a plan that cannot have them is made with the dense products.

Out-of-memory reports are injected on the host (KIFMM_FAIL_ALLOC=k: the k-th device allocation of a plan)."""
import numpy as np
import pytest

from paper_2006_03515_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_transforms_give_way_to_dense_products(kf, monkeypatch):
    import torch
    pts, h, I = W.config_uniform(16)
    a, b = kf.absorption(152.0)
    dp, dI = torch.as_tensor(pts, device="cuda"), torch.as_tensor(I, device="cuda")

    def run():
        p = kf.Plan(dp, float(h[0]), 8, 6, a, b, precision="fp64")
        s = p.eval(dI).clone()
        n = p.info()["eval_launches"]
        p.close()
        return s, n
    s_fft, n_fft = run()
    monkeypatch.setenv("KIFMM_M2L", "simt")
    s_dense, n_dense = run()
    monkeypatch.delenv("KIFMM_M2L")
    assert n_fft != n_dense
    refused = dense = 0
    for k in range(1, 1000):
        monkeypatch.setenv("KIFMM_FAIL_ALLOC", str(k))
        try:
            s, n = run()
        except kf.KifmmError as e:
            assert e.code == -2, str(e)
            assert dense == 0
            refused += 1
            continue
        if n == n_fft:   # past the plan's last allocation
            assert torch.equal(s, s_fft)
            break
        assert n == n_dense and torch.equal(s, s_dense)
        dense += 1
    assert refused > 0 and dense >= 4
