"""Non-finite values in the streamer's source (marked gpu): a NaN density, an infinite one and a NaN electrode
potential reach S_i = mu_e n_e alpha |E|, and so S_ph, where |E| is zero as where it is not."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NX, NY, NZ, H = 8, 8, 16, 0.02


@pytest.mark.parametrize("what", ["nan", "inf", "phi0", "none"])
def test_source_keeps_nonfinite_values(kf, what):
    import torch
    g = [(np.arange(m) + 0.5) * H for m in (NZ, NY, NX)]
    pts = np.stack(np.meshgrid(*g, indexing="ij"), -1)[..., ::-1].reshape(-1, 3)
    a, b = kf.absorption(150.0)
    # one leaf: S_ph at every cell sums every other cell's S_i
    pl = kf.Plan(torch.as_tensor(np.ascontiguousarray(pts), device="cuda"), H, len(pts), 4, a, b, precision="fp64")
    s = kf.Streamer(NX, NY, NZ, H, plan=pl, **(dict(phi0=float("nan")) if what == "phi0" else {}))
    ne = torch.full((NZ, NY, NX), 1e10, dtype=torch.float64, device="cuda")
    npi = ne.clone()
    if what in ("nan", "inf"):
        ne[3, 4, 5] = float(what)   # the potential is still 0 here: a NaN or infinite charge stops the solve at once
    s.set(ne, npi)
    s.rhs()
    sph = s.get()[3]
    if what == "none":
        assert bool(torch.isfinite(sph).all())
    else:
        assert not bool(torch.isfinite(sph).any())
    s.close()
