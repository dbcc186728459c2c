"""The Poisson solve over grid sizes that put the levels of the one-block V-cycle differently (marked gpu):
the whole hierarchy in it, one level above it, several, a coarsest level of a warp, of a block and of more
cells than threads. Against the oracle's direct solve with the bar of the solver's own test (1e-9 of phi at
a relative residual of 1e-12)."""
import numpy as np
import pytest

from oracle import streamer as SD

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz", [(16, 16, 32), (16, 16, 34), (32, 32, 32), (12, 20, 28), (18, 18, 18), (15, 15, 15),
                                      (4, 4, 4), (3, 5, 7), (40, 24, 56)])
def test_poisson(kf, nx, ny, nz):
    import torch
    h = 0.02
    rho = np.random.default_rng(nx).standard_normal((nz, ny, nx)) * 1e8
    s = kf.Streamer(nx, ny, nz, h, mg_tol=1e-12)
    phi, res, cyc = s.poisson(torch.as_tensor(rho, device="cuda"))
    want = SD.solve_poisson(rho, h, 52e3)
    assert res <= 1e-12 and cyc <= 60
    assert np.linalg.norm(phi.cpu().numpy() - want) <= 1e-9 * np.linalg.norm(want)
