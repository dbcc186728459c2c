"""The surrogate's kernels at the edges of their tiles, against the oracle's FP64 forward pass
(marked gpu): odd and even mode counts over every frequency-block width of the folded plane
transforms, 2 modes = n (period n and above), grids whose half is no multiple of the inverse's
point block, planes copied whole and in chunks of columns, odd columns among the chunks.

Bars: forward max |y - y_oracle| <= 1e-4 max |y_oracle| (FP32 sums of at most n = 44 products an
axis against 64 bits, as for the smaller model); loss relative 1e-5; along a random direction of
each parameter block the gradient meets the oracle's central difference to 2e-3 of its norm.
"""
import numpy as np
import pytest

from oracle import sno as O
from paper_2006_03515_gb300 import kifmm

pytestmark = pytest.mark.gpu

SIZES = [   # n, period, width, modes, layers, projection, batch
    (4, 4, 4, 1, 1, 1, 1), (4, 6, 4, 2, 2, 3, 3), (12, 12, 8, 6, 2, 8, 2), (12, 17, 4, 5, 2, 5, 2),
    (20, 30, 4, 7, 2, 16, 1), (24, 24, 8, 8, 1, 8, 1), (28, 42, 4, 9, 1, 7, 1), (40, 60, 12, 3, 2, 16, 2),
    (44, 44, 4, 11, 1, 8, 1), (64, 96, 16, 4, 2, 16, 1),
    (8, 8, 64, 2, 1, 8, 1), (8, 12, 48, 4, 1, 128, 5),   # wide layers, where a block's modes are few
]


def _inputs(C, m, L, P, n, B, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    th = [rng.standard_normal(int(np.prod(s))) * (1.0 / C if name.startswith("R") else 0.5)
          for name, s in O.param_layout(C, m, L, P)]
    u, t = rng.standard_normal((2, B, n, n, n)).astype(np.float32)
    return np.concatenate(th).astype(np.float32), u, t


@pytest.mark.parametrize("n, period, C, m, L, P, B", SIZES)
def test_forward_and_gradient_match_oracle(n, period, C, m, L, P, B):
    import torch
    th, u, t = _inputs(C, m, L, P, n, B, 7 * n + m)
    M = kifmm.SNO(n, C, m, L, P, max_batch=B)
    M.set_bf16(False)
    M.set_period(period)
    M.set_params(th)
    du, dt = (torch.as_tensor(x.reshape(B, -1), device="cuda") for x in (u, t))
    y = M.forward(du).cpu().numpy()
    th64, u64, t64 = th.astype(np.float64), u.astype(np.float64), t.astype(np.float64)
    for b in range(B):
        ref = O.forward(th64, u64[b], C, m, L, P, period).ravel()
        assert np.abs(y[b] - ref).max() <= 1e-4 * np.abs(ref).max()
    loss = M.loss_grad(du, dt)
    g = M.grads().astype(np.float64)
    M.close()
    ref = O.loss(th64, u64, t64, C, m, L, P, period)
    assert abs(loss - ref) <= 1e-5 * ref
    if n > 28:   # (the finite differences of larger grids take minutes; their backward sizes are covered above)
        return
    rng = np.random.Generator(np.random.PCG64(3))
    off, eps = 0, 1e-3
    for name, shp in O.param_layout(C, m, L, P):
        k = int(np.prod(shp))
        d = np.zeros_like(th64)
        d[off:off + k] = rng.standard_normal(k)
        d /= np.linalg.norm(d)
        fd = (O.loss(th64 + eps * d, u64, t64, C, m, L, P, period)
              - O.loss(th64 - eps * d, u64, t64, C, m, L, P, period)) / (2 * eps)
        scale = np.linalg.norm(g[off:off + k]) + 1e-6 * ref
        assert abs(float(g @ d) - fd) <= 2e-3 * scale, (name, float(g @ d), fd, scale)
        off += k


@pytest.mark.parametrize("n, r_in, r_out", [(12, 0.5, 1.0), (12, 1.0, 2.5), (20, 2.0, 5.0), (24, 3.0, 7.0),
                                            (28, 4.0, 8.0), (36, 2.0, 4.0)])
@pytest.mark.parametrize("offset", [0, 1])
def test_near_part_matches_oracle(n, r_in, r_out, offset):
    """The near part alone (all parameters zero) for every kind of halo, grids that are no multiple of
    the kernel's tile, and a field that starts off a 16-byte boundary."""
    import torch
    from oracle import kernel as K
    a, b, h = 5.25, 300.0, 1.0 / n
    M = kifmm.SNO(n, 4, 1, 1, 1, max_batch=2)
    M.set_params(np.zeros(M.num_params(), np.float32))
    M.set_near_field(a, b, h, r_in, r_out)
    u = np.random.Generator(np.random.PCG64(n)).standard_normal((2, n, n, n)).astype(np.float32)
    buf = torch.zeros(u.size + 1, device="cuda")
    du = buf[offset:offset + u.size].copy_(torch.as_tensor(u.ravel())).view(2, -1)
    y = M.forward(du).cpu().numpy()
    M.close()
    sigma = K.self_sigma(h, a, b, "cell_exact")
    for i in range(2):
        ref = O.near_field(u[i].astype(np.float64), a, b, h, sigma, r_in, r_out).ravel()
        assert np.abs(y[i] - ref).max() <= 1e-5 * np.abs(ref).max()
