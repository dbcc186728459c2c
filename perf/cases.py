"""The work a user of this framework has it do, as cases that can be timed and checked.

Each case is one call (or the few calls that belong together) through the Python binding:
`Plan.eval` on uniform, padded, adaptive and small grids in the mixed, FP64 and Chebyshev
forms, a captured `eval_batch`, the surrogate's forward pass and training step, a step of
the streamer loop, and the direct sum without allocation. Sizes are those of the
repository's benchmark, tests and workloads (32^3 to 128^3 cells, the two-level grid of
3.2 million cells, the surrogate's 64^3 grid at width 32 and 12 modes, the 128 x 128 x 256
gap of the streamer loop).

`exact` restates every result in 64 bits with plain torch: the discrete sum by FFT or pair
by pair, the network by explicit transforms, the streamer step with the Poisson equation
solved by its discrete eigenvectors.
"""
import math
import random

import numpy as np
import torch

from paper_2006_03515_gb300 import kifmm
from paper_2006_03515_gb300 import workloads as W

CHI_MIN, CHI_MAX = 0.035, 2.0   # 1/(cm Torr), Sec. 2.1 of arXiv:2006.03515
DEV = "cuda"


# ---- the cases ---------------------------------------------------------------------------

def _fmm(name, nx, ny, nz, m0=6, p=760.0, p_o2=152.0, precision="mixed", repr="surface", pad=False):
    c = dict(kind="fmm", grid="box", nx=nx, ny=ny, nz=nz, m0=m0, p=p, p_o2=p_o2, precision=precision, repr=repr,
             pad=pad)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # one evaluation inside a time loop on a coarse grid: launches and latency
        _fmm("uniform_32", 32, 32, 32),
        # the surrogate's label grid (the call of its data generation and of its fallback)
        _fmm("uniform_64", 64, 64, 64, p_o2=150.0),
        # the headline workload of the benchmark
        _fmm("uniform_128", 128, 128, 128),
        # an uneven grid of the batched workload's sizes on its own: padding, low pressure, a higher order
        _fmm("padded_101_m8", 101, 101, 101, m0=8, p=76.0, p_o2=15.2, pad=True),
        # the two-level refined grid around a streamer head (generic pair kernel, W and X lists)
        dict(name="adaptive_3m", kind="fmm", grid="refined", base_n=128, half=6, m0=6, p=760.0, p_o2=150.0,
             precision="mixed", repr="surface", pad=False),
        # the FP64 form, the one users hold the others against
        _fmm("fp64_48", 48, 48, 48, precision="fp64"),
        # the Chebyshev option at the order that reaches the direct sum to 1e-7
        _fmm("cheb_64_p8", 64, 64, 64, m0=8, repr="cheb"),
        # several streamer fields of uneven sizes as one captured batch on four lanes
        dict(name="batch_8_fields", kind="batch", count=8, n_min=40, n_max=80, m0=6, lanes=4),
        # surrogate inference on a batch of fields, at the sizes of its benchmark
        dict(name="sno_forward_32", kind="sno_forward", n=64, width=32, modes=12, layers=4, proj=64, batch=32),
        # one training step of a smaller surrogate (gradient on the host, as a logging user reads it)
        dict(name="sno_train_4", kind="sno_train", n=64, width=16, modes=8, layers=4, proj=64, batch=4),
        # one Heun step of the streamer loop with S_ph from a padded plan, at the benchmark's grid
        dict(name="streamer_128", kind="streamer", nx=128, ny=128, nz=256, photo=True),
        # the direct sum of a caller that cannot allocate (a captured stream, a real-time loop)
        dict(name="direct_4096", kind="direct", n=4096),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["box", "box", "box", "box", "refined", "fp64", "cheb", "batch", "sno_forward", "sno_train",
                       "streamer", "direct"])
    p, p_o2 = rng.choice([(760.0, 150.0), (760.0, 152.0), (76.0, 15.2), (7.6, 1.52)])
    if kind == "box":
        n = [_log(rng, 24, 128) for _ in range(3)]
        if rng.random() < 0.5:
            n = [n[0]] * 3
        if rng.random() < 0.4:
            n = [8 * ((x + 7) // 8) for x in n]   # (whole leaves without padding when cubic)
        return _fmm(None, *n, m0=rng.choice([4, 6, 6, 6, 8]), p=p, p_o2=p_o2, pad=rng.random() < 0.6)
    if kind == "refined":
        return dict(kind="fmm", grid="refined", base_n=_log(rng, 24, 128), half=rng.randint(1, 6),
                    m0=rng.choice([4, 6, 6]), p=p, p_o2=p_o2, precision="mixed", repr="surface", pad=False)
    if kind == "fp64":
        return _fmm(None, *[_log(rng, 16, 48) for _ in range(3)], m0=rng.choice([4, 6]), p=p, p_o2=p_o2,
                    precision="fp64")
    if kind == "cheb":
        n = _log(rng, 24, 64)
        return _fmm(None, n, n, n, m0=rng.randint(4, 8), p=p, p_o2=p_o2, repr="cheb")
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(2, 8), n_min=24, n_max=rng.randint(40, 80),
                    m0=rng.choice([4, 6, 6]), lanes=rng.choice([1, 2, 4, 8]))
    if kind == "sno_forward":
        n = 4 * rng.randint(6, 16)
        return dict(kind="sno_forward", n=n, width=rng.choice([8, 16, 32, 32]), modes=rng.randint(4, 12),
                    layers=rng.randint(2, 4), proj=rng.choice([16, 32, 64]), batch=_log(rng, 1, 32))
    if kind == "sno_train":
        n = 4 * rng.randint(6, 16)
        return dict(kind="sno_train", n=n, width=rng.choice([8, 16, 16]), modes=rng.randint(4, 8),
                    layers=rng.randint(2, 4), proj=rng.choice([16, 32, 64]), batch=rng.randint(1, 4))
    if kind == "streamer":
        nx, ny = (16 * rng.randint(2, 8) for _ in range(2))
        return dict(kind="streamer", nx=nx, ny=ny, nz=16 * rng.randint(2, 16), photo=rng.random() < 0.7)
    return dict(kind="direct", n=_log(rng, 256, 8192))


# ---- inputs ------------------------------------------------------------------------------

def _axes(nx, ny, nz, h):
    return [(torch.arange(n, dtype=torch.float64, device=DEV) + 0.5) * h for n in (nx, ny, nz)]


def _box_points(nx, ny, nz, h):
    """Cell centres, x fastest."""
    x, y, z = _axes(nx, ny, nz, h)
    zz, yy, xx = torch.meshgrid(z, y, x, indexing="ij")
    return torch.stack([xx.reshape(-1), yy.reshape(-1), zz.reshape(-1)], dim=1)


def _blobs(pts, seed, size):
    """1 to 5 Gaussian blobs, widths log-uniform in [0.02, 0.2], amplitudes in [1e20, 1e23], centres in
    [0.1, 0.9] of the box (the surrogate's field distribution)."""
    r = random.Random(seed)
    out = torch.zeros(pts.shape[0], dtype=torch.float64, device=pts.device)
    for _ in range(r.randint(1, 5)):
        c = torch.tensor([s * r.uniform(0.1, 0.9) for s in size], dtype=torch.float64, device=pts.device)
        w = min(size) * math.exp(r.uniform(math.log(0.02), math.log(0.2)))
        out += 10.0 ** r.uniform(20.0, 23.0) * torch.exp(-((pts - c) ** 2).sum(1) / w ** 2)
    return out


def _fmm_geometry(case):
    """Points, cell edge (a number, or one per point) and the source's box."""
    if case["grid"] == "refined":
        pts, h = W.refined_grid(2.0, case["base_n"], 8, (1.0, 1.0, 1.5), case["half"])
        return torch.as_tensor(pts, device=DEV), torch.as_tensor(h, device=DEV)
    h = 1.0 / max(case["nx"], case["ny"], case["nz"])
    return _box_points(case["nx"], case["ny"], case["nz"], h), h


def _fmm_source(case, pts, seed):
    if case["grid"] == "refined":   # a channel and its head along z, log-normal noise
        g = torch.Generator(device=DEV).manual_seed(seed)
        r2 = (pts[:, 0] - 1.0) ** 2 + (pts[:, 1] - 1.0) ** 2
        on = (pts[:, 2] >= 0.5) & (pts[:, 2] <= 1.5)
        s = torch.where(on, 1e21 * torch.exp(-r2 / 0.05 ** 2), torch.zeros_like(r2))
        s = s + 1e23 * torch.exp(-(r2 + (pts[:, 2] - 1.5) ** 2) / 0.02 ** 2)
        s = s * torch.exp(0.3 * torch.randn(s.shape[0], dtype=torch.float64, device=DEV, generator=g))
    else:
        h = 1.0 / max(case["nx"], case["ny"], case["nz"])
        s = _blobs(pts, seed, [case[k] * h for k in ("nx", "ny", "nz")])
    # the mixed form takes and returns FP32 fields, the FP64 form FP64 fields
    return s if case["precision"] == "fp64" else s.float()


def _batch_fields(case):
    """(n, p, p_o2) of each field: sizes log-uniform in points, pressure 760 or 76 Torr."""
    r = random.Random(case["count"] * 1000 + case["n_max"])
    out = []
    for _ in range(case["count"]):
        n = _log(r, case["n_min"], case["n_max"])
        p = r.choice([760.0, 76.0])
        out.append((n, p, 0.2 * p))
    return out


def _sno_layout(case):
    C, m, P = case["width"], case["modes"], case["proj"]
    K = (2 * m) * (2 * m) * m
    lay = [("Wl", (C,), 1.0), ("bl", (C,), 0.1)]
    for l in range(case["layers"]):
        lay += [("Rr%d" % l, (K, C, C), 1.0 / C), ("Ri%d" % l, (K, C, C), 1.0 / C),
                ("W%d" % l, (C, C), 1.0 / math.sqrt(C)), ("b%d" % l, (C,), 0.1)]
    return lay + [("Q1", (P, C), 1.0 / math.sqrt(C)), ("q1", (P,), 0.1), ("Q2", (P,), 1.0 / math.sqrt(P)),
                  ("q2", (1,), 0.1)]


def _sno_inputs(case, seed):
    """Flat parameters (FP32) and, for `batch` fields, u = I / max I and a target."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    theta = torch.cat([s * torch.randn(math.prod(shp), device=DEV, generator=g) for _, shp, s in _sno_layout(case)])
    n = case["n"]
    pts = _box_points(n, n, n, 1.0 / n)
    U, T = [], []
    for b in range(case["batch"]):
        f = _blobs(pts, 1000003 * seed + b, (1.0, 1.0, 1.0))
        U.append((f / f.max()).float())
        T.append((0.1 * f / f.max()).float())
    return theta, torch.stack(U), torch.stack(T)


def _sno_near(case):
    """The exact near part and the transforms' period, as surrogate.configure sets them."""
    return dict(a=CHI_MIN * 150.0, b=CHI_MAX * 150.0, h=1.0 / case["n"], r_in=3.0, r_out=7.0), (3 * case["n"]) // 2


def _sno_model(case, theta):
    M = kifmm.SNO(case["n"], case["width"], case["modes"], case["layers"], case["proj"], max_batch=case["batch"])
    near, period = _sno_near(case)
    M.set_period(period)
    M.set_near_field(near["a"], near["b"], near["h"], near["r_in"], near["r_out"])
    M.set_params(theta.cpu().numpy())
    return M


def _streamer_state(case, seed):
    """The double-headed initial condition of the streamer model (two Gaussians of 1e14 cm^-3) scaled to
    the gap, a background and a seeded perturbation of n_e."""
    h = 1.0 / case["nz"]
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    pts = _box_points(nx, ny, nz, h)
    L = torch.tensor([nx * h, ny * h, 1.0], dtype=torch.float64, device=DEV)

    def g(c, s):
        return torch.exp(-((pts - torch.tensor(c, dtype=torch.float64, device=DEV) * L) ** 2).sum(1) / s ** 2)
    n0 = 1e14 * (g((0.44, 0.5, 0.41), 0.03) + g((0.56, 0.5, 0.59), 0.03))
    gen = torch.Generator(device=DEV).manual_seed(seed)
    ne = n0 * (1.0 + 0.05 * torch.randn(n0.shape[0], dtype=torch.float64, device=DEV, generator=gen)) + 1e9
    return pts, h, ne.contiguous(), (n0 + 1e9).contiguous()


DT = 2.5e-12   # s, the paper's time step


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fmm":
        pts, h = _fmm_geometry(case)
        I = _fmm_source(case, pts, seed)
        a, b = kifmm.absorption(case["p_o2"])
        plan = kifmm.Plan(pts, h, 64, case["m0"], a, b, precision=case["precision"], repr=case["repr"],
                          pad_lattice=case["pad"])
        return dict(kind=kind, plan=plan, I=I, C=kifmm.scale_c(case["p"]))
    if kind == "batch":
        stream = torch.cuda.Stream()
        plans, Is, Cs = [], [], []
        for k, (n, p, p_o2) in enumerate(_batch_fields(case)):
            pts = _box_points(n, n, n, 1.0 / n)
            a, b = kifmm.absorption(p_o2)
            Is.append(_blobs(pts, 1000003 * seed + k, (1.0, 1.0, 1.0)).float())
            Cs.append(kifmm.scale_c(p))
            torch.cuda.synchronize()   # (the plans read the points on their own stream)
            plans.append(kifmm.Plan(pts, 1.0 / n, 64, case["m0"], a, b, precision="mixed", pad_lattice=True,
                                    stream=stream))
        return dict(kind=kind, plans=plans, Is=Is, Cs=Cs, Ss=[torch.empty_like(x) for x in Is], lanes=case["lanes"])
    if kind in ("sno_forward", "sno_train"):
        theta, U, T = _sno_inputs(case, seed)
        return dict(kind=kind, model=_sno_model(case, theta), U=U, T=T)
    if kind == "streamer":
        pts, h, ne, npi = _streamer_state(case, seed)
        plan = None
        if case["photo"]:
            a, b = kifmm.absorption(150.0)
            plan = kifmm.Plan(pts, h, 64, 6, a, b, precision="mixed", pad_lattice=True)
        s = kifmm.Streamer(case["nx"], case["ny"], case["nz"], h, plan=plan)
        return dict(kind=kind, streamer=s, ne=ne, np=npi)
    n = case["n"]
    side = math.ceil(round(n ** (1.0 / 3.0), 6))
    pts = _box_points(side, side, side, 1.0 / side)[:n].contiguous()
    a, b = kifmm.absorption(152.0)
    return dict(kind=kind, pts=pts, h=1.0 / side, I=_blobs(pts, seed, (1.0, 1.0, 1.0)), a=a, b=b,
                C=kifmm.scale_c(760.0))


def run(s):
    kind = s["kind"]
    if kind == "fmm":
        return s["plan"].eval(s["I"], C=s["C"])
    if kind == "batch":
        return kifmm.eval_batch(s["plans"], s["Is"], s["Ss"], C=s["Cs"], capture=True, lanes=s["lanes"])
    if kind == "sno_forward":
        return s["model"].forward(s["U"])
    if kind == "sno_train":
        loss = s["model"].loss_grad(s["U"], s["T"])
        s["model"].adam_step(1e-3)
        return loss, s["model"].grads()
    if kind == "streamer":   # the same step on every pass: the state is set before it
        s["streamer"].set(s["ne"], s["np"])
        s["streamer"].step(DT, 1)
        ne, npi, _, _ = s["streamer"].get()
        return ne, npi
    return kifmm.direct_noalloc(s["pts"], s["h"], s["I"], s["a"], s["b"], C=s["C"])


# ---- the work a pass cannot do without ---------------------------------------------------

def _fmm_flops(n, m0, repr, precision, leaf=64):
    """Near pairs (a product and a sum each; in the FP64 form the kernel too) and one r x r translation per
    V pair, 189 of them a box."""
    r = m0 ** 3 if repr == "cheb" else {4: 56, 6: 112, 8: 176}[m0]
    boxes = n / leaf * 8.0 / 7.0
    return 27.0 * leaf * n * (2.0 if precision == "mixed" else 30.0) + 189.0 * boxes * 2.0 * r * r


def work(case):
    kind = case["kind"]
    if kind == "fmm":
        if case["grid"] == "refined":
            c = (2 * case["half"] + 1) ** 3
            n = case["base_n"] ** 3 - c + c * 512
        else:
            n = case["nx"] * case["ny"] * case["nz"]
        w = 4 if case["precision"] == "mixed" else 8
        return dict(bytes=2.0 * w * n, flops=_fmm_flops(n, case["m0"], case["repr"], case["precision"]))
    if kind == "batch":
        ns = [n ** 3 for n, _, _ in _batch_fields(case)]
        return dict(bytes=8.0 * sum(ns), flops=sum(_fmm_flops(n, case["m0"], "surface", "mixed") for n in ns))
    if kind in ("sno_forward", "sno_train"):
        n, C, m, L, P, B = (case[k] for k in ("n", "width", "modes", "layers", "proj", "batch"))
        K = 4 * m ** 3
        dft = 2.0 * C * m * (2 * n ** 3 + 2 * 2 * m * n * n + 2 * 2 * m * 2 * n * m)   # one direction, real FMAs
        fwd = B * 2.0 * (L * (2 * dft + 4.0 * K * C * C + n ** 3 * C * C) + n ** 3 * (C * P + P))
        weights = L * 2 * K * C * C
        if kind == "sno_forward":
            return dict(bytes=8.0 * B * n ** 3 + 2.0 * weights, flops=fwd)
        return dict(bytes=8.0 * B * n ** 3 + 28.0 * weights, flops=3.0 * fwd)   # gradient, Adam: 7 words a weight
    if kind == "streamer":
        n = case["nx"] * case["ny"] * case["nz"]
        photo = 2.0 * _fmm_flops(n, 6, "surface", "mixed") if case["photo"] else 0.0
        return dict(bytes=8.0 * 4 * n, flops=2.0 * 400.0 * n + photo)
    return dict(bytes=8.0 * 5 * case["n"], flops=30.0 * case["n"] ** 2)


# ---- the results in 64 bits --------------------------------------------------------------

def _kernel(R, a, b):
    return -torch.exp(-a * R) * torch.expm1(-(b - a) * R) / (4.0 * math.pi * R ** 3 * math.log(b / a))


def _sigma(h, a, b):
    """The kernel's integral over the cell of edge h about its centre: over the six faces, the solid angle
    times (1 / (4 pi ln(b/a))) int_0^rho (e^{-ar} - e^{-br}) / r dr, by Gauss-Legendre."""
    t, w = np.polynomial.legendre.leggauss(64)
    u, wu = 0.5 * h * t, 0.5 * h * w
    rho = np.sqrt(u[:, None] ** 2 + u[None, :] ** 2 + 0.25 * h * h)
    s, ws = 0.5 * (t + 1.0), 0.5 * w
    ein = [(-np.expm1(-k * rho[..., None] * s) / s * ws).sum(-1) for k in (a, b)]   # int_0^1 (1 - e^{-k rho s}) / s ds
    m = (ein[1] - ein[0]) / (4.0 * math.pi * math.log(b / a))
    return float(6.0 * (wu[:, None] * wu[None, :] * (0.5 * h) / rho ** 3 * m).sum())


def _sum_box(I, nx, ny, nz, h, a, b, C):
    """The discrete sum on a box grid by a zero-padded FFT convolution."""
    n = (nz, ny, nx)
    d = [torch.minimum(k, 2 * m - k).double() for k, m in ((torch.arange(2 * m, device=DEV), m) for m in n)]
    R = h * torch.sqrt(d[0][:, None, None] ** 2 + d[1][None, :, None] ** 2 + d[2][None, None, :] ** 2)
    R[0, 0, 0] = 1.0
    K = _kernel(R, a, b) * h ** 3
    K[0, 0, 0] = _sigma(h, a, b)
    s = [2 * m for m in n]
    F = torch.fft.rfftn(K) * torch.fft.rfftn(I.double().reshape(n), s=s)
    return C * torch.fft.irfftn(F, s=s)[:nz, :ny, :nx].reshape(-1)


def _sum_pairs(pts, h, I, a, b, C):
    """The discrete sum pair by pair; h: one edge, or one per point."""
    n = pts.shape[0]
    I = I.double()
    edges = h if isinstance(h, torch.Tensor) else torch.full((n,), float(h), dtype=torch.float64, device=DEV)
    sig = torch.zeros_like(edges)
    for e in edges.unique().tolist():
        sig[edges == e] = _sigma(e, a, b)
    q, out = I * edges ** 3, torch.empty_like(I)
    step = max(1, (1 << 26) // n)
    for i in range(0, n, step):
        r2 = sum((pts[i:i + step, None, k] - pts[None, :, k]) ** 2 for k in range(3))
        j = torch.arange(r2.shape[0], device=DEV)
        r2[j, j + i] = 1.0
        K = _kernel(torch.sqrt(r2), a, b)
        K[j, j + i] = 0.0
        out[i:i + step] = K @ q
    return C * (out + sig * I)


def _sno_forward(case, p, u, near_table):
    """The network on one field u (n, n, n), FP64; p: parameter blocks (spectral ones as they are used)."""
    n, m = case["n"], case["modes"]
    _, N = _sno_near(case)
    j = torch.arange(n, dtype=torch.float64, device=DEV)
    kxy = torch.cat([torch.arange(m), torch.arange(N - m, N)]).double().to(DEV)
    kz = torch.arange(m, dtype=torch.float64, device=DEV)
    E = torch.polar(torch.ones((), dtype=torch.float64, device=DEV), -2.0 * math.pi / N * torch.outer(kxy, j))
    Ez = torch.polar(torch.ones((), dtype=torch.float64, device=DEV), -2.0 * math.pi / N * torch.outer(kz, j))
    wk = torch.where(kz == 0, 1.0, 2.0).double() / float(N) ** 3
    v = p["Wl"][:, None, None, None] * u[None] + p["bl"][:, None, None, None]
    for l in range(case["layers"]):
        V = torch.einsum("cxyz,az->cxya", v.to(E.dtype), Ez)
        V = torch.einsum("cxya,by->cxba", V, E)
        V = torch.einsum("cxba,ex->ceba", V, E)
        R = torch.complex(p["Rr%d" % l], p["Ri%d" % l]).reshape(2 * m, 2 * m, m, case["width"], case["width"])
        G = torch.einsum("ebaoc,ceba->oeba", R, V) * wk
        S = torch.einsum("oeba,ex->oxba", G, E.conj())
        S = torch.einsum("oxba,by->oxya", S, E.conj())
        S = torch.einsum("oxya,az->oxyz", S, Ez.conj()).real
        z = S + torch.einsum("oc,cxyz->oxyz", p["W%d" % l], v) + p["b%d" % l][:, None, None, None]
        v = torch.nn.functional.gelu(z) if l < case["layers"] - 1 else z
    hid = torch.nn.functional.gelu(torch.einsum("pc,cxyz->pxyz", p["Q1"], v) + p["q1"][:, None, None, None])
    y = torch.einsum("p,pxyz->xyz", p["Q2"], hid) + p["q2"]
    F = torch.fft.rfftn(near_table) * torch.fft.rfftn(u, s=near_table.shape)
    return y + torch.fft.irfftn(F, s=near_table.shape)[:n, :n, :n]


def _near_table(case):
    """K(h |d|) w(|d|) h^3 and the self term on the doubled grid (d the offset, 0 beyond r_out)."""
    q, _ = _sno_near(case)
    n = case["n"]
    k = torch.arange(2 * n, device=DEV)
    d = torch.minimum(k, 2 * n - k).double()
    rho = torch.sqrt(d[:, None, None] ** 2 + d[None, :, None] ** 2 + d[None, None, :] ** 2)
    t = ((rho - q["r_in"]) / (q["r_out"] - q["r_in"])).clamp(0.0, 1.0)
    w = torch.where(rho >= q["r_out"], torch.zeros_like(t), torch.cos(0.5 * math.pi * t) ** 2)
    rho[0, 0, 0] = 1.0
    tab = _kernel(q["h"] * rho, q["a"], q["b"]) * w * q["h"] ** 3
    tab[0, 0, 0] = _sigma(q["h"], q["a"], q["b"])
    return tab


def _exact_sno(case, seed):
    theta, U, T = _sno_inputs(case, seed)
    n, train = case["n"], case["kind"] == "sno_train"
    p, blocks, o = {}, [], 0
    for name, shp, _ in _sno_layout(case):
        k = math.prod(shp)
        x = theta[o:o + k].reshape(shp)
        if name.startswith("R"):   # the spectral weights are used in BF16
            x = x.bfloat16()
        p[name] = x.double().requires_grad_(train)
        blocks.append(p[name])
        o += k
    near = _near_table(case)
    if not train:
        return torch.stack([_sno_forward(case, p, U[b].double().reshape(n, n, n), near).reshape(-1)
                            for b in range(case["batch"])])
    total = 0.0
    for b in range(case["batch"]):
        y = _sno_forward(case, p, U[b].double().reshape(n, n, n), near).reshape(-1)
        loss = ((y - T[b].double()) ** 2).sum() / (case["batch"] * n ** 3)
        loss.backward()
        total += float(loss.detach())
    return total, torch.cat([x.grad.reshape(-1) for x in blocks]).cpu().numpy()


def _poisson(rho, h, phi0):
    """-Laplace(phi) = rho on the cells, Neumann side faces, phi = 0 and phi0 on the z faces half a cell out,
    by the eigenvectors of the 7-point operator."""
    rho = rho.clone()
    rho[-1] += 2.0 * phi0 / (h * h)
    nz, ny, nx = rho.shape

    def basis(n, dirichlet):
        j = torch.arange(n, dtype=torch.float64, device=DEV) + 0.5
        k = torch.arange(n, dtype=torch.float64, device=DEV) + (1.0 if dirichlet else 0.0)
        B = (torch.sin if dirichlet else torch.cos)(math.pi / n * torch.outer(k, j))
        return B / B.norm(dim=1, keepdim=True), 2.0 - 2.0 * torch.cos(math.pi / n * k)
    (Bz, lz), (By, ly), (Bx, lx) = basis(nz, True), basis(ny, False), basis(nx, False)

    def along(Mx, My, Mz, f):
        return torch.einsum("az,zbc->abc", Mz, torch.einsum("by,zyc->zbc", My, torch.einsum("cx,zyx->zyc", Mx, f)))
    f = along(Bx, By, Bz, rho) * (h * h) / (lz[:, None, None] + ly[None, :, None] + lx[None, None, :])
    return along(Bx.T, By.T, Bz.T, f)


def _faces(n, v, axis):
    """MUSCL face values with Koren's limiter (two copied ghost cells a side)."""
    m = n.shape[axis]
    lo, hi = n.narrow(axis, 0, 1), n.narrow(axis, m - 1, 1)
    g = torch.cat([lo, lo, n, hi, hi], axis)
    um, u0, u1, u2 = (g.narrow(axis, k, m + 1) for k in range(4))

    def limited(d_up, d):
        r = torch.where(d != 0, d_up / torch.where(d != 0, d, torch.ones_like(d)), torch.zeros_like(d))
        return torch.minimum(torch.minimum(2.0 * r, (1.0 + 2.0 * r) / 3.0), torch.full_like(r, 2.0)).clamp(min=0.0)
    left = u0 + 0.5 * limited(u0 - um, u1 - u0) * (u1 - u0)
    right = u1 + 0.5 * limited(u1 - u2, u0 - u1) * (u0 - u1)
    return torch.where(v >= 0, left, right)


def _exact_streamer(case, seed):
    _, h, ne, npi = _streamer_state(case, seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    ne, npi = ne.reshape(nz, ny, nx), npi.reshape(nz, ny, nx)
    p, phi0, De = 760.0, 52e3, 1800.0
    mu_e, mu_p = 2.9e5 / p, 2.6e3 / p
    C = 0.06 * 30.0 / (p + 30.0)
    e_eps = 1.602176634e-19 / 8.8541878128e-14

    def pad(x, axis, n=1):
        z = torch.zeros_like(x.narrow(axis, 0, 1))
        return torch.cat([z, x, z], axis)

    def rhs(ne, npi):
        phi = _poisson(e_eps * (npi - ne), h, phi0)
        Ex, Ey = pad(-phi.diff(dim=2) / h, 2), pad(-phi.diff(dim=1) / h, 1)
        Ez = torch.cat([-(phi[:1]) / (0.5 * h), -phi.diff(dim=0) / h, -(phi0 - phi[-1:]) / (0.5 * h)])
        mid = [0.5 * (E.narrow(ax, 1, E.shape[ax] - 1) + E.narrow(ax, 0, E.shape[ax] - 1))
               for E, ax in ((Ex, 2), (Ey, 1), (Ez, 0))]
        Em = torch.sqrt(mid[0] ** 2 + mid[1] ** 2 + mid[2] ** 2)
        Si = mu_e * ne * Em * torch.where(Em > 0, 5.7 * p * torch.exp(-260.0 * p / Em), torch.zeros_like(Em))
        src = Si
        if case["photo"]:
            src = Si + _sum_box(Si, nx, ny, nz, h, CHI_MIN * 150.0, CHI_MAX * 150.0, C).reshape(Si.shape)
        de, dp = src.clone(), src.clone()
        for E, ax in ((Ex, 2), (Ey, 1), (Ez, 0)):
            ve, vp = -mu_e * E, mu_p * E
            fe = ve * _faces(ne, ve, ax) + pad(-De * ne.diff(dim=ax) / h, ax)
            fp = vp * _faces(npi, vp, ax)
            de -= fe.diff(dim=ax) / h
            dp -= fp.diff(dim=ax) / h
        return de, dp
    a1, b1 = rhs(ne, npi)
    ne1, np1 = ne + DT * a1, npi + DT * b1
    a2, b2 = rhs(ne1, np1)
    return 0.5 * (ne + ne1 + DT * a2), 0.5 * (npi + np1 + DT * b2)


def exact(case, seed):
    kind = case["kind"]
    if kind == "fmm":
        pts, h = _fmm_geometry(case)
        if case["grid"] == "refined" and pts.shape[0] > 250000:
            return None   # (the pairs of larger sets take minutes)
        I = _fmm_source(case, pts, seed)
        a, b, C = CHI_MIN * case["p_o2"], CHI_MAX * case["p_o2"], 0.06 * 30.0 / (case["p"] + 30.0)
        if case["grid"] == "refined":
            return _sum_pairs(pts, h, I, a, b, C)
        return _sum_box(I, case["nx"], case["ny"], case["nz"], h, a, b, C)
    if kind == "batch":
        out = []
        for k, (n, p, p_o2) in enumerate(_batch_fields(case)):
            I = _blobs(_box_points(n, n, n, 1.0 / n), 1000003 * seed + k, (1.0, 1.0, 1.0)).float()
            out.append(_sum_box(I, n, n, n, 1.0 / n, CHI_MIN * p_o2, CHI_MAX * p_o2, 0.06 * 30.0 / (p + 30.0)))
        return out
    if kind in ("sno_forward", "sno_train"):
        return _exact_sno(case, seed)
    if kind == "streamer":
        return _exact_streamer(case, seed)
    s = prepare(case, seed)   # (inputs only: the direct sum keeps no plan)
    return _sum_pairs(s["pts"], s["h"], s["I"], CHI_MIN * 152.0, CHI_MAX * 152.0, 0.06 * 30.0 / 790.0)
