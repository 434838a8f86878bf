"""Performance cases: the calls a reconstruction makes through the public entry points.

A training step of the framework is E{f} on the grid, the projection P, the loss (LS, or FLS with
the ramp filter), the adjoint P^T, the weighted VJP at a subset of the grid points, and Adam.
The cases are these calls one by one, at the sizes of the repository's own workloads
(`synth.workloads()`), and whole 2-D steps; `draw` spreads the sizes between the small problems
of the batched workload and the largest cone scan.

Outputs that the library hands over as FP64 although they are sums of FP32 (or BF16) results,
the losses and the gradient, are returned in FP32, the form a program logs and feeds to an
optimizer (the binding's own FP32 gradient; the 0-d or [1] losses by one cast).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2604_09884_gb300 import inrct, synth

DEV = "cuda"
LR = 1e-4


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------
def _geom(kind, N, V, A, B=1, sod=1000.0, sdd=1500.0, span=2 * math.pi, angle0=0.0):
    return dict(geom=kind, N=N, V=V, A=A, B=B, sod=sod, sdd=sdd, span=span, angle0=angle0)


def _net(net, d, width, n_hidden, n_feat=0, sigma=8.0, hash_log2_T=0, hash_growth=0.0):
    return dict(net=net, d=d, width=width, n_hidden=n_hidden, n_feat=n_feat, sigma=sigma, hash_log2_T=hash_log2_T,
                hash_growth=hash_growth)


_FAN = _geom("fan2d", 512, 90, 729)
_CONE = _geom("cone3d", 501, 60, 768, 768)
_SIREN = _net("siren", 2, 256, 5)
_HASH = _net("hash", 2, 64, 2, hash_log2_T=19, hash_growth=1.26)


def listed():
    return [
        # the smallest call: one projection of the 128^2 parallel problem (launches and latency)
        dict(name="project_par2d_128", op="project", loss=False, **_geom("par2d", 128, 60, 183, span=math.pi)),
        # the adjoint of the 512^2 fan problem (odd number of bins)
        dict(name="backproject_fan2d_512", op="backproject", **_FAN),
        # the largest projection, with the LS residual and loss as a step takes them (odd side)
        dict(name="project_cone3d_501", op="project", loss=True, **_CONE),
        # its adjoint
        dict(name="backproject_cone3d_501", op="backproject", **_CONE),
        # the FLS loss's filter on the 256^3 scan
        dict(name="ramp_cone3d_256", op="ramp", **_geom("cone3d", 256, 40, 384, 384)),
        # grid evaluation of the 256^3 Fourier-feature network on the tensor cores
        dict(name="eval_256_ffn256_bf16", op="eval", prec="bf16", N=256, **_net("ffn", 3, 256, 4, 256)),
        # grid evaluation in the plain FP32 form (512^2 SIREN)
        dict(name="eval_512_siren256_fp32", op="eval", prec="fp32", N=512, **_SIREN),
        # the virtual loss and its backward through autograd: 2^20 points of the 501^3 grid
        dict(name="vjp_501_ffn512_bf16", op="vjp", prec="bf16", autograd=True, N=501, n_idx=1 << 20,
             **_net("ffn", 3, 256, 5, 512)),
        # the weighted VJP in the plain FP32 form at a quarter of the 512^2 grid
        dict(name="vjp_512_siren256_fp32", op="vjp", prec="fp32", autograd=False, N=512, n_idx=1 << 16, **_SIREN),
        # whole training steps: the small parallel problem (FP32, every grid point) ...
        dict(name="step_par2d_128_ffn64", op="step", prec="fp32", fls=False, n_idx=128 * 128,
             **_geom("par2d", 128, 60, 183, span=math.pi), **_net("ffn", 2, 64, 3, 64, 10.0)),
        # ... the 512^2 fan SIREN on the tensor cores ...
        dict(name="step_fan2d_512_siren256", op="step", prec="bf16", fls=False, n_idx=1 << 16, **_FAN, **_SIREN),
        # ... and the hash-encoded network with the FLS loss
        dict(name="step_fan2d_512_hash64", op="step", prec="fp32", fls=True, n_idx=1 << 16, **_FAN, **_HASH),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_geom2(rng, hi=1024):
    N = _log(rng, 96, hi)
    if rng.random() < 0.5:
        return _geom("par2d", N, rng.randint(30, 180), math.ceil(1.42 * N), span=math.pi)
    return _geom("fan2d", N, rng.randint(30, 180), math.ceil(1.42 * N), sod=4.0 * N, sdd=6.0 * N)


def _draw_geom3(rng):
    N = _log(rng, 64, 400)
    sod = round(rng.uniform(2.0, 4.0) * N, 1)
    return _geom("cone3d", N, rng.randint(20, 60), math.ceil(1.5 * N), math.ceil(rng.uniform(1.0, 1.5) * N), sod=sod,
                 sdd=1.5 * sod, angle0=round(rng.uniform(0.0, 1.0), 3))


def _draw_net(rng):
    """(network, precision) of the kinds the workloads use."""
    k = rng.choice(["ffn_bf16", "siren_bf16", "siren_fp32", "ffn_fp32", "hash_fp32"])
    L = rng.randint(3, 5)
    if k == "ffn_bf16":
        return _net("ffn", 3, rng.choice([128, 256]), L, rng.choice([64, 128, 256, 512])), "bf16"
    if k == "siren_bf16":
        return _net("siren", 2, rng.choice([128, 256]), L), "bf16"
    if k == "siren_fp32":
        return _net("siren", 2, rng.choice([64, 128, 256]), L), "fp32"
    if k == "ffn_fp32":
        return _net("ffn", 2, rng.choice([64, 128, 256]), L, rng.choice([48, 64, 100]), 10.0), "fp32"
    return _net("hash", 2, 64, rng.randint(2, 3), hash_log2_T=rng.randint(14, 19), hash_growth=1.26), "fp32"


def draw(rng):
    op = rng.choice(["project", "backproject", "ramp", "eval", "vjp", "step"])
    if op in ("project", "backproject", "ramp"):
        c = dict(op=op, **(_draw_geom2(rng) if rng.random() < 0.5 else _draw_geom3(rng)))
        if op == "project":
            c["loss"] = rng.random() < 0.5
        return c
    net, prec = _draw_net(rng)
    if op == "step" and net["d"] == 3:  # whole steps are 2-D
        net = _net("siren", 2, net["width"], net["n_hidden"])
    if op == "step":
        g = _draw_geom2(rng, 512)
        n = g["N"] ** 2
        return dict(op=op, prec=prec, fls=rng.random() < 0.5, n_idx=max(1, int(n * rng.choice([0.05, 0.25, 1.0]))), **g, **net)
    N = _log(rng, 48, 256) if net["d"] == 3 else _log(rng, 96, 512 if prec == "fp32" else 1024)
    if op == "eval":
        return dict(op=op, prec=prec, N=N, **net)
    n_idx = min(N ** net["d"], _log(rng, 1 << 12, 1 << (16 if prec == "fp32" else 20)))
    return dict(op=op, prec=prec, autograd=rng.random() < 0.5, N=N, n_idx=n_idx, **net)


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _spec(c):
    return synth.GeomSpec(c["geom"], c["N"], c["V"], c["A"], c["B"], sod=c["sod"], sdd=c["sdd"], angle0=c["angle0"],
                          span=c["span"])


def _arch(c):
    return synth.ArchSpec(c["net"], c["d"], c["width"], c["n_hidden"], n_feat=c["n_feat"], sigma=c["sigma"],
                          hash_log2_T=c["hash_log2_T"], hash_growth=c["hash_growth"])


def _gen(seed, k):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + k)
    return g


def _shapes(d, seed):
    """Ellipses / axis-aligned ellipsoids of a phantom: centres, semi-axes, intensities, angle in the xy plane."""
    rng = np.random.default_rng(int(seed) * 7 + 1)
    return [(rng.uniform(-0.45, 0.45, size=d), rng.uniform(0.05, 0.4, size=d), rng.uniform(0.1, 1.0),
             rng.uniform(0.0, math.pi)) for _ in range(12)]


def _phantom(d, N, seed):
    """Sum of ellipses on the grid (FP32, flat), the kind of object the scans image."""
    c = (torch.arange(N, device=DEV, dtype=torch.float32) * 2 + 1 - N) / N
    img = torch.zeros((N,) * d, device=DEV)
    for ctr, ax, mu, ang in _shapes(d, seed):
        X, Y = c - ctr[0], (c - ctr[1])[:, None]
        xr, yr = X * math.cos(ang) + Y * math.sin(ang), -X * math.sin(ang) + Y * math.cos(ang)
        q = (xr / ax[0]) ** 2 + (yr / ax[1]) ** 2
        if d == 3:
            q = q[None] + (((c - ctr[2]) / ax[2]) ** 2)[:, None, None]
        img += mu * (q <= 1)
    return img.reshape(-1)


def _field(shape, seed, k, noise=0.1):
    """A smooth random field with noise on top, as residuals and their backprojections are (FP32, flat)."""
    g = _gen(seed, k)
    low = torch.randn([1, 1] + [min(s, 13) for s in shape], generator=g, device=DEV)
    mode = {1: "linear", 2: "bilinear", 3: "trilinear"}[len(shape)]
    f = torch.nn.functional.interpolate(low, size=list(shape), mode=mode, align_corners=True).reshape(-1)
    return f.add_(torch.randn(f.shape, generator=g, device=DEV), alpha=noise)


def _sino_shape(c):
    return (c["V"], c["B"], c["A"]) if c["geom"] == "cone3d" else (c["V"], c["A"])


def _data2d(c, seed):
    """Measured data of a 2-D scan: the line integrals of the phantom's ellipses in closed form, plus 1 % noise."""
    px, py, ex, ey = (t.to(torch.float32) for t in _rays2d(c))
    y = torch.zeros_like(px)
    for ctr, ax, mu, ang in _shapes(2, seed):
        ca, sa = math.cos(ang), math.sin(ang)
        u0, u1 = ((px - ctr[0]) * ca + (py - ctr[1]) * sa) / ax[0], (-(px - ctr[0]) * sa + (py - ctr[1]) * ca) / ax[1]
        w0, w1 = (ex * ca + ey * sa) / ax[0], (-ex * sa + ey * ca) / ax[1]
        a, b, q = w0 * w0 + w1 * w1, u0 * w0 + u1 * w1, u0 * u0 + u1 * u1 - 1
        y += mu * 2 * torch.sqrt(torch.clamp(b * b - a * q, min=0)) / a
    y = y.reshape(-1)
    return y + 0.01 * y.max() * torch.randn(y.shape, generator=_gen(seed, 3), device=DEV)


def _fourier(c, seed):
    return synth.fourier_matrix(c["n_feat"], c["d"], c["sigma"], int(seed) + 2) if c["net"] == "ffn" else None


def _theta(c, seed):
    return torch.tensor(synth.init_theta(_arch(c), int(seed) + 3), dtype=torch.float32, device=DEV)


def _indices(n, k, seed):
    if k >= n:
        return torch.arange(n, dtype=torch.int32, device=DEV)
    pick = torch.randperm(n, generator=_gen(seed, 4), device=DEV)[:k]
    return torch.sort(pick).values.to(torch.int32)


def _adam_state(p, seed):
    """Adam moments as in the middle of a run."""
    g = _gen(seed, 5)
    m = torch.randn(p, generator=g, device=DEV)
    s = m * m + torch.rand(p, generator=g, device=DEV)
    return m.mul_(1e-1), s.mul_(1e-2)


def prepare(case, seed):
    c = case
    st = {"case": c}
    if "geom" in c:
        st["g"] = _spec(c)
    if c["op"] == "project":
        # the current image and the data it is compared with
        st["x"] = _phantom(st["g"].d, c["N"], seed) + _field((c["N"],) * st["g"].d, seed, 1, 0.02).mul_(0.1)
        st["y"] = _field(_sino_shape(c), seed, 2).mul_(0.3) if c["loss"] else None
    elif c["op"] in ("backproject", "ramp"):
        st["r"] = _field(_sino_shape(c), seed, 1)
    else:
        prec = inrct.BF16 if c["prec"] == "bf16" else inrct.FP32
        st["mlp"] = inrct.mlp_desc(_arch(c), prec, _fourier(c, seed), device=DEV)
        st["theta"] = _theta(c, seed)
        n = c["N"] ** c["d"]
        if c["op"] in ("vjp", "step"):
            st["idx"] = _indices(n, c["n_idx"], seed)
            st["scale"] = n / st["idx"].numel()
        if c["op"] == "vjp":
            st["v"] = _field((c["N"],) * c["d"], seed, 1)
            st["theta"].requires_grad_(c["autograd"])
        if c["op"] == "step":
            st["y"] = _data2d(c, seed)
            st["m"], st["s"] = _adam_state(st["mlp"].p, seed)
            st["loss"] = torch.zeros(1, dtype=torch.float64, device=DEV)
            st["ws"] = torch.empty(inrct.step_ws_bytes(st["g"], st["mlp"], st["idx"].numel()), dtype=torch.uint8, device=DEV)
            st["t"] = 100
    return st


def run(st):
    c = st["case"]
    if c["op"] == "project":
        if st["y"] is None:
            return inrct.project(st["g"], st["x"])
        z, r, loss = inrct.project(st["g"], st["x"], st["y"])
        return z, r, loss.float()
    if c["op"] == "backproject":
        return inrct.backproject(st["g"], st["r"])
    if c["op"] == "ramp":
        out, loss = inrct.ramp_filter(st["g"], st["r"])
        return out, loss.float()
    if c["op"] == "eval":
        return inrct.inr_eval_grid(st["mlp"], st["theta"], c["N"])
    if c["op"] == "vjp" and c["autograd"]:
        st["theta"].grad = None
        value = inrct.InrVirtualLoss.apply(st["theta"], st["v"], st["idx"], st["scale"], st["mlp"], c["N"])
        value.backward()
        return st["theta"].grad, value.detach().float()
    if c["op"] == "vjp":
        return inrct.inr_weighted_vjp(st["mlp"], st["theta"], c["N"], st["idx"], st["v"], st["scale"], want_f32=True)[1]
    st["t"] += 1
    inrct.grad_step(st["g"], st["mlp"], st["theta"], st["y"], st["idx"], st["scale"], inrct.adam(lr=LR, t=st["t"]), st["m"],
                    st["s"], st["loss"], ws=st["ws"], loss_kind=inrct.LOSS_FLS if c["fls"] else inrct.LOSS_LS)
    return st["theta"], st["m"], st["s"], st["loss"].float()


# ----------------------------------------------------------------------------
# the work of one pass
# ----------------------------------------------------------------------------
def _macs(c):
    """Multiply-adds of one network evaluation at one point."""
    a = _arch(c)
    enc = a.n_feat * a.d if a.kind == "ffn" else a.hash_levels * a.hash_feats * 2 ** a.d if a.kind == "hash" else 0
    return enc + sum(o * i for o, i in a.layer_shapes())


def _proj_flops(c):
    """One linear (bilinear in 3-D) interpolation and accumulation per ray and slice it crosses."""
    g = _spec(c)
    return g.m * g.N * (4 if g.d == 2 else 10)


def work(case):
    c = case
    if "geom" in c:
        n, m = c["N"] ** _spec(c).d, _spec(c).m
    if c["op"] == "project":
        return {"bytes": 4 * n + (12 if c["loss"] else 4) * m, "flops": _proj_flops(c)}
    if c["op"] == "backproject":
        return {"bytes": 4 * n + 4 * m, "flops": _proj_flops(c)}
    if c["op"] == "ramp":
        return {"bytes": 8 * m, "flops": 5 * m * math.log2(2 * c["A"]) * 4}
    p, n = _arch(c).p, c["N"] ** c["d"]
    if c["op"] == "eval":
        return {"bytes": 4 * p + 4 * n, "flops": 2 * _macs(c) * n}
    if c["op"] == "vjp":
        return {"bytes": 8 * p + 8 * c["n_idx"], "flops": 6 * _macs(c) * c["n_idx"]}
    return {"bytes": 24 * p + 4 * c["n_idx"] + 4 * m,
            "flops": 2 * _macs(c) * n + 6 * _macs(c) * c["n_idx"] + 2 * _proj_flops(c)}


# ----------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ----------------------------------------------------------------------------
F64 = dict(dtype=torch.float64, device=DEV)


def _rays2d(c):
    """A point (px, py) and the direction (ex, ey) of every ray, [V][A], in grid coordinates on [-1, 1]^2."""
    D = 2.0 / c["N"]
    beta = (c["angle0"] + c["span"] * torch.arange(c["V"], **F64) / c["V"])[:, None]
    b = (torch.arange(c["A"], **F64) - 0.5 * (c["A"] - 1))[None]
    cb, sb = torch.cos(beta), torch.sin(beta)
    if c["geom"] == "par2d":
        t = b * D
        return t * cb, t * sb, (-sb).expand(c["V"], c["A"]), cb.expand(c["V"], c["A"])
    R, gam = c["sod"] * D, b / c["sod"]
    ex, ey = -torch.cos(beta + gam), -torch.sin(beta + gam)
    Sx, Sy = R * cb, R * sb
    dot = Sx * ex + Sy * ey
    return Sx - dot * ex, Sy - dot * ey, ex, ey


def _crossings(N, px, py, ex, ey):
    """Joseph's crossing of a ray: whether x drives, crossing at slice 0, slope per slice, path length per slice."""
    D = 2.0 / N
    xd = ~(ey.abs() > ex.abs() * (1 + 1e-12))
    ea, eq = torch.where(xd, ex, ey), torch.where(xd, ey, ex)
    pa, pq = torch.where(xd, px, py), torch.where(xd, py, px)
    slope = eq / ea
    a0, q0 = (pa + 1) / D - 0.5, (pq + 1) / D - 0.5
    return xd, q0 - a0 * slope, slope, D / ea.abs(), a0, ea


def _taps2d(c, rays):
    """Flat pixel indices and weights of the two taps of every (ray, slice) of the chosen rays."""
    N = c["N"]
    px, py, ex, ey = (t.reshape(-1)[rays] for t in _rays2d(c))
    xd, u0, slope, sc, _, _ = _crossings(N, px, py, ex, ey)
    j = torch.arange(N, device=DEV)
    u = u0[:, None] + slope[:, None] * j
    i0 = torch.floor(u)
    f = u - i0
    out = []
    for k, w in ((0, 1 - f), (1, f)):
        q = i0.to(torch.int64) + k
        ok = (q >= 0) & (q < N)
        flat = torch.where(xd[:, None], q * N + j, j * N + q)
        out.append((torch.where(ok, flat, 0), torch.where(ok, w, 0.0) * sc[:, None]))
    return out


def _ray_chunks(m, N):
    step = max(1, (1 << 25) // N)
    for k in range(0, m, step):
        yield torch.arange(k, min(m, k + step), device=DEV)


def _project2d(c, x):
    z = torch.empty(c["V"] * c["A"], **F64)
    for rays in _ray_chunks(z.numel(), c["N"]):
        z[rays] = sum((x[i] * w).sum(1) for i, w in _taps2d(c, rays))
    return z


def _backproject2d(c, r):
    v = torch.zeros(c["N"] ** 2, **F64)
    for rays in _ray_chunks(c["V"] * c["A"], c["N"]):
        for i, w in _taps2d(c, rays):
            v.index_add_(0, i.reshape(-1), (w * r[rays][:, None]).reshape(-1))
    return v


def _cone_view(c, k):
    """One view of the cone scan: per column the driving axis, crossing and z magnification per slice, and the
    step length's parts."""
    N, D = c["N"], 2.0 / c["N"]
    beta = c["angle0"] + c["span"] * k / c["V"]
    cb, sb = math.cos(beta), math.sin(beta)
    R, mag = c["sod"] * D, c["sdd"] / c["sod"]
    ua = (torch.arange(c["A"], **F64) - 0.5 * (c["A"] - 1)) * D * mag
    dc = -(c["sdd"] - c["sod"]) * D
    Sx, Sy = R * cb, R * sb
    ex, ey = dc * cb - ua * sb - Sx, dc * sb + ua * cb - Sy
    L2 = ex * ex + ey * ey
    tau0 = -(Sx * ex + Sy * ey) / L2
    xd, u0, slope, sa, a0, ea = _crossings(N, Sx + tau0 * ex, Sy + tau0 * ey, ex, ey)
    j = torch.arange(N, **F64)
    u = u0[:, None] + slope[:, None] * j                       # [A][N] transverse crossing
    h = mag * (tau0[:, None] + (j - a0[:, None]) * D / ea[:, None])  # [A][N] z pitch per detector row, voxels
    rows = torch.arange(c["B"], **F64) - 0.5 * (c["B"] - 1)
    step = torch.sqrt((rows[:, None] * D * mag) ** 2 + L2) * sa  # [B][A] path length per slice
    return xd, u, h, rows, step


def _project3d(c, x):
    N, A, B = c["N"], c["A"], c["B"]
    vol = x.reshape(N, N, N)
    byy = vol.permute(1, 2, 0).contiguous().reshape(N * N, N)   # [y][x][z]
    byx = vol.permute(2, 1, 0).contiguous().reshape(N * N, N)   # [x][y][z]
    z = torch.empty(c["V"], B, A, **F64)
    for k in range(c["V"]):
        xd, u, h, rows, step = _cone_view(c, k)
        i0 = torch.floor(u)
        f = u - i0
        jj = torch.arange(N, device=DEV)
        for a0 in range(0, A, 64):
            s = slice(a0, min(A, a0 + 64))
            T = torch.zeros(s.stop - s.start, N, N + 2, **F64)   # interpolated along q, one empty z at each end
            for t, w in ((0, 1 - f[s]), (1, f[s])):
                q = i0[s].to(torch.int64) + t
                ok = (q >= 0) & (q < N)
                at = torch.where(ok, jj * N + q, 0)
                w = torch.where(ok, w, 0.0)
                T[:, :, 1:-1] += torch.where(xd[s][:, None, None], byx[at], byy[at]) * w[:, :, None]
            uz = 0.5 * N - 0.5 + rows[:, None, None] * h[s]       # [B][a][j]
            iz = torch.floor(uz)
            fz = uz - iz
            base = torch.arange((s.stop - s.start) * N, device=DEV).reshape(1, -1, N) * (N + 2)
            Tf = T.reshape(-1)
            lo = Tf[base + (iz + 1).clamp(0, N + 1).to(torch.int64)]
            hi = Tf[base + (iz + 2).clamp(0, N + 1).to(torch.int64)]
            z[k, :, s] = (lo + fz * (hi - lo)).sum(2) * step[:, s]
    return z.reshape(-1)


def _backproject3d(c, r):
    N, B = c["N"], c["B"]
    Cz = 0.5 * N - 0.5
    acc = {True: torch.zeros(N, N, N, **F64), False: torch.zeros(N, N, N, **F64)}  # [j][q][z]
    r = r.reshape(c["V"], B, c["A"])
    zz, jj, qq = torch.arange(N, **F64), torch.arange(N, device=DEV), torch.arange(N, **F64)
    for k in range(c["V"]):
        xd, u, h, rows, step = _cone_view(c, k)
        scaled = torch.cat([(r[k] * step).T, torch.zeros(c["A"], 1, **F64)], 1)  # [A][B + 1], the last row empty
        for x_drives in (True, False):
            cols = torch.nonzero(xd == x_drives).reshape(-1)
            if cols.numel() == 0:
                continue
            us = u[cols]
            if us.shape[0] > 1 and us[1, 0] < us[0, 0]:
                cols, us = cols.flip(0), us.flip(0)
            hs = h[cols]
            # S[a][j][z]: the column's rows spread along z
            S = torch.empty(cols.numel(), N, N, **F64)
            taps = int(math.ceil(2.0 / float(hs.min()))) + 1
            for a0 in range(0, cols.numel(), 64):
                hb = hs[a0:a0 + 64, :, None]
                b0 = torch.ceil((zz - 1 - Cz) / hb + 0.5 * (B - 1))
                base = torch.arange(cols[a0:a0 + 64].numel(), device=DEV)[:, None, None] * (B + 1)
                sc = scaled[cols[a0:a0 + 64]].reshape(-1)
                t = torch.zeros(hb.shape[0], N, N, **F64)
                for q in range(taps):
                    b = b0 + q
                    w = (1 - (Cz + (b - 0.5 * (B - 1)) * hb - zz).abs()).clamp_(min=0)
                    b = torch.where((b >= 0) & (b < B), b, float(B)).to(torch.int64)
                    t += w * sc[base + b]
                S[a0:a0 + 64] = t
            # the columns whose crossing lies within one pixel of q at slice j
            uT = us.T.contiguous()                                   # [j][a], rising
            first = torch.searchsorted(uT, (qq - 1).expand(N, N).contiguous(), right=True)  # [j][q]
            gap = float((uT[:, 1:] - uT[:, :-1]).min()) if cols.numel() > 1 else 1.0
            Sp = S.reshape(-1, N)
            for q in range(int(math.ceil(2.0 / gap)) + 1):
                a = first + q
                ok = a < cols.numel()
                a = torch.where(ok, a, 0)
                w = (1 - (uT.gather(1, a) - qq).abs()).clamp_(min=0) * ok
                acc[x_drives] += Sp[a * N + jj[:, None]] * w[:, :, None]
    return (acc[False].permute(2, 0, 1) + acc[True].permute(2, 1, 0)).reshape(-1)  # y-driven [y][x][z], x-driven [x][y][z]


def _ramp(c, r):
    A, tau = c["A"], 2.0 / c["N"]
    k = torch.arange(A, **F64)
    h = torch.where(k % 2 == 1, -1.0 / (math.pi * k.clamp(min=1) * tau) ** 2, torch.zeros_like(k))
    h[0] = 0.25 / tau ** 2
    i = torch.arange(A, device=DEV)
    out = (r.reshape(-1, A) @ h[(i[:, None] - i[None]).abs()] * tau).reshape(-1)
    return out, 0.5 * (r * out).sum().reshape(1)


def _encode(c, B, tables, i):
    """Layer-1 input at flat grid indices i."""
    N, d = c["N"], c["d"]
    k = torch.stack([(i // N ** a) % N for a in range(d)], 1)
    x = (2 * k + 1 - N).double() / N
    if c["net"] == "siren":
        return x
    if c["net"] == "ffn":
        ph = 2 * math.pi * (x @ B.T)
        return torch.cat([torch.cos(ph), torch.sin(ph)], 1)
    a, T, out = _arch(c), 1 << c["hash_log2_T"], []
    for l in range(a.hash_levels):
        Nl = int(math.floor(a.hash_base * a.hash_growth ** l))
        num = (2 * k + 1) * Nl
        c0, fr = num // (2 * N), (num % (2 * N)).double() / (2 * N)
        feat = 0.0
        for v in range(2 ** d):
            bits = torch.tensor([(v >> q) & 1 for q in range(d)], device=DEV)
            cc = c0 + bits
            w = torch.where(bits == 1, fr, 1 - fr).prod(1)
            if (Nl + 1) ** d <= T:
                e = sum(cc[:, q] * (Nl + 1) ** q for q in range(d))
            else:
                e = cc[:, 0] ^ ((cc[:, 1] * 2654435761) & 0xFFFFFFFF)
                if d == 3:
                    e = e ^ ((cc[:, 2] * 805459861) & 0xFFFFFFFF)
                e = e & (T - 1)
            feat = feat + w[:, None] * tables[l][e]
        out.append(feat)
    return torch.cat(out, 1)


def _net64(c, theta):
    """theta (FP64, flat) as the tables and the layers' (W, b)."""
    a = _arch(c)
    tables = theta[:a.table_params].reshape(a.hash_levels, -1, a.hash_feats) if c["net"] == "hash" else None
    off, layers = a.table_params, []
    for o, i in a.layer_shapes():
        layers.append((theta[off:off + o * i].reshape(o, i), theta[off + o * i:off + o * i + o]))
        off += o * i + o
    return tables, layers


def _forward64(c, B, theta, i):
    tables, layers = _net64(c, theta)
    h = _encode(c, B, tables, i)
    for W, b in layers[:-1]:
        z = h @ W.T + b
        h = torch.sin(_arch(c).omega0 * z) if c["net"] == "siren" else torch.relu(z)
    W, b = layers[-1]
    return (h @ W.T + b).reshape(-1)


_CHUNK = 1 << 17


def _eval64(c, B, theta):
    n = c["N"] ** c["d"]
    with torch.no_grad():
        return torch.cat([_forward64(c, B, theta, torch.arange(k, min(n, k + _CHUNK), device=DEV)) for k in range(0, n, _CHUNK)])


def _vjp64(c, B, theta, idx, v, scale):
    theta = theta.detach().requires_grad_(True)
    value = torch.zeros((), **F64)
    for k in range(0, idx.numel(), _CHUNK):
        i = idx[k:k + _CHUNK].to(torch.int64)
        part = scale * (v[i] * _forward64(c, B, theta, i)).sum()
        part.backward()
        value += part.detach()
    return theta.grad, value


def exact(case, seed):
    c = case
    w = work(c)
    if "net" in c and w["flops"] > 1.3e13:  # at the card's FP64 rate
        return None
    st = prepare(c, seed)
    if c["op"] == "project":
        z = (_project3d if c["geom"] == "cone3d" else _project2d)(c, st["x"].double())
        if not c["loss"]:
            return z
        r = z - st["y"].double()
        return z, r, 0.5 * (r * r).sum().reshape(1)
    if c["op"] == "backproject":
        return (_backproject3d if c["geom"] == "cone3d" else _backproject2d)(c, st["r"].double())
    if c["op"] == "ramp":
        return _ramp(c, st["r"].double())
    B = st["mlp"].B.double() if st["mlp"].B is not None else None
    theta = st["theta"].detach().double()
    if c["op"] == "eval":
        return _eval64(c, B, theta)
    if c["op"] == "vjp":
        grad, value = _vjp64(c, B, theta, st["idx"], st["v"].double(), st["scale"])
        return (grad, value) if c["autograd"] else grad
    r = _project2d(c, _eval64(c, B, theta)) - st["y"].double()
    loss = 0.5 * (r * r).sum().reshape(1)
    if c["fls"]:
        r, loss = _ramp(c, r)
    g, _ = _vjp64(c, B, theta, st["idx"], _backproject2d(c, r), st["scale"])
    t, b1, b2 = st["t"] + 1, 0.9, 0.999
    m = b1 * st["m"].double() + (1 - b1) * g
    s = b2 * st["s"].double() + (1 - b2) * g * g
    theta = theta - LR * (m / (1 - b1 ** t)) / (torch.sqrt(s / (1 - b2 ** t)) + 1e-8)
    return theta, m, s, loss
