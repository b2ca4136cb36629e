"""The work that users of this package have it do, as measurable cases.

Every case is one pass through the public entry points (``Plan``,
``PointsPlan``, ``hex_sources``, ``autograd.gravity``) with the inputs already
on the GPU, over the range the package is used in: latency-sized direct sums,
forward solves of the smallest and the largest models, leaf-aligned and ragged
grids, plans kept and plans rebuilt, both precisions, the misfit gradient,
closed-form voxels, deformed cells and scattered points.

A program that chose mixed precision holds its models and its fields in FP32
(its densities are FP32 and the field is handed on in the densities' type); a
program that chose FP64 holds both in FP64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1107_5951_gb300 as gf
from paper_1107_5951_gb300.autograd import gravity

G_SI = 6.67428e-11      # the package's default gravitational constant
MAX_PAIRS = 6e10        # exact() sums every pair up to this many


# ---------------------------------------------------------------- the cases
def _voxel(name, nx, ny, nz, sx, sy, p, **more):
    c = {"name": name, "kind": "forward", "nx": nx, "ny": ny, "nz": nz, "sx": sx, "sy": sy, "p": p, "h": 250.0,
         "gauss": 1, "precision": "mixed", "mode": "fmm", "voxels": "quadrature", "batch": 1,
         "volume": False, "scatter": False, "out": "g", "model": "random", "rebuild": False}
    c.update(more)
    return c


def listed():
    return [
        # a unit-test-sized direct sum, as in a script that checks a handful of stations: launches and latency
        _voxel("direct_small_mixed", 12, 10, 9, 300, 1, 0, gauss=2, mode="direct", scatter=True),
        # the FP64 reference sum of a small survey: 16^3 voxels, 2x2x2 Gauss, 64 x 64 stations
        _voxel("direct_fp64_16_gauss2", 16, 16, 16, 64, 64, 0, gauss=2, mode="direct", precision="fp64", h=1000.0),
        # the smallest request of a serving stream: 32^3 voxels, 256 x 256 stations, g_z only
        _voxel("forward_32", 32, 32, 32, 256, 256, 12, out="gz"),
        # a survey area that fits neither the leaves nor a power of two, with stations over it
        _voxel("forward_ragged_157", 157, 113, 71, 301, 223, 10),
        # field of a random-property volume at the surface and at every voxel centre (inside the sources)
        _voxel("forward_volume_128", 128, 128, 128, 512, 512, 12, volume=True),
        # the largest model of the package's benchmark: about 1e8 voxels under 1024^2 stations
        _voxel("forward_layered_464", 464, 464, 464, 1024, 1024, 10, h=100.0, model="layered"),
        # a solve on a geometry seen once: plan built, used and released in every pass
        _voxel("rebuild_layered_232", 232, 232, 232, 512, 512, 10, h=200.0, model="layered", rebuild=True),
        # the accuracy reference: the FP64 FMM at the degree of the 1e-6 bar
        _voxel("forward_fp64_128", 128, 128, 128, 256, 256, 14, precision="fp64"),
        # closed-form voxels (SUM-AN) under a dense station grid
        _voxel("sum_an_128", 128, 128, 128, 512, 512, 12, voxels="closed_form"),
        # an ensemble inversion step: 16 models, predicted g_z and the misfit gradient
        _voxel("gradient_128_x16", 128, 128, 128, 256, 256, 12, kind="gradient", batch=16, out="gz"),
        # terrain-following hexahedra whose shape changes from pass to pass: sources, plan and field
        {"name": "hex_topo_256", "kind": "hex", "nx": 256, "ny": 256, "nz": 64, "s": 512, "p": 12, "gauss": 2,
         "precision": "mixed"},
        # scattered density points carrying volumes, the plan kept
        {"name": "points_16m", "kind": "points", "n": 1 << 24, "s": 512, "p": 12, "mode": "fmm",
         "precision": "mixed", "batch": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same kinds of work over the same ranges."""
    pick = rng.choice(["direct", "forward", "forward", "ragged", "gauss2", "volume", "layered", "rebuild", "fp64",
                       "sum_an", "sum_an_direct", "gradient", "hex", "points"])
    if pick == "direct":
        prec = rng.choice(["fp64", "mixed"])
        c = _voxel("", _log(rng, 5, 40), _log(rng, 5, 40), _log(rng, 4, 32), _log(rng, 8, 6000), 1, 0,
                   gauss=rng.choice([1, 2]), mode="direct", precision=prec, scatter=True,
                   out=rng.choice(["g", "gz"]), batch=rng.choice([1, 1, 2]))
    elif pick == "forward":      # the serving range: cubes of side 32 .. 256
        n = _log(rng, 32, 256)
        c = _voxel("", n, n, n, 256, 256, rng.choice([8, 10, 12]), out=rng.choice(["g", "gz"]))
    elif pick == "ragged":
        c = _voxel("", _log(rng, 24, 260), _log(rng, 24, 260), _log(rng, 9, 140), _log(rng, 40, 700),
                   _log(rng, 40, 700), rng.choice([6, 9, 10, 12, 13]), batch=rng.choice([1, 1, 3]),
                   scatter=rng.choice([False, True]))
    elif pick == "gauss2":
        n = _log(rng, 24, 128)
        c = _voxel("", n, n, max(8, n // 2), 2 * n, 2 * n, rng.choice([10, 12]), gauss=2)
    elif pick == "volume":
        n = _log(rng, 24, 128)
        c = _voxel("", n, n, n, 2 * n, 2 * n, rng.choice([10, 12]), volume=True)
    elif pick == "layered":
        n = 4 * _log(rng, 40, 116)
        c = _voxel("", n, n, n, 1024, 1024, rng.choice([8, 10, 11]), h=46400.0 / n, model="layered")
    elif pick == "rebuild":
        n = _log(rng, 48, 320)
        s = _log(rng, 128, 1024)
        c = _voxel("", n, n, n, s, s, rng.choice([8, 10, 11]), h=46400.0 / n, model="layered", rebuild=True)
    elif pick == "fp64":
        n = _log(rng, 24, 128)
        c = _voxel("", n, n, n, 2 * n, 2 * n, rng.choice([10, 12, 14]), precision="fp64")
    elif pick == "sum_an":
        n = _log(rng, 24, 128)
        c = _voxel("", n, n, n, 2 * n, 2 * n, 12, voxels="closed_form", precision=rng.choice(["mixed", "mixed", "fp64"]))
    elif pick == "sum_an_direct":
        n = _log(rng, 6, 16)
        c = _voxel("", n, n, n, _log(rng, 100, 4096), 1, 0, voxels="closed_form", mode="direct", precision="fp64",
                   scatter=True)
    elif pick == "gradient":
        n = _log(rng, 24, 128)
        c = _voxel("", n, n, n, 2 * n, 2 * n, rng.choice([8, 10, 12]), kind="gradient",
                   batch=rng.choice([1, 2, 5, 16]), out="gz", precision=rng.choice(["mixed", "mixed", "mixed", "fp64"]))
        if c["precision"] == "fp64":
            c.update(batch=1, nx=min(n, 64), ny=min(n, 64), nz=min(n, 64), sx=2 * min(n, 64), sy=2 * min(n, 64))
    elif pick == "hex":
        n = _log(rng, 16, 224)
        c = {"kind": "hex", "nx": n, "ny": _log(rng, 16, 224), "nz": max(4, n // 4), "s": _log(rng, 32, 512),
             "p": rng.choice([8, 10, 12]), "gauss": rng.choice([1, 2, 2]), "precision": "mixed"}
    else:
        direct = rng.random() < 0.2
        c = {"kind": "points", "n": _log(rng, 1000, 8000) if direct else _log(rng, 20000, 1 << 24),
             "s": _log(rng, 8, 60) if direct else _log(rng, 32, 512), "p": rng.choice([8, 11, 12]),
             "mode": "direct" if direct else "fmm", "precision": rng.choice(["mixed", "mixed", "mixed", "fp64"]),
             "batch": 1}
        if c["precision"] == "fp64" and not direct:
            c["n"] = min(c["n"], 300000)
            c["s"] = min(c["s"], 128)
    c.pop("name", None)
    return c


# ---------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _rule(gauss):
    x, w = np.polynomial.legendre.leggauss(gauss)
    zz, yy, xx = np.meshgrid(x, x, x, indexing="ij")
    wz, wy, wx = np.meshgrid(w, w, w, indexing="ij")
    return np.stack([xx.ravel(), yy.ravel(), zz.ravel()], axis=1), (wx * wy * wz).ravel()


def _field(shape, h, corr, sigma, gen):
    """Zero-mean random field of exponential covariance on the periodic box, FP32."""
    f = torch.fft.rfftn(torch.randn(shape, generator=gen, device="cuda"))
    k2 = 0.0
    for a, n in enumerate(shape):
        freq = torch.fft.rfftfreq(n, d=h, device="cuda") if a == len(shape) - 1 else torch.fft.fftfreq(n, d=h, device="cuda")
        view = [1] * len(shape)
        view[a] = -1
        k2 = k2 + (2 * math.pi * corr * freq.reshape(view)) ** 2
    f *= (1 + k2) ** (-0.25 * (len(shape) + 1))
    f[(0,) * len(shape)] = 0
    f = torch.fft.irfftn(f, s=shape)
    return f * (sigma / float(f.std()))


def _densities(c, seed):
    gen = _gen(seed)
    shape = (c["nz"], c["ny"], c["nx"])
    h = c["h"]
    if c["model"] == "layered":
        # thirds of 2900 / 2700 / 2600 kg/m^3 (bottom to top) and three ellipsoids of +-400
        nz, ny, nx = shape
        t = nz // 3
        rho = torch.full(shape, 2700.0, device="cuda")
        rho[: nz - 2 * t] = 2900.0
        rho[nz - t:] = 2600.0
        u = torch.rand((3, 6), generator=gen, device="cuda").cpu().numpy()
        z, y, x = [(torch.arange(n, device="cuda") + 0.5) * h for n in shape]
        for e, sign in enumerate((1.0, -1.0, 1.0)):
            ctr = [n * h * (0.1 + 0.8 * u[e, a]) for a, n in enumerate((nx, ny, nz))]
            ax = 2000.0 + 6000.0 * u[e, 3:]
            q = ((x - ctr[0]) / ax[0]) ** 2 + (((y - ctr[1]) / ax[1]) ** 2)[:, None] + (((z - ctr[2]) / ax[2]) ** 2)[:, None, None]
            rho += (400.0 * sign) * (q < 1.0)
        rho = rho[None]
    else:
        rho = torch.stack([_field(shape, h, 2000.0, 150.0, gen) for _ in range(c["batch"])])
    rho = rho.to(torch.float64 if c["precision"] == "fp64" else torch.float32)
    return (rho if c["batch"] > 1 else rho[0]).contiguous()


def _lattice(x1, y1, sx, sy, z):
    """sx * sy stations, cell-centred over [0, x1] x [0, y1] at height z, x fastest."""
    xs = (torch.arange(sx, device="cuda", dtype=torch.float64) + 0.5) * (x1 / sx)
    ys = (torch.arange(sy, device="cuda", dtype=torch.float64) + 0.5) * (y1 / sy)
    yy, xx = torch.meshgrid(ys, xs, indexing="ij")
    return torch.stack([xx.ravel(), yy.ravel(), torch.full((sx * sy,), float(z), device="cuda", dtype=torch.float64)], dim=1)


def _centres(c):
    h = c["h"]
    x, y, z = [(torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * h for n in (c["nx"], c["ny"], c["nz"])]
    zz, yy, xx = torch.meshgrid(z - c["nz"] * h, y, x, indexing="ij")
    return torch.stack([xx.ravel(), yy.ravel(), zz.ravel()], dim=1)


def _stations(c, seed):
    """The grid's top face is z = 0; scattered stations fly up to 300 m over it, as an aerial survey does."""
    X, Y, m = c["nx"] * c["h"], c["ny"] * c["h"], c["sx"] * c["sy"]
    if c["scatter"]:
        u = torch.rand((m, 3), generator=_gen(seed + 7919), device="cuda", dtype=torch.float64)
        return u * torch.tensor([X, Y, 300.0], device="cuda", dtype=torch.float64)
    obs = _lattice(X, Y, c["sx"], c["sy"], 100.0 if c["mode"] == "direct" else 0.0)
    return torch.cat([obs, _centres(c)]) if c["volume"] else obs.contiguous()


def _plan(c, obs):
    xi, w = _rule(c["gauss"])
    return gf.Plan((c["nx"], c["ny"], c["nz"]), (0.0, 0.0, -c["nz"] * c["h"]), (c["h"],) * 3, xi, w, obs, mode=c["mode"],
                   precision=c["precision"], p=c["p"] or 8, max_batch=c["batch"], voxels=c["voxels"])


def _surface(x, y, seed):
    """Five Gaussian hills and valleys of up to 800 m over 16 km x 16 km."""
    u = torch.rand((5, 4), generator=_gen(seed), device="cuda", dtype=torch.float64).cpu().numpy()
    z = torch.zeros_like(x)
    for cx, cy, wd, a in u:
        wd = 16000.0 * (0.08 + 0.17 * wd)
        z = z + 800.0 * (2 * a - 1) * torch.exp(-((x - 16000.0 * cx) ** 2 + (y - 16000.0 * cy) ** 2) / (2 * wd * wd))
    return z


def _hex_inputs(c, seed):
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    x = torch.linspace(0, 16000.0, nx + 1, device="cuda", dtype=torch.float64)
    y = torch.linspace(0, 16000.0, ny + 1, device="cuda", dtype=torch.float64)
    yy, xx = torch.meshgrid(y, x, indexing="ij")
    t = torch.linspace(0, 1, nz + 1, device="cuda", dtype=torch.float64)[:, None, None]
    zz = -8000.0 + (_surface(xx, yy, seed) + 8000.0) * t
    nodes = torch.stack([xx.expand_as(zz), yy.expand_as(zz), zz], dim=-1)
    verts = torch.stack([nodes[k:nz + k, j:ny + j, i:nx + i] for k in (0, 1) for j in (0, 1) for i in (0, 1)], dim=3)
    rho = 2670.0 + _field((nz, ny, nx), 16000.0 / nx, 2000.0, 150.0, _gen(seed + 1)).reshape(-1)
    obs = _lattice(16000.0, 16000.0, c["s"], c["s"], 0.0)
    obs[:, 2] = _surface(obs[:, 0], obs[:, 1], seed) + 50.0
    return verts.reshape(-1, 8, 3).contiguous(), rho.contiguous(), obs


def _points_inputs(c, seed):
    gen = _gen(seed)
    n = c["n"]
    ext = torch.tensor([16000.0, 16000.0, 4000.0], device="cuda", dtype=torch.float64)
    x = torch.rand((n, 3), generator=gen, device="cuda", dtype=torch.float64) * ext
    x[:, 2] -= 4000.0
    a = (16000.0 * 16000.0 * 4000.0 / n) * (0.5 + torch.rand(n, generator=gen, device="cuda", dtype=torch.float64))
    dt = torch.float64 if c["precision"] == "fp64" else torch.float32
    rho = (2670.0 + 250.0 * torch.randn((c["batch"], n), generator=gen, device="cuda")).to(dt)
    obs = _lattice(16000.0, 16000.0, c["s"], c["s"], 50.0)
    return x, a, (rho if c["batch"] > 1 else rho[0]).contiguous(), obs


def _data(c, seed):
    """Observed g_z: a smooth anomaly of 1e-4 m/s^2, one map for each model."""
    gen = _gen(seed + 104729)
    d = torch.stack([_field((c["sy"], c["sx"]), c["nx"] * c["h"] / c["sx"], 2000.0, 1e-4, gen).reshape(-1)
                     for _ in range(c["batch"])]).double()
    return d if c["batch"] > 1 else d[0]


def prepare(case, seed):
    c = case
    if c["kind"] == "hex":
        verts, rho, obs = _hex_inputs(c, seed)
        return {"case": c, "verts": verts, "rho": rho, "obs": obs, "rule": _rule(c["gauss"])}
    if c["kind"] == "points":
        x, a, rho, obs = _points_inputs(c, seed)
        return {"case": c, "rho": rho, "plan": gf.PointsPlan(x, a, obs, per_cell=1, mode=c["mode"], precision=c["precision"],
                                                             p=c["p"], max_batch=c["batch"])}
    s = {"case": c, "rho": _densities(c, seed), "obs": _stations(c, seed)}
    if not c["rebuild"]:
        s["plan"] = _plan(c, s["obs"])
    if c["kind"] == "gradient":
        s["rho"].requires_grad_(True)
        s["data"] = _data(c, seed)
    return s


# ---------------------------------------------------------------- one pass
def _field_of(plan, c, rho):
    g, gz = plan.forward(rho, want_g=c.get("out", "g") == "g", want_gz=c.get("out", "g") == "gz")
    return (g if g is not None else gz).to(rho.dtype)


def run(state):
    c = state["case"]
    if c["kind"] == "hex":
        xi, w = state["rule"]
        x, a = gf.hex_sources(state["verts"], xi, w, precision=c["precision"])
        with gf.PointsPlan(x, a, state["obs"], per_cell=len(w), mode="fmm", precision=c["precision"], p=c["p"]) as plan:
            return _field_of(plan, c, state["rho"])
    if c["kind"] == "gradient":
        rho = state["rho"]
        gz = gravity(rho, state["plan"], "gz")
        grad, = torch.autograd.grad(gz, rho, gz.detach() - state["data"])
        return {"gz": gz.detach().to(rho.dtype), "grad": grad}
    if c.get("rebuild"):
        with _plan(c, state["obs"]) as plan:
            return _field_of(plan, c, state["rho"])
    return _field_of(state["plan"], c, state["rho"])


# ---------------------------------------------------------------- what a pass cannot do without
def _fmm_flops(leaf_sources, obs, leaves, offsets, near_leaves, nsrc, p, p2m_per_source):
    """Near pairs at 20 flops, one 2 K^2 product per interaction-list pair, the P2M."""
    K = (p + 1) ** 2
    return obs * near_leaves * leaf_sources * 20.0 + leaves * offsets * 2.0 * K * K + nsrc * p2m_per_source


def work(case):
    c = case
    if c["kind"] in ("hex", "points"):
        nsrc = c["n"] if c["kind"] == "points" else c["nx"] * c["ny"] * c["nz"] * c["gauss"] ** 3
        ncell = c["n"] if c["kind"] == "points" else c["nx"] * c["ny"] * c["nz"]
        m, p, el = c["s"] ** 2, c["p"], 8 if c["precision"] == "fp64" else 4
        read = (192.0 * ncell + 24.0 * m) if c["kind"] == "hex" else (16.0 if el == 4 else 32.0) * nsrc
        if c.get("mode") == "direct":
            return {"bytes": read + el * (nsrc + 3 * m), "flops": 20.0 * nsrc * m}
        side = (16000.0 * 16000.0 * (8000.0 if c["kind"] == "hex" else 4000.0) / max(1.0, nsrc / 48.0)) ** (1 / 3)
        leaves = min(m, (16000.0 / side) ** 2)
        return {"bytes": read + el * (ncell + 3.0 * m),
                "flops": _fmm_flops(48.0, m, leaves * 4 / 3, 100.0, 15.0, nsrc, p, 5.0 * (p + 1) * (p + 2))}
    el = 8 if c["precision"] == "fp64" else 4
    nvox, m, B = c["nx"] * c["ny"] * c["nz"], c["sx"] * c["sy"], c["batch"]
    nq = c["gauss"] ** 3 if c["voxels"] == "quadrature" else 1
    if c["volume"]:
        m += nvox
    ncomp = 3 if c["out"] == "g" else 1
    bytes_ = B * el * (nvox + ncomp * m) + (24.0 if c["rebuild"] else 3.0 * el) * m
    if c["mode"] == "direct":
        flops = B * m * (20.0 * nvox * nq if c["voxels"] == "quadrature" else 100.0 * (nvox + 1))
    else:
        b = 4 if nq == 1 else 2
        leaves = (c["nx"] / b) * (c["ny"] / b) * (c["nz"] / b if c["volume"] else 1)
        full = 8 / 7 * 189 if c["volume"] else 4 / 3 * 63
        near = 27 if c["volume"] else 9
        flops = B * _fmm_flops(b ** 3 * nq, m, min(leaves, m), full, near, nvox, c["p"], 2.0 * (c["p"] + 1) ** 2)
        if c["voxels"] == "closed_form":
            flops += B * m * 150 * 100.0
    if c["kind"] == "gradient":
        bytes_ += B * (el * nvox + 8.0 * m)
        flops *= 2
    return {"bytes": float(bytes_), "flops": float(flops)}


# ---------------------------------------------------------------- the same in plain 64-bit torch
def _all_pairs(src, mass, obs, comps):
    """G sum_s m_s (r - x_s) / |r - x_s|^3, components `comps`; mass [B][S].  Returns [B][M][len(comps)]."""
    out = torch.empty((mass.shape[0], obs.shape[0], len(comps)), device="cuda", dtype=torch.float64)
    step = max(1, int(3e7) // max(1, src.shape[0]))
    cut = min(src.shape[0], int(3e7))
    for m0 in range(0, obs.shape[0], step):
        o = obs[m0:m0 + step]
        acc = torch.zeros((mass.shape[0], o.shape[0], len(comps)), device="cuda", dtype=torch.float64)
        for s0 in range(0, src.shape[0], cut):
            d = [o[:, a, None] - src[None, s0:s0 + cut, a] for a in range(3)]
            r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
            k = torch.where(r2 > 0, r2, torch.inf).rsqrt() ** 3
            for q, a in enumerate(comps):
                acc[:, :, q] += (mass[:, s0:s0 + cut] @ (k * d[a]).T)
        out[:, m0:m0 + step] = acc
    return G_SI * out


def _corner(u, v, w):
    """Closed-form corner terms of a prism, the vanishing ones zero (u, v, w: corner minus observer)."""
    r = torch.sqrt(u * u + v * v + w * w)

    def ln(a, q):
        v_ = torch.where(a >= 0, a + r, q / (r - a).clamp_min(1e-300))
        return torch.where(q > 0, torch.log(v_.clamp_min(1e-300)), torch.zeros_like(v_))

    def at(x, n):
        den = x * r
        return torch.where(x != 0, x * torch.atan(n / torch.where(den != 0, den, torch.ones_like(den))), torch.zeros_like(den))

    lu, lv, lw = ln(u + 0 * r, v * v + w * w + 0 * r), ln(v + 0 * r, u * u + w * w + 0 * r), ln(w + 0 * r, u * u + v * v + 0 * r)
    return v * lw + w * lv - at(u + 0 * r, v * w), w * lu + u * lw - at(v + 0 * r, w * u), u * lv + v * lu - at(w + 0 * r, u * v)


def _unit_kernel(c, dx, dy, dz, comps):
    """Field (without G) per unit density of a voxel centred at the origin, at the separations dx, dy, dz (broadcast)."""
    h = c["h"]
    if c["voxels"] == "closed_form":
        out = [0.0, 0.0, 0.0]
        for k in (0, 1):
            for j in (0, 1):
                for i in (0, 1):
                    f = _corner((i - 0.5) * h - dx, (j - 0.5) * h - dy, (k - 0.5) * h - dz)
                    s = 1.0 if (i + j + k) & 1 else -1.0
                    out = [o + s * t for o, t in zip(out, f)]
        return [out[a] for a in comps]
    xi, w = _rule(c["gauss"])
    out = [0.0 for _ in comps]
    for q in range(len(w)):
        d = [dx - 0.5 * h * xi[q, 0], dy - 0.5 * h * xi[q, 1], dz - 0.5 * h * xi[q, 2]]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        k = torch.where(r2 > 0, r2, torch.inf).rsqrt() ** 3 * (h ** 3 * w[q] / w.sum())
        out = [o + k * d[a] for o, a in zip(out, comps)]
    return out


def _offsets(n, h, shift):
    """Separations shift + h * (station index - voxel index) in wrap-around order on 2 n points."""
    i = torch.arange(2 * n, device="cuda", dtype=torch.float64)
    return shift + h * torch.where(i < n, i, i - 2 * n)


def _by_convolution(c, rho, comps, r=None):
    """The field at a station lattice with whole numbers of stations per voxel (and at the voxel centres) by FFT over the
    layers; with r [B][M] (g_z only): the transpose applied to it.  rho [B][nz][ny][nx] FP64."""
    nx, ny, nz, h = c["nx"], c["ny"], c["nz"], c["h"]
    fx, fy = c["sx"] // nx, c["sy"] // ny
    B = rho.shape[0]
    size = (2 * ny, 2 * nx)
    m = c["sx"] * c["sy"]
    out = torch.empty((B, m + (nx * ny * nz if c["volume"] else 0), len(comps)), device="cuda", dtype=torch.float64)
    grad = torch.zeros_like(rho)
    layer = torch.arange(nz, device="cuda", dtype=torch.float64)
    dz = (nz - layer - 0.5) * h          # the stations lie on the top face
    top = out[:, :m].reshape(B, ny, fy, nx, fx, len(comps))
    for j in range(fy):
        for i in range(fx):
            dx = _offsets(nx, h, ((i + 0.5) / fx - 0.5) * h)[None, None, :]
            dy = _offsets(ny, h, ((j + 0.5) / fy - 0.5) * h)[None, :, None]
            for z0 in range(0, nz, 16):
                kern = _unit_kernel(c, dx, dy, dz[z0:z0 + 16, None, None], comps)
                if r is None:
                    f = torch.fft.rfft2(rho[:, z0:z0 + 16], s=size)
                    for q, k in enumerate(kern):
                        g = torch.fft.irfft2((f * torch.fft.rfft2(k)).sum(1), s=size)[:, :ny, :nx]
                        if z0 == 0:
                            top[:, :, j, :, i, q] = G_SI * g
                        else:
                            top[:, :, j, :, i, q] += G_SI * g
                else:
                    f = torch.fft.rfft2(r.reshape(B, ny, fy, nx, fx)[:, :, j, :, i], s=size)
                    g = torch.fft.irfft2(f[:, None] * torch.fft.rfft2(kern[0]).conj(), s=size)[:, :, :ny, :nx]
                    grad[:, z0:z0 + 16] += G_SI * g
    if r is not None:
        return grad
    if c["volume"]:
        s3 = (2 * nz, 2 * ny, 2 * nx)
        kern = _unit_kernel(c, _offsets(nx, h, 0.0)[None, None, :], _offsets(ny, h, 0.0)[None, :, None],
                            _offsets(nz, h, 0.0)[:, None, None], comps)
        f = torch.fft.rfftn(rho, s=s3, dim=(1, 2, 3))
        for q, k in enumerate(kern):
            out[:, m:, q] = G_SI * torch.fft.irfftn(f * torch.fft.rfftn(k), s=s3, dim=(1, 2, 3))[:, :nz, :ny, :nx].reshape(B, -1)
    return out


def _hex_nodes(c, verts):
    xi, w = _rule(c["gauss"])
    xs, ws = [], []
    for q in range(len(w)):
        p, J = 0.0, [0.0, 0.0, 0.0]
        for a in range(8):
            s = np.array([2.0 * (a & 1) - 1, 2.0 * ((a >> 1) & 1) - 1, 2.0 * (a >> 2) - 1])
            f = 1.0 + s * xi[q]
            v = verts[:, a]
            p = p + 0.125 * f[0] * f[1] * f[2] * v
            J = [J[0] + 0.125 * s[0] * f[1] * f[2] * v, J[1] + 0.125 * f[0] * s[1] * f[2] * v, J[2] + 0.125 * f[0] * f[1] * s[2] * v]
        xs.append(p)
        ws.append(8.0 * w[q] / w.sum() * torch.linalg.det(torch.stack(J, dim=2)).abs())
    return torch.stack(xs, dim=1).reshape(-1, 3), torch.stack(ws, dim=1).reshape(-1)


def exact(case, seed):
    c = case
    if c["kind"] in ("hex", "points"):
        m = c["s"] ** 2
        n = c["n"] if c["kind"] == "points" else c["nx"] * c["ny"] * c["nz"] * c["gauss"] ** 3
        if float(m) * n > MAX_PAIRS:
            return None
        if c["kind"] == "points":
            x, a, rho, obs = _points_inputs(c, seed)
            mass = rho.reshape(c["batch"], -1).double() * a
        else:
            verts, rho, obs = _hex_inputs(c, seed)
            x, a = _hex_nodes(c, verts)
            mass = (rho.double().repeat_interleave(c["gauss"] ** 3) * a)[None]
        g = _all_pairs(x, mass, obs, (0, 1, 2))
        return g if c.get("batch", 1) > 1 else g[0]
    rho = _densities(c, seed).double().reshape(c["batch"], c["nz"], c["ny"], c["nx"])
    comps = (0, 1, 2) if c["out"] == "g" else (2,)
    obs = _stations(c, seed)
    lattice = c["mode"] == "fmm" and not c["scatter"] and c["sx"] % c["nx"] == 0 and c["sy"] % c["ny"] == 0
    nq = c["gauss"] ** 3
    pairs = float(obs.shape[0]) * rho[0].numel() * (nq if c["voxels"] == "quadrature" else 60)
    if lattice:
        f = _by_convolution(c, rho, comps)
    elif pairs > MAX_PAIRS:
        return None
    else:
        cen = _centres(c)
        if c["voxels"] == "quadrature":
            xi, w = _rule(c["gauss"])
            xi = torch.tensor(xi, device="cuda") * (0.5 * c["h"])
            src = (cen[:, None, :] + xi[None]).reshape(-1, 3)
            wq = torch.tensor(w / w.sum(), device="cuda") * c["h"] ** 3
            mass = (rho.reshape(c["batch"], -1, 1) * wq).reshape(c["batch"], -1)
            f = _all_pairs(src, mass, obs, comps)
        else:
            f = torch.zeros((c["batch"], obs.shape[0], len(comps)), device="cuda", dtype=torch.float64)
            for m0 in range(0, obs.shape[0], 1024):
                o = obs[m0:m0 + 1024]
                k = _unit_kernel(c, *[o[:, a, None] - cen[None, :, a] for a in range(3)], comps)
                for q in range(len(comps)):
                    f[:, m0:m0 + 1024, q] = G_SI * (rho.reshape(c["batch"], -1) @ k[q].T)
    if c["kind"] == "gradient":
        gz = f[:, :, 0]
        resid = gz - _data(c, seed).reshape(c["batch"], -1)
        if not lattice:
            return None
        grad = _by_convolution(c, rho, (2,), resid)
        one = c["batch"] == 1
        return {"gz": gz[0] if one else gz, "grad": grad[0] if one else grad}
    f = f if c["out"] == "g" else f[:, :, 0]
    return f if c["batch"] > 1 else f[0]
