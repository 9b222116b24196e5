"""The work that users of this package have it do, as cases that can be timed and checked.

Every case is one call (or one short run) through the public entry points of ``paper_1201_2450_gb300`` on
seeded synthetic inputs of the kinds ``synth`` makes: layered ellipsoid phantoms with a moving tumour, their
analytic projections with Poisson noise, and noisy streaked images.  ``exact`` restates the operations in
FP64 with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1201_2450_gb300 as tnlm
from paper_1201_2450_gb300 import synth

DEV = "cuda"
DTYPES = {"fp32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16}


# --------------------------------------------------------------------------------------------------
# cases
# --------------------------------------------------------------------------------------------------


def _scan(kind, *, np_, nx, ny, nz, field, views, nu, nv, pixel, dz=None, i0=5e4, uneven=False, offset=0.0, **more):
    """A case on a cone-beam scan: np_ phases of nx x ny x nz voxels over `field` mm in x, `views` per phase."""
    dx = field / nx
    return dict(kind=kind, np=np_, nx=nx, ny=ny, nz=nz, dx=dx, dz=dz if dz else dx, views=views, uneven=uneven,
                nu=nu, nv=nv, pixel=pixel, i0=i0, offset=offset, **more)


def _images(kind, *, np_, nx, ny, nz, d, M, h, **more):
    return dict(kind=kind, np=np_, nx=nx, ny=ny, nz=nz, d=d, M=M, h=h, **more)


def listed():
    return [
        # a phantom study or a unit-test-sized reconstruction: a few short launches per iteration
        _scan("recon", np_=4, nx=32, ny=32, nz=32, field=32.0, views=20, nu=64, nv=48, pixel=1.5, i0=1e5, d=1, M=2,
              h=0.02, n_outer=5, dtype="fp32") | {"name": "recon_small"},
        # one FBS iteration of the NCAT-shaped 4D reconstruction, the workload the package is quoted on
        _scan("recon", np_=10, nx=256, ny=256, nz=64, field=512.0, views=36, nu=512, nv=384, pixel=0.78, d=1, M=3,
              h=0.02, n_outer=1, dtype="fp32") | {"name": "recon_ncat"},
        # the forward projection on its own (simulated scans, residual checks), cubic phases and a half-size detector
        _scan("project", np_=10, nx=128, ny=128, nz=128, field=256.0, views=40, nu=256, nv=192, pixel=1.56)
        | {"name": "project_cubic"},
        # the transpose on its own with odd sizes on every axis, uneven phase bins and a gantry offset
        _scan("backproject", np_=6, nx=189, ny=173, nz=57, field=430.0, dz=2.5, views=31, uneven=True, nu=389, nv=287,
              pixel=1.1, offset=0.13) | {"name": "backproject_odd"},
        # the weights + Gauss-Jacobi sweep of a reconstruction, the largest phase volume of the batch protocol
        _images("sweep", np_=8, nx=256, ny=256, nz=96, d=1, M=3, h=0.02, dtype="fp32") | {"name": "sweep_d1"},
        # enhancement of a clinical set: patch 5^3, window 7^3, full-resolution FP32 images
        _images("enhance", np_=10, nx=512, ny=512, nz=128, d=2, M=3, h=0.04, n_outer=1, dtype="fp32")
        | {"name": "enhance_large"},
        # the same enhancement on 16-bit images at half the in-plane resolution and odd sizes
        _images("enhance", np_=10, nx=251, ny=243, nz=61, d=2, M=3, h=0.04, n_outer=1, dtype="bf16")
        | {"name": "enhance_bf16"},
        # one training step on the total energy, weights frozen: forward and backward through autograd
        _scan("energy", np_=10, nx=128, ny=128, nz=128, field=256.0, views=40, nu=256, nv=192, pixel=1.56, d=1, M=2,
              h=0.02, through=False) | {"name": "energy_frozen"},
        # the same with the weights differentiated, on a smaller set with odd sizes
        _scan("energy", np_=6, nx=95, ny=90, nz=71, field=190.0, views=24, nu=192, nv=150, pixel=1.56, offset=0.05,
              d=1, M=2, h=0.02, through=True) | {"name": "energy_weights"},
        # (P1) by conjugate gradients, the solver the paper names, on the smallest grid of the batch protocol
        _scan("cgls", np_=6, nx=128, ny=128, nz=48, field=512.0, views=20, nu=384, nv=288, pixel=1.04, n_iter=3)
        | {"name": "cgls"},
        # FDK of every phase: the initial image of a reconstruction and the input of an enhancement
        _scan("fdk", np_=10, nx=256, ny=256, nz=64, field=512.0, views=36, nu=512, nv=384, pixel=0.78)
        | {"name": "fdk_ncat"},
        # uneven reconstructions of several patients in one captured plan, 16-bit storage, two iterations
        dict(kind="batch", problems=4, iterations=2, dtype="bf16", name="batch_bf16"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_scan(rng, kind, nx_hi=256, nz_hi=96, **more):
    nx = _log(rng, 32, nx_hi)
    ny = max(24, int(nx * rng.uniform(0.8, 1.0)))
    nz = _log(rng, 12, min(nz_hi, 2 * nx))
    nu = _log(rng, 64, 512)
    nv = max(40, int(nu * rng.uniform(0.6, 0.8)))
    field = nx * rng.uniform(1.0, 4.0) if nx < 100 else rng.uniform(250.0, 512.0)
    c = _scan(kind, np_=rng.randint(3, 10), nx=nx, ny=ny, nz=nz, field=field, dz=field / nx * rng.uniform(1.0, 1.3),
              views=rng.randint(9, 60), uneven=rng.random() < 0.5, nu=nu, nv=nv,
              pixel=1.6 * field / nu * rng.uniform(0.8, 1.1), offset=rng.uniform(0.01, 0.2))
    return c | more


def _draw(rng):
    kind = rng.choice(["recon", "project", "backproject", "sweep", "enhance", "energy", "cgls", "fdk"])
    M = rng.randint(1, 3)
    if kind in ("sweep", "enhance"):
        d = rng.choice([1, 1, 2, 2, 2, 0, 3]) if rng.random() < 0.5 else rng.choice([1, 2])
        # the direct form serves the other radii: small images, FP32
        box = d in (1, 2)
        nx = _log(rng, 30, 400 if box else 100)
        c = _images(kind, np_=rng.randint(2, 10), nx=nx, ny=max(20, int(nx * rng.uniform(0.7, 1.1))),
                    nz=_log(rng, 12, 128 if box else 48), d=d, M=M, h=0.02 if d < 2 else 0.04,
                    dtype=rng.choice(["fp32", "fp32", "bf16", "fp16"]) if box else "fp32")
        return c | ({"n_outer": 1 if c["dtype"] != "fp32" else rng.randint(1, 2)} if kind == "enhance" else {})
    if kind == "recon":
        return _draw_scan(rng, kind, d=rng.choice([1, 1, 2]), M=M, h=0.02, n_outer=rng.randint(1, 2),
                          dtype=rng.choice(["fp32", "fp32", "fp16"]))
    if kind == "energy":
        return _draw_scan(rng, kind, nx_hi=128, d=1, M=min(M, 2), h=0.02, through=rng.random() < 0.4)
    if kind == "cgls":
        return _draw_scan(rng, kind, nx_hi=160, n_iter=rng.randint(2, 4))
    return _draw_scan(rng, kind)


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        c = _draw(rng)
        if _cost(c) <= most:
            return c


# --------------------------------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------------------------------


def _views(case):
    """Views of each phase: equal bins, or bins that differ by up to a quarter."""
    v = case["views"]
    return [v + (k * 5) % 7 - 3 if case["uneven"] else v for k in range(case["np"])]


def _geom(case):
    return synth.make_geometry(nx=case["nx"], ny=case["ny"], nz=case["nz"], dx=case["dx"], dz=case["dz"],
                               nu=case["nu"], nv=case["nv"], du=case["pixel"], n_phases=case["np"],
                               views_per_phase=_views(case), angle_offset=case["offset"])


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _noise(shape, gen, sigma):
    return torch.randn(shape, generator=gen, device=DEV, dtype=torch.float32) * sigma


def _phantom(case, geom, seed):
    """(objects, rasterised phantom): a thorax scaled to the field, its size drawn from the seed (0.9 .. 1 of it)."""
    scale = (0.9 + 0.1 * np.random.default_rng(seed).random()) * case["nx"] * case["dx"] / 512.0
    objs = synth._thorax_objects(case["np"], scale)
    return objs, synth.rasterize(geom, objs, device=DEV)


def _measured(geom, objs, i0, seed):
    return synth.poisson_log(synth.analytic_projections(geom, objs, device=DEV), i0, seed).float()


def _tau(geom):
    """A gradient step below 1 / ||P||^2: the norm is at most the largest row sum times the largest column sum of
    P, here the diagonal of the field times the views' magnified voxel cross-sections."""
    path = math.hypot(geom["nx"] * geom["dx"], geom["ny"] * geom["dy"])
    voxel = geom["dx"] * geom["dy"] * geom["dz"] * (geom["sdd"] / geom["sad"]) ** 2 / (geom["du"] * geom["dv"])
    return 1.0 / (float(max(geom["nviews"])) * path * voxel)


def _streaked(case, seed):
    cfg = synth.EnhanceConfig("images", case["np"], (case["nx"], case["ny"], case["nz"]), 1.0, 0.002, 0.003, 36,
                              case["d"], case["M"], case["h"], 1.0, 1, seed)
    return synth.enhance_input(cfg, device=DEV)[0].to(DTYPES[case["dtype"]])


def _batch_cases(case):
    """Uneven problems over the batch protocol: 6-10 phases, 128^2 x 48 .. 256^2 x 96, 20-60 views."""
    out = []
    for k in range(case["problems"]):
        t = k / max(1, case["problems"] - 1)
        nx = 16 * int(round((128 + 128 * t) / 16))
        out.append(_scan("recon", np_=6 + (3 * k) % 5, nx=nx, ny=nx, nz=8 * int(round((48 + 48 * t) / 8)), field=512.0,
                         views=24 + (13 * k) % 24, uneven=True, nu=384 + 32 * (k % 4), nv=288 + 24 * (k % 4), pixel=1.0,
                         d=1, M=3, h=0.02, n_outer=1, dtype=case["dtype"]))
    return out


def _recon_inputs(case, seed):
    geom = _geom(case)
    objs, truth = _phantom(case, geom, seed)
    t = DTYPES[case.get("dtype", "fp32")]
    y = _measured(geom, objs, case["i0"], seed).to(t)
    return geom, y, (truth + _noise(truth.shape, _gen(seed + 1), 0.001)).to(t)


def _params(case, geom=None):
    return tnlm.Params(d=case["d"], M=case["M"], h=case["h"], mu=1.0, tau=_tau(geom) if geom else 0.0,
                       n_outer=case.get("n_outer", 1), clip_nonneg=1)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("sweep", "enhance"):
        s["g"] = _streaked(case, seed)
        s["params"] = _params(case)
        return s
    if kind == "batch":
        s["geoms"], s["ys"], s["f0"], params = [], [], [], []
        for k, c in enumerate(_batch_cases(case)):
            geom, y, f0 = _recon_inputs(c, seed + 100 * k)
            s["geoms"].append(tnlm.tnlm_create_geometry(geom))
            s["ys"].append(y)
            s["f0"].append(f0)
            params.append(_params(c, geom))
        s["f"] = [f.clone() for f in s["f0"]]
        s["plan"] = tnlm.BatchPlan(s["geoms"], s["ys"], s["f"], params)
        return s
    if kind == "project":
        geom = _geom(case)
        _, truth = _phantom(case, geom, seed)
        s["vol"] = truth + _noise(truth.shape, _gen(seed + 1), 0.002)
    else:
        geom, s["y"], f0 = _recon_inputs(case, seed)
        s["f0"] = f0
        if kind in ("recon", "energy"):
            s["params"] = _params(case, geom)
    s["geom"] = tnlm.tnlm_create_geometry(geom)
    return s


# --------------------------------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------------------------------

_RECON = {"fp32": "tnlm_reconstruct", "bf16": "tnlm_reconstruct_bf16", "fp16": "tnlm_reconstruct_fp16"}
_SWEEP = {"fp32": "tnlm_gauss_jacobi", "bf16": "tnlm_gauss_jacobi_bf16", "fp16": "tnlm_gauss_jacobi_fp16"}
_ENHANCE = {"fp32": "tnlm_enhance", "bf16": "tnlm_enhance_bf16", "fp16": "tnlm_enhance_fp16"}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "recon":
        return getattr(tnlm, _RECON[case["dtype"]])(s["geom"], s["y"], s["f0"].clone(), s["params"])[0]
    if kind == "project":
        return tnlm.tnlm_project(s["geom"], s["vol"])
    if kind == "backproject":
        return tnlm.tnlm_backproject(s["geom"], s["y"])
    if kind == "sweep":
        g = s["g"]
        return getattr(tnlm, _SWEEP[case["dtype"]])(g, g, g, case["d"], case["M"], case["h"], 1.0, clip=1)
    if kind == "enhance":
        return getattr(tnlm, _ENHANCE[case["dtype"]])(s["g"], s["params"])
    if kind == "energy":
        f = s["f0"].detach().requires_grad_()
        E = tnlm.TNLMEnergy.apply(f, s["geom"], s["y"], f if case["through"] else f.detach(), s["params"])
        E.backward()
        return {"energy": E.detach().float(), "grad": f.grad}  # the kernels work in FP32: so does the loss
    if kind == "cgls":
        return tnlm.tnlm_cgls(s["geom"], s["y"], torch.zeros_like(s["f0"]), case["n_iter"])[0]
    if kind == "fdk":
        return tnlm.tnlm_fdk(s["geom"], s["y"])
    if kind == "batch":
        for f, f0 in zip(s["f"], s["f0"]):
            f.copy_(f0)
        s["plan"].run(case["iterations"])
        return s["f"]
    raise ValueError(kind)


# --------------------------------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------------------------------


def _nvox(case):
    return case["np"] * case["nx"] * case["ny"] * case["nz"]


def _npix(case):
    return sum(_views(case)) * case["nu"] * case["nv"]


def _ray_cells(case):
    """Voxels crossed by all rays: a ray through the field crosses about 4 / pi of nx + ny over 2 cells per axis."""
    return _npix(case) * (2 / math.pi) * (case["nx"] + case["ny"])


def _pairs(case, directions=2):
    s = 2 * case["M"] + 1
    valid = 1.0
    for n in (case["nx"], case["ny"], case["nz"]):
        valid *= max(1.0, s - case["M"] * (case["M"] + 1) / n)
    return _nvox(case) * directions * valid


def _pair_flops(case):
    # separable patch distance: the difference and square, then 2d additions on each axis; weight and two sums
    return 2 + 6 * case["d"] + 6


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [work(c) for c in _batch_cases(case)]
        return {k: case["iterations"] * sum(x[k] for x in w) for k in ("bytes", "flops")}
    size = 4 if case.get("dtype", "fp32") == "fp32" else 2
    vox = _nvox(case)
    if kind in ("sweep", "enhance"):
        n = case.get("n_outer", 1)
        return {"bytes": 2 * size * vox * n, "flops": n * _pairs(case) * _pair_flops(case)}
    pix, cells = _npix(case), _ray_cells(case)
    if kind in ("project", "backproject"):
        return {"bytes": 4 * (vox + pix), "flops": 2 * cells}
    if kind == "recon":
        return {"bytes": case["n_outer"] * size * (2 * vox + pix),
                "flops": case["n_outer"] * (4 * cells + _pairs(case) * _pair_flops(case))}
    if kind == "energy":
        f = 4 * cells + _pairs(case) * (_pair_flops(case) + 2)
        if case["through"]:  # the patch adjoint: a box sum and two differences per pair and direction
            f += _pairs(case, 1) * (_pair_flops(case) + 6 * case["d"] + 8)
        return {"bytes": 4 * (2 * vox + pix), "flops": f}
    if kind == "cgls":
        n = case["n_iter"] + 1
        return {"bytes": 4 * n * (4 * vox + 2 * pix), "flops": 4 * n * cells}
    if kind == "fdk":
        return {"bytes": 4 * (vox + pix), "flops": pix * case["nu"] + 20 * vox * case["views"]}
    raise ValueError(kind)


def _cost(case):
    """A figure that grows with a pass's time, for keeping drawn cases below the largest listed one."""
    w = work(case)
    direct = case.get("d") in (0, 3)  # patch sums without the separable form
    return w["flops"] * (8 if direct else 1) + 50 * w["bytes"]


# --------------------------------------------------------------------------------------------------
# the same in FP64
# --------------------------------------------------------------------------------------------------


class _Rays:
    """The rays of every view in FP64: the xy cells each detector column crosses, and the z range of each row."""

    def __init__(self, geom):
        self.g = geom
        f8 = dict(device=DEV, dtype=torch.float64)
        self.u = (torch.arange(geom["nu"], **f8) - 0.5 * (geom["nu"] - 1)) * geom["du"] + geom["u_off"]
        self.v = (torch.arange(geom["nv"], **f8) - 0.5 * (geom["nv"] - 1)) * geom["dv"] + geom["v_off"]
        self.len = torch.sqrt(geom["sdd"] ** 2 + self.u[None, :] ** 2 + self.v[:, None] ** 2)
        self.owner = np.repeat(np.arange(len(geom["nviews"])), geom["nviews"])

    def _axis(self, S, D, n, step, centre):
        """Crossing parameters of the n + 1 planes of one axis, and the parameter range inside them."""
        X0 = (S - (centre - 0.5 * n * step)) / step
        G = D / step
        flat = G == 0
        a = (torch.arange(n + 1, device=DEV, dtype=torch.float64)[None, :] - X0) / torch.where(flat, 1.0, G)[:, None]
        a = torch.where(flat[:, None], 2.0, a)
        inside = 1.0 if 0 <= X0 < n else -1.0
        lo = torch.where(flat, 0.0, torch.minimum(a[:, 0], a[:, -1]))
        hi = torch.where(flat, inside, torch.maximum(a[:, 0], a[:, -1]))
        return X0, G, a, lo, hi

    def columns(self, vg):
        """(alpha [nu, K + 1], cell [nu, K]) of view vg: the segments of each detector column in the xy plane."""
        g = self.g
        c, s = math.cos(g["angles"][vg]), math.sin(g["angles"][vg])
        Sx, Sy = g["sad"] * c, g["sad"] * s
        Dx, Dy = -g["sdd"] * c - self.u * s, -g["sdd"] * s + self.u * c
        X0, GX, ax, lx, hx = self._axis(Sx, Dx, g["nx"], g["dx"], g["cx"])
        Y0, GY, ay, ly, hy = self._axis(Sy, Dy, g["ny"], g["dy"], g["cy"])
        lo = torch.clamp(torch.maximum(lx, ly), 0.0, 1.0)
        hi = torch.clamp(torch.maximum(torch.minimum(hx, hy), lo), 0.0, 1.0)
        al = torch.cat([ax, ay, lo[:, None], hi[:, None]], 1)
        al = torch.sort(torch.minimum(torch.maximum(al, lo[:, None]), hi[:, None]), 1).values
        mid = 0.5 * (al[:, 1:] + al[:, :-1])
        ix = torch.clamp(torch.floor(X0 + mid * GX[:, None]), 0, g["nx"] - 1).long()
        iy = torch.clamp(torch.floor(Y0 + mid * GY[:, None]), 0, g["ny"] - 1).long()
        return al, iy * g["nx"] + ix

    def _ends(self, al, v, side):
        """z cell and offset in it at one end (0 near, 1 far) of every segment of rows v, clipped to the volume."""
        g = self.g
        a = al[:, side:al.shape[1] - 1 + side]
        z = (a[None] * v[:, None, None] - (g["cz"] - 0.5 * g["nz"] * g["dz"])) / g["dz"]
        z = z.clamp_(0.0, float(g["nz"]))
        k = torch.floor(z).clamp_(max=g["nz"] - 1.0)
        return k.long(), z - k

    def _rows(self):
        g = self.g
        n = max(1, int(3e7 / (g["nu"] * (g["nx"] + g["ny"]))))
        level = self.v == 0
        for rows in torch.split(torch.nonzero(~level).flatten(), n):
            yield rows, False
        if bool(level.any()):
            yield torch.nonzero(level).flatten(), True

    def _level(self, al):
        """Rows in the plane z = 0: their z cell (None outside the volume) and the segment lengths."""
        g = self.g
        z = -(g["cz"] - 0.5 * g["nz"] * g["dz"]) / g["dz"]
        return (int(math.floor(z)) if 0 <= z < g["nz"] else None), al[:, 1:] - al[:, :-1]

    def project(self, vol):
        g = self.g
        nz, out = g["nz"], torch.zeros((len(g["angles"]), g["nv"], g["nu"]), device=DEV, dtype=torch.float64)
        for ph in range(vol.shape[0]):
            f = vol[ph].double().reshape(nz, -1).t().contiguous()  # [cell][z]
            C = torch.cat([torch.zeros_like(f[:, :1]), torch.cumsum(f, 1)], 1).flatten()
            f = f.flatten()
            for vg in np.flatnonzero(self.owner == ph):
                al, cell = self.columns(int(vg))
                for rows, level in self._rows():
                    if level:
                        k, seg = self._level(al)
                        if k is not None:
                            out[vg, rows] = (f[cell * nz + k] * seg).sum(1)
                        continue
                    v = self.v[rows]
                    acc = 0.0
                    for side, sign in ((1, 1.0), (0, -1.0)):
                        k, t = self._ends(al, v, side)
                        acc = acc + sign * (C[cell * (nz + 1) + k] + t * f[cell * nz + k])
                    out[vg, rows] = acc.sum(2) * (g["dz"] / v)[:, None]
                out[vg] *= self.len
        return out

    def backproject(self, proj):
        g = self.g
        nz, ncell = g["nz"], g["nx"] * g["ny"]
        out = torch.zeros((len(g["nviews"]), nz, ncell), device=DEV, dtype=torch.float64)
        for ph in range(out.shape[0]):
            whole = torch.zeros(ncell * (nz + 1), device=DEV, dtype=torch.float64)  # adjoint of the z prefix sums
            part = torch.zeros(ncell * nz, device=DEV, dtype=torch.float64)         # adjoint of the cells themselves
            for vg in np.flatnonzero(self.owner == ph):
                al, cell = self.columns(int(vg))
                r = proj[vg].double() * self.len
                for rows, level in self._rows():
                    if level:
                        k, seg = self._level(al)
                        if k is not None:
                            part.index_add_(0, (cell * nz + k).flatten(), (seg * r[rows].sum(0)[:, None]).flatten())
                        continue
                    v = self.v[rows]
                    w = r[rows] * (g["dz"] / v)[:, None]
                    for side, sign in ((1, 1.0), (0, -1.0)):
                        k, t = self._ends(al, v, side)
                        ws = (sign * w)[:, :, None].expand_as(t)
                        whole.index_add_(0, (cell * (nz + 1) + k).flatten(), ws.flatten())
                        part.index_add_(0, (cell * nz + k).flatten(), (ws * t).flatten())
            # the prefix sum at k holds the cells below k
            suffix = torch.flip(torch.cumsum(torch.flip(whole.view(ncell, nz + 1), [1]), 1), [1])
            out[ph] = (suffix[:, 1:] + part.view(ncell, nz)).t()
        return out.view(out.shape[0], nz, g["ny"], g["nx"])


def _pad(a, r):
    return torch.nn.functional.pad(a[None, None], (r,) * 6, mode="replicate")[0, 0] if r else a


def _fold(a, r):
    """The adjoint of _pad."""
    for ax in range(3 if r else 0):
        n = a.shape[ax] - 2 * r
        b = a.narrow(ax, r, n).clone()
        b.narrow(ax, 0, 1).add_(a.narrow(ax, 0, r).sum(ax, keepdim=True))
        b.narrow(ax, n - 1, 1).add_(a.narrow(ax, r + n, r).sum(ax, keepdim=True))
        a = b
    return a


def _box(s, d):
    """Sums over (2d + 1)^3 neighbourhoods, each axis shrinking by 2d."""
    for ax in range(3 if d else 0):
        n = s.shape[ax] - 2 * d
        t = s.narrow(ax, 0, n).clone()
        for k in range(1, 2 * d + 1):
            t += s.narrow(ax, k, n)
        s = t
    return s


class _Pair:
    """Window offsets of phase image a toward phase image b: patch distances and index ranges."""

    def __init__(self, a, b, d, M):
        self.d, self.M, self.shape = d, M, a.shape
        self.ap, self.bp = _pad(a, d), _pad(b, d + M)
        self.base = self.distance((0, 0, 0))
        self.offsets = [(z, y, x) for z in range(-M, M + 1) for y in range(-M, M + 1) for x in range(-M, M + 1)
                        if abs(z) < a.shape[0] and abs(y) < a.shape[1] and abs(x) < a.shape[2]]

    def neighbour(self, o):
        return tuple(slice(self.M + k, self.M + k + n) for k, n in zip(o, self.ap.shape))

    def distance(self, o):
        return _box((self.ap - self.bp[self.neighbour(o)]) ** 2, self.d)

    def inside(self, o):
        """Slices of the voxels whose candidate is in the volume, and of those candidates."""
        own = tuple(slice(max(0, -k), min(n, n - k)) for k, n in zip(o, self.shape))
        return own, tuple(slice(s.start + k, s.stop + k) for s, k in zip(own, o))

    def weight(self, o, c):
        """Unnormalised weights relative to the centre's (window offset 0)."""
        return torch.exp((self.base - self.distance(o)) * c)


def _mean_of(a, b, vals, d, M, h):
    """sum w vals(x + o) over the window, weights of a toward b normalised."""
    p = _Pair(a, b, d, M)
    N, Z = torch.zeros_like(a), torch.zeros_like(a)
    for o in p.offsets:
        w = p.weight(o, 1.0 / (2.0 * h * h))
        own, cand = p.inside(o)
        N[own] += w[own] * vals[cand]
        Z[own] += w[own]
    return N / Z


def _sweep64(g, d, M, h, fid=None, clip=True):
    """One Gauss-Jacobi sweep of the FP64 images g (weights and values from g, fidelity image fid), mu = 1."""
    fid = g if fid is None else fid
    n = g.shape[0]
    out = torch.stack([(fid[i] + _mean_of(g[i], g[(i + 1) % n], g[(i + 1) % n], d, M, h)
                        + _mean_of(g[i], g[i - 1], g[i - 1], d, M, h)) / 3.0 for i in range(n)])
    return out.clamp_(min=0.0) if clip else out


def _energy64(geom, y, f, d, M, h, through):
    """E and its gradient in f (mu = 1), weights from f itself; `through`: the weights differentiated too."""
    R = _Rays(geom)
    r = R.project(f) - y.double()
    E = 0.5 * float((r * r).sum())
    grad = R.backproject(r)
    n, c = f.shape[0], 1.0 / (2.0 * h * h)
    for i in range(n):
        j = (i + 1) % n
        fi, fj = f[i], f[j]
        p = _Pair(fi, fj, d, M)
        Z, Q = torch.zeros_like(fi), torch.zeros_like(fi)
        for o in p.offsets:
            w = p.weight(o, c)
            own, cand = p.inside(o)
            Z[own] += w[own]
            Q[own] += w[own] * (fi[own] - fj[cand]) ** 2
        Q /= Z
        E += 0.5 * float(Q.sum())
        ga, gb = torch.zeros_like(p.ap), torch.zeros_like(p.bp)
        for o in p.offsets:
            own, cand = p.inside(o)
            w = (p.weight(o, c) / Z)[own]
            df = fi[own] - fj[cand]
            grad[i][own] += w * df
            grad[j][cand] -= w * df
            if through:
                G = torch.zeros(tuple(k + 4 * d for k in fi.shape), device=DEV, dtype=torch.float64)
                G[tuple(slice(s.start + 2 * d, s.stop + 2 * d) for s in own)] = 0.5 * c * w * (Q[own] - df * df)
                nb = p.neighbour(o)
                v = 2.0 * _box(G, d) * (p.ap - p.bp[nb])
                ga += v
                gb[nb] -= v
        if through:
            grad[i] += _fold(ga, d)
            grad[j] += _fold(gb, d + M)
    return E, grad


def _fdk64(geom, y):
    R = _Rays(geom)
    nu, du = geom["nu"], geom["du"]
    m = torch.arange(nu, device=DEV, dtype=torch.float64)
    m = m[:, None] - m[None, :]
    H = torch.where(m == 0, 1.0 / (4 * du * du),
                    torch.where(m.long() % 2 == 0, 0.0, -1.0 / (math.pi * du * torch.where(m == 0, 1.0, m)) ** 2))
    F = torch.matmul(y.double() * geom["sdd"] / R.len, H) * du
    F = torch.nn.functional.pad(F, (1, 1, 1, 1))  # zero outside the detector

    def centres(n, step, c):
        return (torch.arange(n, device=DEV, dtype=torch.float64) - 0.5 * (n - 1)) * step + c

    z, yy, x = torch.meshgrid(centres(geom["nz"], geom["dz"], geom["cz"]), centres(geom["ny"], geom["dy"], geom["cy"]),
                              centres(geom["nx"], geom["dx"], geom["cx"]), indexing="ij")
    out = torch.zeros((len(geom["nviews"]),) + tuple(x.shape), device=DEV, dtype=torch.float64)
    for vg, th in enumerate(geom["angles"]):
        ph = int(R.owner[vg])
        c, s = math.cos(th), math.sin(th)
        U = geom["sad"] - (x * c + yy * s)
        fu = (geom["sdd"] * (yy * c - x * s) / U - geom["u_off"]) / du + 0.5 * (nu - 1) + 1
        fv = (geom["sdd"] * z / U - geom["v_off"]) / geom["dv"] + 0.5 * (geom["nv"] - 1) + 1
        fu, fv = fu.clamp_(0, nu + 1 - 1e-9), fv.clamp_(0, geom["nv"] + 1 - 1e-9)
        iu, iv = torch.floor(fu), torch.floor(fv)
        au, av = fu - iu, fv - iv
        at = (iv * (nu + 2) + iu).long()
        P = F[vg].flatten()
        val = (1 - av) * ((1 - au) * P[at] + au * P[at + 1]) + av * ((1 - au) * P[at + nu + 2] + au * P[at + nu + 3])
        out[ph] += math.pi / float(geom["nviews"][ph]) * geom["sad"] * geom["sdd"] / (U * U) * val
    return out


def _cgls64(geom, y, n_iter):
    R = _Rays(geom)
    n = len(geom["nviews"])
    seg = torch.as_tensor(R.owner, device=DEV)

    def norms(t):
        q = (t * t).flatten(1).sum(1)
        return q if t.shape[0] == n else torch.zeros(n, device=DEV, dtype=torch.float64).index_add_(0, seg, q)

    r = y.double()
    p = R.backproject(r)
    x = torch.zeros_like(p)
    gam = norms(p)
    for it in range(n_iter):
        q = R.project(p)
        # phase by phase; the rows of a projection set go by the phase that owns the view
        a = gam / torch.zeros(n, device=DEV, dtype=torch.float64).index_add_(0, seg, (q * q).flatten(1).sum(1))
        x += a[:, None, None, None] * p
        if it + 1 == n_iter:
            break
        r = r - a[seg][:, None, None] * q
        s = R.backproject(r)
        new = (s * s).flatten(1).sum(1)
        p = s + (new / gam)[:, None, None, None] * p
        gam = new
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return None
    if kind in ("sweep", "enhance"):
        if _pairs(case) * case.get("n_outer", 1) * (1 + case["d"]) > 1.2e11:
            return None
        g = _streaked(case, seed).double()
        f = _sweep64(g, case["d"], case["M"], case["h"])
        for _ in range(case.get("n_outer", 1) - 1):
            f = _sweep64(f, case["d"], case["M"], case["h"], fid=g)
        return f
    if kind != "fdk":
        passes = {"recon": 4 * case.get("n_outer", 1), "energy": 4, "cgls": 4 * case.get("n_iter", 1)}.get(kind, 3)
        if passes * _ray_cells(case) > 6e10:
            return None
    if kind == "project":
        geom = _geom(case)
        _, truth = _phantom(case, geom, seed)
        return _Rays(geom).project(truth + _noise(truth.shape, _gen(seed + 1), 0.002))
    geom, y, f0 = _recon_inputs(case, seed)
    if kind == "backproject":
        return _Rays(geom).backproject(y)
    if kind == "fdk":
        return _fdk64(geom, y)
    if kind == "cgls":
        return _cgls64(geom, y, case["n_iter"])
    if kind == "energy":
        E, grad = _energy64(geom, y, f0.double(), case["d"], case["M"], case["h"], case["through"])
        return {"energy": E, "grad": grad}
    R, f, tau = _Rays(geom), f0.double(), float(np.float32(_tau(geom)))
    for _ in range(case["n_outer"]):
        g = f - tau * R.backproject(R.project(f) - y.double())
        f = _sweep64(g, case["d"], case["M"], case["h"])
    return f
