"""Performance cases: the traces and set-up calls a user of the library makes.

A case is a dict of plain values.  ``prepare`` makes what the user's program
has in hand (extinction fields, heights, suns, cameras, scenes on the device,
a network, a captured batch), ``run`` makes one pass through the public entry
points, ``work`` states the bytes and operations a pass cannot do without, and
``exact`` gives the outputs that have a value independent of random draws.

Fields are seeded stand-ins for cloud-resolving model output: Gaussian blobs
over clear sky, or shallow cumulus over a 12.8 x 12.8 x 4 km domain (20 %
cover from a band-limited k^-8/3 field, cloud base 0.8 km, tops to 2.8 km,
log-normal liquid water, 10 um droplets).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1902_01137_gb300 as m

DEVICE = "cuda"
LX, LZ = 12.8, 4.0          # km: cumulus domain width (x) and height

# Mean events of one path (measured with the library's event counters on the
# 512 x 512 x 160 cumulus and the 64 x 64 x 32 blob field): leaves crossed,
# tentative collisions, scattering or ground events, sun rays included.
EVENTS = {
    ("image", "cumulus", "pyramid"): (163.0, 27.0, 15.0),
    ("image", "cumulus", "octree"): (77.0, 39.0, 15.0),
    ("image", "blobs", "pyramid"): (107.0, 36.0, 19.0),
    ("image", "blobs", "octree"): (60.0, 45.0, 19.0),
    ("flux", "cumulus", "pyramid"): (128.0, 22.0, 11.0),
    ("flux", "cumulus", "octree"): (43.0, 37.0, 11.0),
    ("flux", "blobs", "pyramid"): (100.0, 34.0, 17.0),
    ("flux", "blobs", "octree"): (55.0, 42.0, 17.0),
}
# Floating-point operations of one event: a leaf crossed (three face
# distances, the exit point, the optical depth spent), a tentative collision
# (the point, the test, the next optical depth), a scattering or ground event
# (phase function, new direction, two ray starts).
OPS = (30.0, 20.0, 150.0)


# --------------------------------------------------------------------------
# Cases
# --------------------------------------------------------------------------
def listed():
    return [
        # A live preview inside another program's memory budget: a few paths
        # per pixel of a small coarse scene, straight into the caller's device
        # buffers.  The smallest call there is.
        dict(name="frame_64x48x4_blobs", kind="frame", field="blobs", nx=64, ny=64, nz=32, storage="f32",
             grid="pyramid", finest=0, width=64, height=48, spp=4, zenith=30.0),
        # The plain method's first picture: a 64 x 64 image at 16 paths a pixel
        # of the 100 m blob field.
        dict(name="image_64x64x16_blobs", kind="image", field="blobs", nx=64, ny=64, nz=32, storage="f32",
             grid="pyramid", finest=0, width=64, height=64, spp=16, zenith=30.0, sun="ratio", phase="hg"),
        # The rendering of a whole cloud field at production quality: the
        # 512 x 512 x 160 cumulus, 1024 x 1024 pixels at 64 paths each.
        dict(name="image_1024x1024x64_cumulus", kind="image", field="cumulus", nx=512, ny=512, nz=160, storage="f32",
             grid="pyramid", finest=0, width=1024, height=1024, spp=64, zenith=60.0, sun="ratio", phase="hg"),
        # The same field over the 2^L octree, at an odd picture size and at the
        # sampling of a draft.
        dict(name="image_1023x767x15_octree", kind="image", field="cumulus", nx=512, ny=512, nz=160, storage="f32",
             grid="octree", finest=1, width=1023, height=767, spp=15, zenith=60.0, sun="ratio", phase="hg"),
        # Molecular (Rayleigh) clear air and decomposition tracking of the sun
        # rays over half-precision voxels, on a ragged field.
        dict(name="image_500x301x16_rayleigh", kind="image", field="cumulus", nx=250, ny=250, nz=70, storage="bf16",
             grid="octree", finest=0, width=500, height=301, spp=16, zenith=40.0, sun="decomp", phase="rayleigh"),
        # Ground irradiance of the cloud field, direct and diffuse.
        dict(name="flux_16M_cumulus", kind="flux", field="cumulus", nx=512, ny=512, nz=160, storage="f32",
             grid="pyramid", finest=0, paths=1 << 24, terrain=0, zenith=60.0, sun="ratio", phase="hg"),
        # Ground irradiance over a mountain relief, half-precision voxels.
        dict(name="flux_4M_terrain", kind="flux", field="cumulus", nx=256, ny=256, nz=80, storage="bf16",
             grid="octree", finest=1, paths=4_000_037, terrain=4096, zenith=60.0, sun="ratio", phase="hg"),
        # A study over many fields, gas bands and suns in one launch, with
        # sensitivities to g: uneven fields and path counts.
        dict(name="batch_12_fields", kind="batch", fields=12, max_nx=512, storage="f32", grid="octree", finest=1,
             paths=30_000_000, dalpha=False),
        # The same kind of study as a captured plan that is replayed with new
        # seeds, with the sensitivity to droplet absorption too.
        dict(name="plan_4_fields", kind="plan", fields=4, max_nx=256, storage="f32", grid="pyramid", finest=0,
             paths=3_000_000, dalpha=True),
        # An image traced with a trained (here: fixed) scattering proposal.
        dict(name="learned_512x512x16", kind="learned", field="cumulus", nx=512, ny=512, nz=160, storage="f32",
             grid="pyramid", finest=0, width=512, height=512, spp=16, zenith=60.0, n_learned=8),
        # Training a proposal from its initial weights on one batch of ground
        # flux paths (tensor-core gradients, four optimiser steps).
        dict(name="train_flux_500k", kind="train", field="cumulus", nx=256, ny=256, nz=80, storage="f32",
             grid="pyramid", finest=0, paths=500_000, zenith=60.0, n_learned=2, steps=4),
        # A new time step of a simulation arrives on the device: bricks, both
        # majorant grids and a quick look at it in single scattering.
        dict(name="newfield_1024x1024x160", kind="newfield", field="cumulus", nx=1024, ny=1024, nz=160,
             storage="f32", grid="octree", finest=1, width=128, height=96, spp=2, zenith=60.0),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "image", "image", "flux", "flux", "batch", "plan", "learned", "train", "newfield"])
    c = {"kind": kind, "storage": rng.choice(["f32", "f32", "bf16"]), "grid": rng.choice(["pyramid", "octree"])}
    c["finest"] = rng.choice([0, 1]) if c["grid"] == "octree" else 0
    if kind in ("batch", "plan"):
        c.update(fields=rng.randint(2, 12), max_nx=rng.choice([128, 256, 512]), paths=_logint(rng, 3e5, 3e7),
                 dalpha=rng.choice([False, True]))
        return c
    if kind == "frame" or (kind in ("image", "flux") and rng.random() < 0.25):
        c.update(field="blobs", nx=rng.randint(40, 96), ny=rng.randint(40, 96), nz=rng.randint(20, 48))
    else:
        nx = _logint(rng, 96, 1024 if kind == "newfield" else 640)
        c.update(field="cumulus", nx=nx, ny=max(64, nx + rng.choice([0, 0, -3, 5, nx // 3])), nz=rng.randint(40, 160))
    c["zenith"] = round(rng.uniform(0.0, 70.0), 2)
    if kind in ("image", "flux"):
        c["sun"] = rng.choice(["ratio", "ratio", "ratio", "delta", "decomp"])
        c["phase"] = rng.choice(["hg", "hg", "hg", "rayleigh"])
    if kind == "frame":
        c.update(width=rng.randint(20, 160), height=rng.randint(20, 120), spp=rng.randint(1, 12))
    elif kind == "newfield":
        c.update(width=rng.randint(32, 160), height=rng.randint(32, 120), spp=rng.randint(1, 3))
    elif kind in ("image", "learned"):
        w = _logint(rng, 48, 1100)
        h = max(32, int(w * rng.uniform(0.5, 1.0)))
        most = 4_000_000 if kind == "learned" else 24_000_000
        c.update(width=w, height=h, spp=max(1, min(_logint(rng, 2, 70), most // (w * h))))
        if kind == "learned":
            c["n_learned"] = rng.randint(1, 8)
    elif kind == "flux":
        c.update(paths=_logint(rng, 4e4, 1.6e7), terrain=rng.choice([0, 0, 0, 256, 1000, 4096]))
    else:
        c.update(paths=_logint(rng, 3e4, 5e5), n_learned=2, steps=rng.randint(1, 4))
    return c


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    return g


def _randc(shape, g):
    return torch.complex(torch.randn(shape, generator=g, device=DEVICE), torch.randn(shape, generator=g, device=DEVICE))


def _freq(k):
    return torch.arange(-k, k + 1, device=DEVICE)


def _cumulus(nx, ny, nz, seed):
    """Extinction [km^-1] of a shallow cumulus field, [z][y][x]."""
    g = _gen(seed)
    kx, ky = min(48, (nx - 1) // 2), min(48, (ny - 1) // 2)
    KY, KX = torch.meshgrid(_freq(ky), _freq(kx), indexing="ij")
    kk = (KX.double() ** 2 + KY.double() ** 2).sqrt()
    amp = torch.where(kk > 0, kk.clamp_min(1e-12) ** (-4.0 / 3.0), torch.zeros_like(kk)).float()
    F = torch.zeros((ny, nx), dtype=torch.complex64, device=DEVICE)
    F[KY % ny, KX % nx] = _randc(KX.shape, g) * amp
    f = torch.fft.ifft2(F).real
    f = (f - f.mean()) / f.std()
    thr = f.flatten().kthvalue(max(1, int(0.8 * f.numel()))).values
    top = torch.where(f > thr, 0.8 + 2.0 * (f - thr) / (f.max() - thr), torch.full_like(f, 0.8))
    k3, kz = min(24, (min(nx, ny) - 1) // 2), min(6, (nz - 1) // 2)
    KZ, KY, KX = torch.meshgrid(_freq(kz), _freq(k3), _freq(k3), indexing="ij")
    kk = (KX.double() ** 2 + KY.double() ** 2 + (KZ.double() * 3.2) ** 2).sqrt()
    amp = torch.where(kk > 0, kk.clamp_min(1e-12) ** (-11.0 / 6.0), torch.zeros_like(kk)).float()
    F = torch.zeros((nz, ny, nx), dtype=torch.complex64, device=DEVICE)
    F[KZ % nz, KY % ny, KX % nx] = _randc(KX.shape, g) * amp
    g3 = torch.fft.ifftn(F).real
    del F
    g3 = (g3 - g3.mean()) / g3.std()
    zc = (torch.arange(nz, device=DEVICE) + 0.5) * (LZ / nz)
    incloud = (zc[:, None, None] >= 0.8) & (zc[:, None, None] < top[None])
    lwc = 0.3 * torch.exp(0.6 * g3)                        # g m^-3, median 0.3
    return torch.where(incloud, 150.0 * lwc, torch.zeros((), device=DEVICE)).add_(0.01).contiguous()


def _blobs(nx, ny, nz, seed):
    """Extinction [km^-1] of three Gaussian blobs (peak 50) over clear sky, 100 m voxels, [z][y][x]."""
    r = torch.rand(12, generator=_gen(seed), device=DEVICE)
    x, y, z = (((torch.arange(n, device=DEVICE) + 0.5) * 0.1) for n in (nx, ny, nz))
    Lx, Ly, Lz = nx * 0.1, ny * 0.1, nz * 0.1
    k = torch.full((nz, ny, nx), 0.01, device=DEVICE)
    for b in range(3):
        dx = x - r[4 * b] * Lx
        dy = y - r[4 * b + 1] * Ly
        dx = dx - Lx * torch.round(dx / Lx)
        dy = dy - Ly * torch.round(dy / Ly)
        dz = z - Lz * (0.3 + 0.35 * r[4 * b + 2])
        s = 0.4 + 0.4 * r[4 * b + 3]
        k += 50.0 * torch.exp(-(dx[None, None, :] ** 2 + dy[None, :, None] ** 2) / (2 * s * s)
                              - dz[:, None, None] ** 2 / 0.18)
    return k


def _heights(n, seed, relief=0.3):
    """Periodic fractal relief, n x n heights in [0, relief] km."""
    k = torch.fft.fftfreq(n, device=DEVICE) * n
    kk = (k[None, :] ** 2 + k[:, None] ** 2).sqrt()
    amp = torch.where(kk > 0, kk.clamp_min(1e-12) ** -1.6, torch.zeros_like(kk))
    f = torch.fft.ifft2(_randc((n, n), _gen(seed)) * amp).real
    f = (f - f.min()) / (f.max() - f.min())
    return (f * relief).clamp_(0.0, relief).contiguous()


def _field(case, seed):
    """(extinction on the device, dx, dy, dz, optical constants)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["field"] == "blobs":
        return _blobs(nx, ny, nz, seed), 0.1, 0.1, 0.1, dict(ssa_cloud=1.0, g=0.85, albedo=0.2)
    return _cumulus(nx, ny, nz, seed), LX / nx, LX / nx, LZ / nz, dict(ssa_cloud=0.999, g=0.86, albedo=0.1)


class _Camera:
    """Pinhole camera 10 km above the domain, looking straight down on its whole width."""

    def __init__(self, k, dx, dy, dz, width, height):
        nz, ny, nx = k.shape
        z = nz * dz + 10.0
        self.pos, self.target, self.up = (0.5 * nx * dx, 0.5 * ny * dy, z), (0.5 * nx * dx, 0.5 * ny * dy, 0.0), (0.0, 1.0, 0.0)
        self.fov_deg = 2.0 * math.degrees(math.atan(0.5 * nx * dx / z))
        self.width, self.height = width, height

    def desc(self):
        d = m.CameraDesc()
        for i in range(3):
            d.pos[i], d.target[i], d.up[i] = self.pos[i], self.target[i], self.up[i]
        d.fov_deg, d.width, d.height = self.fov_deg, self.width, self.height
        return d


class _State:
    """What the user's program keeps; releases the library's objects when it goes."""

    def __init__(self, case, seed):
        self.case, self.seed = case, seed
        self.ctx, self.scenes, self.prop, self.plan = m.Context(0), [], None, None

    def scene(self, k, dx, dy, dz, const, storage, zenith, azimuth=0.0, levels=3):
        sc = m.Scene(self.ctx, k, dx, dy, dz, k_clear=0.01, ssa_clear=0.9, ssa_cloud=const["ssa_cloud"], g=const["g"],
                     storage=m.MCRT_STORAGE_BF16 if storage == "bf16" else m.MCRT_STORAGE_F32, levels=levels,
                     albedo=const["albedo"], sun_zenith_deg=zenith, sun_azimuth_deg=azimuth)
        self.scenes.append(sc)
        return sc

    def __del__(self):
        if self.plan is not None:
            self.plan.close()
        if self.prop is not None:
            self.prop.close()
        for sc in self.scenes:
            sc.close()
        self.ctx.close()


def _opts(case):
    kw = dict(grid=m.MCRT_GRID_OCTREE if case["grid"] == "octree" else m.MCRT_GRID_PYRAMID,
              finest_level=case["finest"])
    if case.get("sun") == "delta":
        kw["sun_mode"] = m.MCRT_SUN_DELTA
    elif case.get("sun") == "decomp":
        kw["sun_mode"] = m.MCRT_SUN_DECOMP
    return kw


def _study(case, seed):
    """Fields, suns and gas bands of a batch: [(nx, nz, zenith, azimuth, [k_gas], paths per band)]."""
    shape, r = np.random.default_rng(case["fields"]), np.random.default_rng(seed)
    sizes = [s for s in ((64, 32), (128, 40), (256, 80), (512, 160)) if s[0] <= case["max_nx"]]
    share = np.exp(shape.uniform(0.0, math.log(100.0), case["fields"]))
    share *= case["paths"] / share.sum()
    out = []
    for i in range(case["fields"]):
        nx, nz = sizes[i % len(sizes)]
        nb = int(shape.integers(1, 17))
        out.append((nx, nz, float(r.uniform(0.0, 75.0)), float(r.uniform(0.0, 360.0)),
                    [float(v) for v in np.exp(math.log(1e-3) + 2.0 * r.standard_normal(nb))],
                    max(1, int(share[i] / nb))))
    return out


def prepare(case, seed):
    s = _State(case, seed)
    kind = case["kind"]
    if kind in ("batch", "plan"):
        items = []
        for i, (nx, nz, zen, azi, gas, n) in enumerate(_study(case, seed)):
            c = dict(field="cumulus", nx=nx, ny=nx, nz=nz)
            k, dx, dy, dz, const = _field(c, 1000 * seed + i)
            sc = s.scene(k, dx, dy, dz, const, case["storage"], zen, azi)
            if case["grid"] == "octree":
                sc.build_octree()
            items += [(sc, kg, zen, azi, n, (seed << 16) | (i << 8) | j) for j, kg in enumerate(gas)]
        s.items = items
        if kind == "plan":
            s.plan = m.BatchPlan(s.ctx, items, batch_dalpha=int(case["dalpha"]), **_opts(case))
            s.seeds = [(seed << 20) + 7 * i for i in range(len(items))]
        return s
    k, dx, dy, dz, const = _field(case, seed)
    if "width" in case:
        s.cam = _Camera(k, dx, dy, dz, case["width"], case["height"])
    if kind == "newfield":
        s.k, s.geometry, s.const = k, (dx, dy, dz), const
        return s
    sc = s.scene(k, dx, dy, dz, const, case["storage"], case["zenith"], levels=2 if case["field"] == "blobs" else 3)
    if case["grid"] == "octree":
        sc.build_octree()
    if case.get("phase") == "rayleigh":
        m.mcrt_scene_set_clear_sky_phase(s.ctx.h, sc.h, m.MCRT_PHASE_RAYLEIGH)
    if case.get("terrain"):
        sc.set_heightfield(_heights(case["terrain"], seed + 1), const["albedo"])
    if kind == "learned":
        s.prop = m.Proposal(s.ctx, seed=seed)
    if kind == "frame":
        s.mean = torch.empty((case["height"], case["width"]), dtype=torch.float64, device=DEVICE)
        s.se = torch.empty_like(s.mean)
        s.opts = m.Scene._opts(**_opts(case))
    return s


# --------------------------------------------------------------------------
# One pass
# --------------------------------------------------------------------------
def _out(r):
    return {"mean": r.mean, "se": r.se, "n": r.n.astype(np.int64)}


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "batch":
        return _out(m.trace_batch(s.ctx, s.items, batch_dalpha=int(case["dalpha"]), **_opts(case)))
    if kind == "plan":
        s.plan.set_seeds(s.seeds)
        r = s.plan.run()
        return {"mean": r.mean, "se": r.se}
    if kind == "newfield":
        sc = s.scene(s.k, *s.geometry, s.const, case["storage"], case["zenith"])
        if case["grid"] == "octree":
            sc.build_octree()
        out = _out(sc.trace_camera(s.cam, case["spp"], s.seed, max_order=1, **_opts(case)))
        out["majorants"] = [sc.majorants(level) for level in range(1, 4)]
        s.scenes.remove(sc)
        sc.close()
        return out
    sc = s.scenes[0]
    if kind == "frame":
        m.mcrt_trace_camera_noalloc(s.ctx.h, sc.h, s.cam.desc(), case["spp"], s.seed, s.opts, s.mean.data_ptr(),
                                    s.se.data_ptr())
        return {"mean": s.mean, "se": s.se}
    if kind == "image":
        return _out(sc.trace_camera(s.cam, case["spp"], s.seed, **_opts(case)))
    if kind == "flux":
        return _out(sc.trace_flux(case["paths"], s.seed, **_opts(case)))
    if kind == "learned":
        return _out(sc.trace_camera(s.cam, case["spp"], s.seed, proposal=s.prop, n_learned=case["n_learned"],
                                    mis_alpha=0.5, **_opts(case)))
    prop = m.Proposal(s.ctx, seed=s.seed)
    try:
        out = _out(sc.trace_flux(case["paths"], s.seed, proposal=prop, n_learned=case["n_learned"], mis_alpha=0.5,
                                 learn=1, batch_paths=case["paths"], train_steps=case["steps"], **_opts(case)))
        out["params"] = prop.params
    finally:
        prop.close()
    return out


# --------------------------------------------------------------------------
# What a pass cannot do without
# --------------------------------------------------------------------------
def _path_ops(sensor, field, grid):
    return sum(n * o for n, o in zip(EVENTS[(sensor, field, grid)], OPS))


def work(case):
    kind, size = case["kind"], 2 if case["storage"] == "bf16" else 4
    if kind in ("batch", "plan"):
        study = _study(case, 0)
        voxels = sum(nx * nx * nz for nx, nz, *_ in study)
        items = sum(len(gas) for *_, gas, _ in study)
        paths = sum(len(gas) * n for *_, gas, n in study)
        return {"bytes": size * voxels + 16 * 5 * items, "flops": paths * _path_ops("flux", "cumulus", case["grid"])}
    voxels = case["nx"] * case["ny"] * case["nz"]
    if "width" in case:
        cells, paths = case["width"] * case["height"], case["width"] * case["height"] * case["spp"]
    else:
        cells, paths = 3, case["paths"]
    sensor = "image" if "width" in case else "flux"
    flops = paths * _path_ops(sensor, case["field"], case["grid"])
    nbytes = size * voxels + 16 * cells
    if kind == "newfield":
        # the field read once, its bricks and both grids' maxima and minima written once
        nbytes += 4 * voxels + 2 * 4 * voxels / 8 * (8 / 7)
    if kind in ("learned", "train"):
        # the network on each learned vertex; forward 2 * 11,392 operations, training three times that and four passes
        vertices = 0.25 * paths * case["n_learned"]
        flops += vertices * 2 * 11392 * (1 + 3 * case.get("steps", 0))
    return {"bytes": nbytes, "flops": flops}


# --------------------------------------------------------------------------
# Outputs that do not depend on random draws
# --------------------------------------------------------------------------
def exact(case, seed):
    """The majorant levels of a new field: the largest extinction of each 8^L cell (of the stored values' bound)."""
    if case["kind"] != "newfield" or case["storage"] != "f32":
        return None      # Monte Carlo tallies: no value without the draws
    k = _field(case, seed)[0].double()[None, None]
    levels = []
    for _ in range(3):
        k = torch.nn.functional.pad(k, [v for n in reversed(k.shape[2:]) for v in (0, -n % 8)])
        k = torch.nn.functional.max_pool3d(k, 8)
        levels.append(k[0, 0].cpu().numpy())
    return {"mean": None, "se": None, "n": None, "majorants": levels}
