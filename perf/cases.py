"""Performance cases: the work a user of the library has it do, through its public Python entry points.

A case is a dict of plain values; `prepare` makes the inputs and the context a program holds before the call,
`run` makes one pass, `work` counts what a pass cannot do without, and `exact` gives the same outputs in 64 bits
with plain torch where that is possible.  Sizes follow the workloads of mc_inputs/workloads.py, the benchmark's
modes and the tests; `draw` gives more of the same ranges, odd sizes among them.
"""

import math
import os
import struct
import tempfile

import numpy as np
import torch

import paper_2201_13191_gb300 as mcx
from mc_inputs import default_table_path, kramers_spectrum, mono_spectrum, read_tables, table_response
from mc_inputs.meshes import assemble, cylinder_mesh
from mc_inputs.phantoms import NOMINAL_DENSITY, cylinder_variant_phantom, ellipsoid_params, tiny_phantom
from mc_inputs.tables import MAT_AL, MAT_WATER

DEV = "cuda:0"
WEIGHTS = os.path.join(os.path.dirname(mcx.__file__), "weights", "unet_c4_256.bin")
SPLIT = 10  # pseudo-particles per interaction (the library's default)


def listed():
    return [
        # The smallest call: a quick look at a coarse phantom; launches, copies and host time are all of it.
        dict(name="project_tiny", kind="project", phantom="tiny", nx=8, ny=8, nz=8, dv=4.0, kvp=0, sod=100.0,
             nu=8, nv=8, pu=8.0, angles=1, photons=20_000, step=0.5, primary=True),
        # One projection of a small scan: cylinder with rod and inserts, 60 keV, 1e6 photons.
        dict(name="project_cyl64", kind="project", phantom="cylinder", nx=64, ny=64, nz=64, dv=1.0, kvp=0, sod=300.0,
             nu=128, nv=128, pu=1.0, angles=1, photons=1_000_000, step=0.5, primary=True),
        # The polyenergetic projection the benchmark is quoted on (fewer photons): volume in L2.
        dict(name="project_ell256", kind="project", phantom="ellipsoids", nx=256, ny=256, nz=256, dv=0.5, kvp=120,
             sod=400.0, nu=512, nv=512, pu=0.4, angles=1, photons=20_000_000, step=0.25, primary=True),
        # A batch of angles in one launch, replayed as a graph: volume in HBM, megapixel panel.
        dict(name="project_ell512_batch", kind="project", phantom="ellipsoids", nx=512, ny=512, nz=512, dv=0.2, kvp=0,
             sod=300.0, nu=1024, nv=1024, pu=0.2, angles=6, photons=800_000, step=0.2, primary=True, graph=1),
        # The physics options together: bound electrons, Doppler broadening, expected-value scoring, the panel's
        # response, the variance image; ragged volume and panel.
        dict(name="project_options", kind="project", phantom="ellipsoids", nx=70, ny=66, nz=61, dv=1.5, kvp=100,
             sod=250.0, nu=96, nv=80, pu=2.0, angles=3, photons=300_000, step=0.75, primary=True, bound=1, doppler=1,
             nee=1, response=1, batches=10),
        # The correction's primary image: every angle on the full panel, no histories.
        dict(name="primary_panel", kind="project", phantom="ellipsoids", nx=512, ny=512, nz=512, dv=0.2, kvp=0,
             sod=300.0, nu=2048, nv=2048, pu=0.1, angles=3, photons=0, step=0.2, primary=True),
        # CAD surfaces instead of voxels (5460 triangles).
        dict(name="project_mesh", kind="mesh", seg=1024, kvp=120, sod=300.0, nu=512, nv=512, pu=0.25, angles=3,
             photons=500_000),
        # Reconstruction of a scan.
        dict(name="fdk", kind="fdk", proj=360, nu=1024, nv=1024, pu=0.2, sod=300.0, nx=256, ny=256, nz=256, dv=0.4),
        # Smoothing, angle and pixel interpolation of the simulated scatter onto the panel.
        dict(name="smooth_upsample", kind="upsample", n_in=43, nu=256, nv=256, n_out=256, NU=2048, NV=1536),
        # The correction's re-projection: a reconstruction becomes materials and densities (also down-sampled), is
        # loaded and projected; every new reconstruction pays for the load.
        dict(name="reproject", kind="reproject", nx=256, ny=256, nz=256, dv=0.4, kvp=0, sod=300.0, nu=512, nv=512,
             pu=0.4, sim=128, angles=8, photons=400_000, step=0.4, classes=3),
        # The learned denoiser over the angles of a scan, in batches, the last one short.
        dict(name="denoise_infer", kind="infer", size=256, images=40, batch=16),
        # Two optimiser steps that fine-tune it on new pairs, then the network is read back.
        dict(name="denoise_train", kind="train", size=256, batch=16, steps=2),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["project", "project", "project", "primary", "mesh", "fdk", "upsample", "reproject", "infer",
                       "train"])
    kvp = rng.choice([0, 80, 100, 120])
    if kind == "primary":
        n, panel = int(_log(rng, 48, 512)), int(_log(rng, 100, 2048))
        m = int(n * rng.uniform(0.6, 1.0))
        return dict(kind="project", phantom="ellipsoids", nx=n, ny=n - rng.randrange(7), nz=m, dv=102.4 / n, kvp=kvp,
                    sod=300.0, nu=panel, nv=int(panel * rng.uniform(0.5, 1.0)), pu=204.8 / panel,
                    angles=rng.randint(1, 3), photons=0, step=rng.choice([0.5, 1.0]) * 102.4 / n, primary=True)
    if kind == "project":
        n, panel = int(_log(rng, 16, 512)), int(_log(rng, 16, 1024))
        c = dict(kind="project", phantom="ellipsoids", nx=n, ny=n - rng.randrange(5), nz=int(n * rng.uniform(0.7, 1.0)),
                 dv=110.0 / n, kvp=kvp, sod=300.0, nu=panel, nv=int(panel * rng.uniform(0.6, 1.0)), pu=200.0 / panel,
                 angles=rng.randint(1, 6), photons=0, step=max(0.2, rng.choice([0.5, 1.0]) * 110.0 / n),
                 primary=rng.random() < 0.7)
        c["photons"] = int(_log(rng, 2e4, 4e6) / c["angles"])
        for key, p in (("bound", 0.3), ("nee", 0.3), ("response", 0.3), ("graph", 0.3)):
            if rng.random() < p:
                c[key] = 1
        if c.get("bound") and rng.random() < 0.5:
            c["doppler"] = 1
        if rng.random() < 0.3 and panel <= 512:
            c["batches"] = rng.randint(2, 12)
        if rng.random() < 0.2:
            c["tile"] = 16
        return c
    if kind == "mesh":
        panel = int(_log(rng, 32, 512))
        c = dict(kind="mesh", seg=int(_log(rng, 24, 1024)), kvp=kvp, sod=300.0, nu=panel,
                 nv=int(panel * rng.uniform(0.6, 1.0)), pu=128.0 / panel, angles=rng.randint(1, 3), photons=0)
        c["photons"] = int(_log(rng, 2e4, 1e6) / c["angles"])
        return c
    if kind == "fdk":
        n, nu = int(_log(rng, 48, 256)), int(_log(rng, 100, 1400))
        return dict(kind="fdk", proj=int(_log(rng, 60, 360)), nu=nu, nv=min(1024, int(nu * rng.uniform(0.4, 1.0))),
                    pu=204.8 / nu, sod=300.0, nx=n, ny=n - rng.randrange(6), nz=int(n * rng.uniform(0.5, 1.0)),
                    dv=102.4 / n)
    if kind == "upsample":
        nu, NU = int(_log(rng, 32, 300)), int(_log(rng, 200, 2048))
        return dict(kind="upsample", n_in=int(_log(rng, 3, 60)), nu=nu, nv=max(16, int(nu * rng.uniform(0.6, 1.0))),
                    n_out=int(_log(rng, 8, 200)), NU=NU, NV=int(NU * rng.uniform(0.5, 1.0)))
    if kind == "reproject":
        n, panel = 2 * int(_log(rng, 24, 128)), int(_log(rng, 64, 512))
        return dict(kind="reproject", nx=n, ny=n, nz=2 * int(0.5 * n * rng.uniform(0.5, 1.0)), dv=102.4 / n, kvp=kvp,
                    sod=300.0, nu=panel, nv=panel, pu=204.8 / panel, sim=int(_log(rng, 32, 128)),
                    angles=rng.randint(2, 8), photons=int(_log(rng, 2e4, 3e5)), step=102.4 / n,
                    classes=rng.choice([2, 3]))
    size = 16 * rng.randint(3, 16)
    if kind == "infer":
        return dict(kind="infer", size=size, images=rng.randint(1, 40), batch=rng.choice([1, 4, 8, 16]))
    return dict(kind="train", size=size, batch=rng.randint(2, 16), steps=2)


# ---------------------------------------------------------------------------- inputs
_data = None


def _tables(variant):
    """The cross-section file of the standard materials (written once per process)."""
    global _data
    if _data is None:
        _data = tempfile.mkdtemp(prefix="mcxcases")
    path = default_table_path(variant, _data)
    return path, read_tables(path)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _ellipsoids(c, seed):
    """Air with 8-16 ellipsoids of water, PMMA, aluminium and bone (painter's order): uint8 material ids on the GPU."""
    nx, ny, nz, dv = c["nx"], c["ny"], c["nz"], c["dv"]
    ax = [((torch.arange(n, device=DEV, dtype=torch.float32) - (n - 1) / 2) * dv) for n in (nz, ny, nx)]
    mat = torch.zeros((nz, ny, nx), dtype=torch.uint8, device=DEV)
    half = 0.5 * dv * min(nx, ny, nz)
    for centre, axes, rot, m in ellipsoid_params(seed, fov_half=half, axis_range=(0.08 * half, 0.62 * half)):
        z, y, x = (a - float(centre[k]) for a, k in zip(ax, (2, 1, 0)))
        q = rot / axes[None, :]
        r2 = 0.0
        for j in range(3):
            r2 = r2 + (x[None, None, :] * float(q[0, j]) + y[None, :, None] * float(q[1, j]) + z[:, None, None] * float(q[2, j])) ** 2
        mat[r2 <= 1.0] = m
    return mat


def _volume(c, seed):
    """Material ids and FP16 density bits on the GPU."""
    if c["phantom"] == "ellipsoids":
        mat = _ellipsoids(c, seed)
    elif c["phantom"] == "cylinder":
        mat = torch.from_numpy(cylinder_variant_phantom(seed, n=c["nx"], dv=c["dv"])["mat"]).to(DEV)
    else:
        mat = torch.from_numpy(tiny_phantom(c["nx"], c["dv"])["mat"]).to(DEV)
    dens = torch.tensor(NOMINAL_DENSITY, device=DEV).to(torch.float16)
    return mat, dens[mat.long()] if mat.numel() < 1 << 24 else torch.stack([dens[m.long()] for m in mat])


def _angles(n, seed):
    return (2.0 * np.pi * (np.arange(n) + (seed % 997) / 997.0) / n).astype(np.float32)


def _spectrum(c, tables):
    return kramers_spectrum(tables, kvp=c["kvp"]) if c["kvp"] else mono_spectrum(60.0)


def _context(c):
    path, tables = _tables("bound" if c.get("bound") else "full")
    opt = dict(n_batches=c.get("batches", 1), nee_mode=c.get("nee", 0), doppler=c.get("doppler", 0),
               use_graph=c.get("graph", 0))
    if c.get("tile"):
        opt.update(tally_mode=4, tile_u=c["tile"], tile_v=c["tile"])
    ctx = mcx.Context(0, **opt)
    ctx.load_tables(path)
    ctx.set_spectrum(*_spectrum(c, tables))
    ctx.set_geometry(c["sod"], 2 * c["sod"], c["nu"], c["nv"], c["pu"], c["pu"])
    if c.get("response"):
        ctx.set_detector_response(table_response(tables))
    return ctx, tables


def _shadows(c, seed):
    """Line integrals of a few balls of water and aluminium, seen from a circular orbit, with noise: [proj][nv][nu]."""
    rng = np.random.default_rng(seed)
    sod, pu = c["sod"], c["pu"]
    u = (torch.arange(c["nu"], device=DEV, dtype=torch.float32) - (c["nu"] - 1) / 2) * pu
    v = (torch.arange(c["nv"], device=DEV, dtype=torch.float32) - (c["nv"] - 1) / 2) * pu
    b = torch.from_numpy(_angles(c["proj"], seed)).to(DEV)
    out = torch.empty((c["proj"], c["nv"], c["nu"]), device=DEV)
    torch.randn(out.shape, generator=_gen(seed), device=DEV, out=out).mul_(0.003)
    for k in range(5):
        r = rng.uniform(25.0, 40.0) if k == 0 else rng.uniform(3.0, 9.0)
        x, y, z = rng.uniform(-1.0, 1.0, 3) * (4.0 if k == 0 else 18.0)
        mu = 0.02 if k < 3 else 0.05
        mag = 2 * sod / (sod - (x * torch.cos(b) + y * torch.sin(b)))
        uc, vc, rr = (-x * torch.sin(b) + y * torch.cos(b)) * mag, z * mag, r * mag
        for i in range(0, c["proj"], 64):
            s = slice(i, i + 64)
            t = 1.0 - ((u[None, None, :] - uc[s, None, None]) ** 2 + (v[None, :, None] - vc[s, None, None]) ** 2) / (rr[s, None, None] ** 2)
            out[s] += (2.0 * r * mu) * t.clamp_(min=0.0).sqrt_()
    return out


def _scatter_like(n, h, w, seed):
    """Smooth scatter images and the same with the grain of a low photon count: ([n][h][w] clean, noisy)."""
    g = _gen(seed)
    y = torch.linspace(-1, 1, h, device=DEV)[None, :, None]
    x = torch.linspace(-1, 1, w, device=DEV)[None, None, :]
    p = torch.rand((6, n, 1, 1), generator=g, device=DEV)
    clean = 1.0 + p[0] - 0.5 * (0.5 + p[1]) * (x * x + y * y) + 0.3 * torch.exp(-((x - p[2] + 0.5) ** 2 + (y - p[3] + 0.5) ** 2) / (0.05 + 0.3 * p[4]))
    clean = clean.clamp(min=0.05) * 3e-4 * (0.5 + p[5])
    k = torch.poisson(torch.full((n, h, w), 4.0, device=DEV), generator=g) * 0.25
    return clean.contiguous(), (clean * k * (0.6 + 0.8 * torch.rand((n, h, w), generator=g, device=DEV))).contiguous()


# ---------------------------------------------------------------------------- one pass
def prepare(case, seed):
    c, s = case, {"case": case, "seed": seed}
    if c["kind"] == "project":
        ctx, _ = _context(c)
        mat, rho = _volume(c, seed)
        ctx.load_volume(mat, rho, (c["dv"],) * 3)
        s.update(ctx=ctx, angles=_angles(c["angles"], seed))
    elif c["kind"] == "mesh":
        ctx, _ = _context(c)
        ctx.load_mesh(_mesh(c, seed))
        s.update(ctx=ctx, angles=_angles(c["angles"], seed))
    elif c["kind"] == "fdk":
        ctx = mcx.Context(0)
        ctx.set_geometry(c["sod"], 2 * c["sod"], c["nu"], c["nv"], c["pu"], c["pu"])
        s.update(ctx=ctx, angles=_angles(c["proj"], seed), p=_shadows(c, seed))
    elif c["kind"] == "upsample":
        _, noisy = _scatter_like(c["n_in"], c["nv"], c["nu"], seed)
        s.update(ctx=mcx.Context(0), images=noisy, a_in=_angles(c["n_in"], 0), a_out=_angles(c["n_out"], seed))
    elif c["kind"] == "reproject":
        ctx, tables = _context(c)
        mat = _ellipsoids(c, seed)
        mu = torch.tensor([0.1 * tables.mu_rho_at(m, 60.0) * NOMINAL_DENSITY[m] for m in range(5)], device=DEV, dtype=torch.float32)
        vol = mu[mat.long()] + 0.002 * torch.randn(mat.shape, generator=_gen(seed), device=DEV)
        s.update(ctx=ctx, angles=_angles(c["angles"], seed), vol=vol.contiguous())
    else:
        ctx = mcx.Context(0)
        n = c["images"] if c["kind"] == "infer" else c["batch"] * c["steps"]
        if c["size"] == 256:  # the trained network is one for 256^2 images; other sizes start from a fresh one
            ctx.denoise_load(WEIGHTS, c["batch"])
        else:
            ctx.denoise_init(c["size"], c["size"], c["batch"], seed % 1000)
        clean, noisy = _scatter_like(n, c["size"], c["size"], seed)
        s.update(ctx=ctx, clean=clean, noisy=noisy)
    return s


def _mesh(c, seed):
    """A water cylinder with an aluminium rod inside it, as closed surfaces; the rod's place by the seed."""
    rng = np.random.default_rng(seed)
    at, off = rng.uniform(0, 2 * np.pi), rng.uniform(5.0, 16.0)
    cyl = cylinder_mesh(25.0, 60.0, c["seg"])
    rod = cylinder_mesh(5.0, 60.0, max(16, c["seg"] // 3), center=(off * np.cos(at), off * np.sin(at), 0.0))
    return assemble([(cyl[0], cyl[1], MAT_WATER, 1.0, -1), (rod[0], rod[1], MAT_AL, 2.7, 0)])


def run(state):
    c, ctx, seed = state["case"], state["ctx"], state["seed"]
    if c["kind"] == "project":
        return ctx.project(state["angles"], max(1, c["photons"]), c["step"], seed, primary=c["primary"],
                           scatter=c["photons"] > 0, variance=c.get("batches", 1) > 1 and c["photons"] > 0)
    if c["kind"] == "mesh":
        return ctx.project(state["angles"], c["photons"], 0.5, seed)
    if c["kind"] == "fdk":
        return {"volume": ctx.fdk(state["p"], state["angles"], c["nu"], c["nv"], (c["nx"], c["ny"], c["nz"]) + (c["dv"],) * 3)}
    if c["kind"] == "upsample":
        return {"images": ctx.smooth_upsample(state["images"], state["a_in"], state["a_out"], c["NU"], c["NV"])}
    if c["kind"] == "reproject":
        mat, rho, hist, thr = ctx.segment(state["vol"], c["classes"], (0, MAT_WATER, MAT_AL), 0.001205, 60.0, -0.01, 0.09)
        mat2, rho2 = ctx.bin_volume(mat, rho, 60.0)
        ctx.load_volume(mat, rho, (c["dv"],) * 3)
        ctx.set_geometry(c["sod"], 2 * c["sod"], c["nu"], c["nv"], c["pu"], c["pu"])
        ip = ctx.project(state["angles"], 1, c["step"], seed, scatter=False)["primary"]
        k = c["sim"]
        ctx.load_volume(mat2, rho2, (2 * c["dv"],) * 3)
        ctx.set_geometry(c["sod"], 2 * c["sod"], k, k, c["pu"] * c["nu"] / k, c["pu"] * c["nv"] / k)
        sc = ctx.project(state["angles"], c["photons"], c["step"], seed, primary=False)["scatter"]
        return {"mat": mat, "rho": rho, "hist": hist.astype(np.int64), "thr": thr.astype(np.int64), "mat2": mat2,
                "rho2": rho2, "primary": ip, "scatter": sc}
    if c["kind"] == "infer":
        return {"images": ctx.denoise_infer(state["noisy"])}
    losses = []
    for k in range(c["steps"]):
        b = slice(k * c["batch"], (k + 1) * c["batch"])
        losses.append(ctx.denoise_train_step(state["noisy"][b], state["clean"][b], 5e-6))
    # after training a program reads the network: weights, biases and the last gradients of every layer
    out = {"losses": losses}
    for i in range(15):
        w, bias, gw, gb = ctx.denoise_layer(i)
        out["weights%02d" % i], out["grads%02d" % i] = np.append(w.ravel(), bias), np.append(gw.ravel(), gb)
    return out


# Channels of the denoiser's 15 convolutions and the level (halved resolution) each runs at.
_CIN = (16, 32, 32, 64, 64, 128, 128, 256, 384, 128, 192, 64, 96, 32, 32)
_COUT = (32, 32, 64, 64, 128, 128, 256, 256, 128, 128, 64, 64, 32, 32, 16)
_LEVEL = (0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0, 0)


def work(case):
    """Bytes: inputs once, outputs once.  Flops of a march: 10 per fixed step over the expected chords (a history
    flies about half the object's chord, 0.7 interactions send SPLIT rays over the other half)."""
    c = case
    if c["kind"] in ("project", "reproject"):
        vox, img = c["nx"] * c["ny"] * c["nz"], c["nu"] * c["nv"] * c["angles"]
        chord = 0.6 * c["dv"] * (c["nx"] + c["ny"]) / 2 / c["step"]
        hist = c["photons"] * c["angles"]
        flops = 10.0 * chord * (hist * (0.8 + 0.7 * SPLIT * 0.6) + img)
        if c["kind"] == "project":
            return {"bytes": 3 * vox + 4 * img * (c["primary"] + (c["photons"] > 0) + (c.get("batches", 1) > 1)), "flops": flops}
        return {"bytes": 4 * vox + 3 * vox * 9 / 8 + 4 * img + 4 * c["sim"] ** 2 * c["angles"], "flops": flops}
    if c["kind"] == "mesh":
        img, hist = c["nu"] * c["nv"] * c["angles"], c["photons"] * c["angles"]
        tris = 4 * c["seg"] + 4 * max(16, c["seg"] // 3)
        return {"bytes": 36 * tris + 8 * img, "flops": 400.0 * (img + hist * (1.7 + 0.7 * SPLIT))}
    if c["kind"] == "fdk":
        n, nu = c["proj"] * c["nv"], c["nu"]
        vox = c["nx"] * c["ny"] * c["nz"]
        return {"bytes": 4 * n * nu + 4 * vox, "flops": n * 20.0 * nu * math.log2(4 * nu) + 14.0 * vox * c["proj"]}
    if c["kind"] == "upsample":
        i, o = c["n_in"] * c["nu"] * c["nv"], c["n_out"] * c["NU"] * c["NV"]
        return {"bytes": 4 * i + 4 * o, "flops": 36.0 * i + 8.0 * o}
    n = c["images"] if c["kind"] == "infer" else 3 * c["batch"] * c["steps"]
    flops = sum(18.0 * ci * co * (c["size"] >> lv) ** 2 for ci, co, lv in zip(_CIN, _COUT, _LEVEL)) * n
    px = 8 * c["size"] ** 2
    if c["kind"] == "infer":
        return {"bytes": px * n, "flops": flops}
    par = sum(9 * ci * co + co for ci, co in zip(_CIN, _COUT))
    return {"bytes": px * c["batch"] * c["steps"] + par * 4 * (6 * c["steps"] + 2), "flops": flops}


# ---------------------------------------------------------------------------- the same in 64 bits
def exact(case, seed):
    c = case
    if c["kind"] == "project" and c["primary"]:
        # the scatter image is a sum over random walks: no closed value
        return {"primary": _exact_primary(c, seed), "scatter": None, "variance": None}
    if c["kind"] == "fdk":
        return {"volume": _exact_fdk(c, seed)}
    if c["kind"] == "upsample":
        return {"images": _exact_upsample(c, seed)}
    if c["kind"] in ("infer", "train") and c["size"] == 256:
        n = c["images"] if c["kind"] == "infer" else c["batch"] * c["steps"]
        clean, noisy = (t.double() for t in _scatter_like(n, c["size"], c["size"], seed))
        if c["kind"] == "infer":
            return {"images": _exact_unet(noisy)}
        # the loss before the first step; an optimiser step divides each gradient by its own size, so the weights
        # after it have no value that 16-bit activations could be held to
        b = slice(0, c["batch"])
        s = noisy[b].mean(dim=(1, 2), keepdim=True)
        return {"losses": [float((((_exact_unet(noisy[b]) - clean[b]) / s) ** 2).mean())] + [None] * (c["steps"] - 1)}
    return None


def _exact_primary(c, seed):
    _, tables = _tables("bound" if c.get("bound") else "full")
    E, w = _spectrum(c, tables)
    w = torch.as_tensor(np.asarray(w, dtype=np.float64) / np.sum(w))
    eta = np.interp(E, tables.energies, table_response(tables)) if c.get("response") else np.asarray(E, dtype=np.float64)
    mu = torch.as_tensor(np.stack([tables.mu_rho_at(m, np.asarray(E, dtype=np.float64)) for m in range(tables.n_mat)])).to(DEV) * 0.1
    mat, rho = _volume(c, seed)
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    dv, pu = float(np.float32(c["dv"])), float(np.float32(c["pu"]))
    step, sod = float(np.float32(c["step"])), c["sod"]
    half = torch.tensor([0.5 * nx * dv, 0.5 * ny * dv, 0.5 * nz * dv], dtype=torch.float64, device=DEV)
    u = (torch.arange(c["nu"], device=DEV, dtype=torch.float64) - (c["nu"] - 1) / 2) * pu
    v = (torch.arange(c["nv"], device=DEV, dtype=torch.float64) - (c["nv"] - 1) / 2) * pu
    out = torch.empty((c["angles"], c["nv"], c["nu"]), dtype=torch.float64, device=DEV)
    for k, b in enumerate(_angles(c["angles"], seed).astype(np.float64)):
        cb, sb = math.cos(b), math.sin(b)
        U, V = u[None, :].expand(c["nv"], -1).reshape(-1), v[:, None].expand(-1, c["nu"]).reshape(-1)
        D = torch.stack([-2 * sod * cb - U * sb, -2 * sod * sb + U * cb, V])
        d = D.square().sum(0).sqrt()
        D = D / d
        src = torch.tensor([sod * cb, sod * sb, 0.0], dtype=torch.float64, device=DEV)
        t0 = (-half[:, None] - src[:, None]) / D
        t1 = (half[:, None] - src[:, None]) / D
        lo = torch.minimum(t0, t1).amax(0).clamp(min=0.0)
        hi = torch.minimum(torch.maximum(t0, t1).amin(0), d)
        L = (hi - lo).clamp(min=0.0)
        n = torch.ceil(L / step).clamp(min=1.0)
        h = L / n
        mass = torch.zeros((tables.n_mat, U.numel()), dtype=torch.float64, device=DEV)
        for i in range(int(n.max())):
            t = lo + (i + 0.5) * h
            j = [((src[a] + t * D[a] + half[a]) / dv).floor_().clamp_(0, m - 1).long() for a, m in enumerate((nx, ny, nz))]
            q = (j[2] * ny + j[1]) * nx + j[0]
            r = torch.where((i < n) & (L > 0), rho.view(-1)[q].double(), 0.0)
            mass.scatter_add_(0, mat.view(-1)[q].long()[None], r[None])
        mass *= h
        s = torch.zeros_like(d)
        for e in range(len(E)):
            s += float(w[e]) * float(eta[e]) * torch.exp(-(mu[:, e] @ mass))
        out[k] = (s * pu * pu * 2 * sod / (4 * math.pi * d**3)).view(c["nv"], c["nu"])
    return out


def _exact_fdk(c, seed):
    sod, pu, nu, nv = c["sod"], float(np.float32(c["pu"])) / 2, c["nu"], c["nv"]
    u = (torch.arange(nu, device=DEV, dtype=torch.float64) - (nu - 1) / 2) * pu
    v = (torch.arange(nv, device=DEV, dtype=torch.float64) - (nv - 1) / 2) * pu
    k = torch.arange(-(nu - 1), nu, device=DEV, dtype=torch.float64)
    taps = torch.where(k % 2 != 0, -1.0 / (math.pi * torch.where(k == 0, 1.0, k) * pu) ** 2, 0.0)
    taps[nu - 1] = 0.25 / pu**2
    N = 1 << (3 * nu - 1).bit_length()
    H = torch.fft.rfft(taps, N)
    wgt = sod / (sod**2 + u[None, :] ** 2 + v[:, None] ** 2).sqrt()
    ax = [((torch.arange(c[n], device=DEV, dtype=torch.float64) - (c[n] - 1) / 2) * float(np.float32(c["dv"]))) for n in ("nx", "ny", "nz")]
    X, Y, Z = ax[0][None, :], ax[1][:, None], ax[2]
    vol = torch.zeros((c["nz"], c["ny"], c["nx"]), dtype=torch.float64, device=DEV)
    p = _shadows(c, seed)
    for i, b in enumerate(_angles(c["proj"], seed).astype(np.float64)):
        q = torch.fft.irfft(torch.fft.rfft(p[i].double() * wgt, N) * H, N)[:, nu - 1:2 * nu - 1] * pu
        cb, sb = math.cos(b), math.sin(b)
        mag = sod / (sod - (X * cb + Y * sb))
        fu = (-X * sb + Y * cb) * mag / pu + 0.5 * (nu - 1)
        u0 = fu.floor()
        au, iu = fu - u0, u0.long().clamp(0, nu - 2)
        inu = (u0 >= 0) & (u0 + 1 < nu)
        for z in range(c["nz"]):
            fv = Z[z] * mag / pu + 0.5 * (nv - 1)
            v0 = fv.floor()
            av, j = fv - v0, v0.long().clamp(0, nv - 2) * nu + iu
            f = q.view(-1)
            val = (1 - av) * ((1 - au) * f[j] + au * f[j + 1]) + av * ((1 - au) * f[j + nu] + au * f[j + nu + 1])
            vol[z] += torch.where(inu & (v0 >= 0) & (v0 + 1 < nv), mag * mag * val, 0.0)
    return vol * math.pi / c["proj"]


def _exact_upsample(c, seed):
    _, x = _scatter_like(c["n_in"], c["nv"], c["nu"], seed)
    x = x.double()
    win, order, a = 9, 3, -0.5

    def smooth(n):  # least-squares cubic over the nearest 9 samples, as a matrix
        M, pos = np.zeros((n, n)), np.arange(win) - win // 2
        V = np.vander(pos, order + 1, increasing=True).astype(np.float64)
        hat = V @ np.linalg.inv(V.T @ V) @ V.T
        for i in range(n):
            s = min(max(i - win // 2, 0), n - win)
            M[i, s:s + win] = hat[i - s]
        return torch.as_tensor(M, device=DEV)

    def keys(n, N):  # cubic convolution from n to N samples, edges clamped, as a matrix
        M = np.zeros((N, n))
        for i in range(N):
            s = (i + 0.5) * n / N - 0.5
            for k in range(math.floor(s) - 1, math.floor(s) + 3):
                t = abs(s - k)
                wt = (a + 2) * t**3 - (a + 3) * t**2 + 1 if t <= 1 else (a * t**3 - 5 * a * t**2 + 8 * a * t - 4 * a if t < 2 else 0.0)
                M[i, min(max(k, 0), n - 1)] += wt
        return torch.as_tensor(M, device=DEV)

    low = keys(c["nv"], c["NV"]) @ smooth(c["nv"]) @ x @ (keys(c["nu"], c["NU"]) @ smooth(c["nu"])).T
    ia, oa = _angles(c["n_in"], 0).astype(np.float64), _angles(c["n_out"], seed).astype(np.float64)
    rel = np.append(ia - ia[0], 2 * np.pi)
    out = torch.empty((c["n_out"], c["NV"], c["NU"]), dtype=torch.float64, device=DEV)
    for o, b in enumerate(oa):
        t = (b - ia[0]) % (2 * np.pi)
        k = min(int(np.searchsorted(rel, t, side="right")) - 1, c["n_in"] - 1)
        f = (t - rel[k]) / (rel[k + 1] - rel[k])
        torch.lerp(low[k], low[(k + 1) % c["n_in"]], float(f), out=out[o])
    return out


def _exact_unet(x):
    """The trained network on images x [n][h][w], every number in 64 bits."""
    layers, at = [], 24
    with open(WEIGHTS, "rb") as f:
        data = f.read()
    for ci, co in zip(_CIN, _COUT):
        assert struct.unpack_from("<2i", data, at) == (ci, co)
        w = np.frombuffer(data, "<f4", co * 9 * ci, at + 8).reshape(co, 3, 3, ci).transpose(0, 3, 1, 2)
        b = np.frombuffer(data, "<f4", co, at + 8 + 36 * ci * co)
        at += 8 + 36 * ci * co + 4 * co
        layers.append((torch.as_tensor(w.astype(np.float64)).to(DEV), torch.as_tensor(b.astype(np.float64)).to(DEV)))

    def conv(i, t):  # nine shifted products
        w, b = layers[i]
        n, ci, h, wd = t.shape
        p = torch.nn.functional.pad(t, (1, 1, 1, 1))
        y = b[None, :, None].expand(n, -1, h * wd).clone()
        for k in range(9):
            y += w[:, :, k // 3, k % 3] @ p[:, :, k // 3:k // 3 + h, k % 3:k % 3 + wd].reshape(n, ci, h * wd)
        y = y.view(n, -1, h, wd)
        return y if i == 14 else y.clamp_(min=0.0)

    pool = lambda t: torch.nn.functional.max_pool2d(t, 2)  # noqa: E731
    up = lambda t: t.repeat_interleave(2, 2).repeat_interleave(2, 3)  # noqa: E731
    out = []
    for img in x.split(4):
        s = img.mean(dim=(1, 2), keepdim=True)
        t = torch.zeros((len(img), 16) + img.shape[1:], dtype=torch.float64, device=DEV)
        t[:, 0] = img / s
        s0 = conv(1, conv(0, t))
        s1 = conv(3, conv(2, pool(s0)))
        s2 = conv(5, conv(4, pool(s1)))
        t = conv(7, conv(6, pool(s2)))
        t = conv(9, conv(8, torch.cat([up(t), s2], 1)))
        t = conv(11, conv(10, torch.cat([up(t), s1], 1)))
        t = conv(14, conv(13, conv(12, torch.cat([up(t), s0], 1))))
        out.append(img + s * t[:, 0])
    return torch.cat(out)
