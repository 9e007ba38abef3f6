"""Performance cases of the avalanche-overlay library: what its users have it do.

Every case goes through the package's public entry points.  The sizes and
parameters are those of this repository's own workloads (``inputs.py``,
``bench.py`` and the GPU tests): the parabola-shaped stand-in, the 256^2
plane, the 2048^2 and 8192^2 terrains, the regions of the batched form, the
1024^2 differentiable problem, and the streaming stages alone.  Terrains are
made on the GPU by the recipes of ``inputs.py`` (spectral fBm, and a D8 valley
network for the 8192^2 one), because inputs are made anew for every seed.

Kinds (``case["kind"]``):
  flow      Overlay.terrain -> simulate -> overlay on one DEM
  mask      the same from a caller's mask of known release points
  batch     Batch.run over several regions
  soft      SoftOverlay.deposit and its gradient
  terrain   Overlay.terrain alone (normals, steepness, release list)
  display   velocity, mipmap and the colour-mapped overlay over a base map
  snow      the snow-cover mask
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2506_23364_gb300 as awo

CELL_M = 10.0
MU = math.tan(math.radians(25.0))
RELEASE_FBM = (43.1, 45.0)      # about 4.5% of an fBm surface's cells
RELEASE_VALLEYS = (27.6, 45.0)  # about 4.5% of the 8192^2 terrain's cells
SLOPE_FBM, SLOPE_VALLEYS = 0.87, 0.32  # root mean square slopes of these terrains (m/m)
OPS_PER_MOVE = 126              # algorithmic operations of one attempted move


def listed():
    return [
        # Known release points on a small slope, 2048 particles each (the
        # paper's particle count): the interactive call, where latency and
        # launches count.
        dict(name="parabola-501x151", kind="mask", width=501, height=151, N=2048, cap=2000, moves=187),
        # One 256^2 FP32 slope: the smallest whole workflow, long trajectories.
        dict(name="plane-256", kind="flow", terrain="plane", width=256, height=256, u16=False, levels=1, r=0, N=16,
             cap=1000, P=0.9, k=0.0, s=1.0, lo=30.0, hi=45.0, slope=False, share=0.98, moves=131),
        # A preview on an odd-sized crop of a map with few particles per cell:
        # buffers and rows without any alignment, several mipmap levels.
        dict(name="preview-1021x763", kind="flow", terrain="fbm", width=1021, height=763, u16=True, levels=5, r=0, N=8,
             cap=2000, P=0.9, k=0.0, s=1.0, lo=RELEASE_FBM[0], hi=RELEASE_FBM[1], slope=False, share=0.045, moves=12),
        # The ordinary region: 2048^2 uint16 DEM, 64 particles per release cell.
        dict(name="region-2048", kind="flow", terrain="fbm", width=2048, height=2048, u16=True, levels=1, r=0, N=64,
             cap=4000, P=0.9, k=0.0, s=1.0, lo=RELEASE_FBM[0], hi=RELEASE_FBM[1], slope=False, share=0.045, moves=12),
        # Release points at twice the DEM's resolution, with drag and half-cell
        # steps and the slope raster: the options of the parameter panel.
        dict(name="options-1536x1152", kind="flow", terrain="fbm", width=1536, height=1152, u16=False, levels=4, r=1,
             N=32, cap=4000, P=0.8, k=1e-3, s=0.5, lo=RELEASE_FBM[0], hi=RELEASE_FBM[1], slope=True, share=0.045,
             moves=25),
        # The whole map: 8192^2, 256 particles per release cell, 6 mipmap
        # levels (the benchmark's workload).
        dict(name="map-8192", kind="flow", terrain="valleys", width=8192, height=8192, u16=True, levels=6, r=0, N=256,
             cap=8000, P=0.9, k=0.0, s=1.0, lo=RELEASE_VALLEYS[0], hi=RELEASE_VALLEYS[1], slope=False, share=0.045,
             moves=2.4),
        # Many regions and parameter sets in one batched launch.
        dict(name="batch-12", kind="batch", regions=12, side_lo=512, side_hi=2048, N_lo=32, N_hi=128, cap=4000,
             pick=0, share=0.045, moves=12),
        # Fitting friction and release weights: forward and gradient.
        dict(name="fit-1024", kind="soft", width=1024, height=1024, N=128, cap=2048, moves=15),
        # Terrain analysis of the whole map: decode, normals, slope, release list.
        dict(name="terrain-8192", kind="terrain", terrain="valleys", width=8192, height=8192, u16=True, r=0,
             lo=RELEASE_VALLEYS[0], hi=RELEASE_VALLEYS[1], slope=True, share=0.045),
        # The same at twice the DEM's resolution for the release points.
        dict(name="terrain-texture-4096", kind="terrain", terrain="fbm", width=4096, height=4096, u16=True, r=1,
             lo=RELEASE_FBM[0], hi=RELEASE_FBM[1], slope=False, share=0.045),
        # Display of the finished map: velocity, full mipmap chain, colours
        # blended over the base map.
        dict(name="display-8192", kind="display", width=8192, height=8192, levels=14),
        # Snow cover of an odd-sized map.
        dict(name="snow-5003x4099", kind="snow", width=5003, height=4099),
    ]


def _spread(rng, lo, hi):
    """An integer spread evenly over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    """Width and height, half of them multiples of 64 (map tiles), the others as they fall."""
    w = _spread(rng, lo, hi)
    h = max(48, int(w * rng.uniform(0.6, 1.4)))
    if rng.random() < 0.5:
        w, h = max(64, w // 64 * 64), max(64, h // 64 * 64)
    return w, h


def draw(rng):
    kind = rng.choice(["flow", "flow", "flow", "mask", "batch", "soft", "terrain", "display", "snow"])
    if kind == "mask":
        return dict(kind=kind, width=rng.randint(401, 900), height=rng.randint(101, 400), N=_spread(rng, 256, 4096),
                    cap=2000, moves=187)
    if kind == "batch":
        return dict(kind=kind, regions=rng.randint(2, 12), side_lo=256, side_hi=rng.choice([512, 1024, 2048]),
                    N_lo=16, N_hi=_spread(rng, 32, 128), cap=4000, pick=rng.randint(0, 999), share=0.045, moves=12)
    if kind == "soft":
        w, h = _size(rng, 256, 1200)
        return dict(kind=kind, width=w, height=h, N=_spread(rng, 16, 128), cap=2048, moves=15)
    if kind == "terrain":
        w, h = _size(rng, 200, 6000)
        r = rng.choice([0, 0, 1, 2, -1]) if w * h <= 12_000_000 else 0
        return dict(kind=kind, terrain="fbm", width=w, height=h, u16=rng.random() < 0.7, r=r, lo=RELEASE_FBM[0],
                    hi=RELEASE_FBM[1], slope=rng.random() < 0.5, share=0.045)
    if kind == "display":
        w, h = _size(rng, 200, 8000)
        return dict(kind=kind, width=w, height=min(h, 8000), levels=rng.randint(1, 14))
    if kind == "snow":
        w, h = _size(rng, 200, 8000)
        return dict(kind=kind, width=w, height=min(h, 8000))
    terrain = rng.choice(["fbm", "fbm", "valleys"])
    w, h = _size(rng, 200, 4500)
    r = rng.choice([0, 0, 0, 1, -1])
    s = rng.choice([1.0, 1.0, 0.5])
    share, moves = 0.045, 12 / s
    most = 4e8 / (w * h * 4.0 ** r * share * moves)  # within the largest listed case's work
    return dict(kind="flow", terrain=terrain, width=w, height=h, u16=rng.random() < 0.7, levels=rng.randint(1, 8), r=r,
                N=max(1, min(256, int(most), _spread(rng, 4, 256))), cap=rng.choice([1000, 4000, 8000]),
                P=rng.choice([0.9, 0.9, 0.7]), k=rng.choice([0.0, 0.0, 1e-3]), s=s,
                lo=(RELEASE_FBM if terrain == "fbm" else RELEASE_VALLEYS)[0], hi=45.0, slope=rng.random() < 0.3,
                share=share, moves=moves)


# ----------------------------------------------------------------------------
# Inputs
# ----------------------------------------------------------------------------
def _fbm(H, W, slope, seed):
    """H x W heights from 0: fBm of Hurst exponent 0.8 by spectral synthesis,
    scaled to the root mean square ``slope`` (m/m), within the 6.5 km that
    uint16 decimetres hold."""
    n, m = (H + 63) // 64 * 64, (W + 63) // 64 * 64
    gen = torch.Generator(device="cuda").manual_seed(seed)
    ky = torch.fft.fftfreq(n, device="cuda")[:, None]
    kx = torch.fft.rfftfreq(m, device="cuda")[None, :]
    amp = (ky * ky + kx * kx)
    amp[0, 0] = 1.0
    amp = amp ** (-0.9)
    amp[0, 0] = 0.0
    spec = torch.complex(torch.randn(amp.shape, generator=gen, device="cuda") * amp,
                         torch.randn(amp.shape, generator=gen, device="cuda") * amp)
    z = torch.fft.irfft2(spec, s=(n, m))[:H, :W]
    z = z - z.min()
    dx, dy = (z[:, 1:] - z[:, :-1]) / CELL_M, (z[1:] - z[:-1]) / CELL_M
    scale = torch.minimum(slope / (dx.square().mean() + dy.square().mean()).sqrt(), 6500.0 / z.max())
    return (z * scale).contiguous()


def _carve(z):
    """Lowers a surface along its drainage network: D8 accumulation on the
    block means of 8 x 8 cells, depth min(2 sqrt(A), 150 m)."""
    H, W = z.shape
    c = torch.nn.functional.avg_pool2d(z[None, None], 8)[0, 0]
    h, w = c.shape
    pad = torch.nn.functional.pad(c[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
    idx = torch.arange(h * w, device=z.device).reshape(h, w)
    ys, xs = idx // w, idx % w
    best, to = torch.zeros_like(c), torch.full_like(idx, h * w)
    for dy in (-1, 0, 1):
        for dx in (-1, 0, 1):
            if dx or dy:
                drop = (c - pad[1 + dy:1 + dy + h, 1 + dx:1 + dx + w]) / math.hypot(dx, dy)
                there = (ys + dy).clamp(0, h - 1) * w + (xs + dx).clamp(0, w - 1)
                to = torch.where(drop > best, there, to)
                best = torch.maximum(best, drop)
    to = torch.cat([to.reshape(-1), torch.tensor([h * w], device=z.device)])
    acc = torch.ones(h * w + 1, dtype=torch.int64, device=z.device)
    acc[-1] = 0
    for _ in range(14):  # flow of paths of up to 2^14 cells, doubled each time
        acc = acc.index_add(0, to, acc)
        acc[-1] = 0
        to = to[to]
    depth = (2.0 * acc[:-1].to(torch.float32).sqrt()).clamp(max=150.0).reshape(1, 1, h, w)
    z = z - torch.nn.functional.interpolate(depth, size=(H, W), mode="bilinear", align_corners=True)[0, 0]
    return z - z.min()


def _plane(H, W, seed):
    """A 35 degree slope falling towards +y with a bump and a gully; where they lie follows from the seed."""
    rng = np.random.default_rng(seed)
    y, x = torch.meshgrid(torch.arange(H, device="cuda", dtype=torch.float64),
                          torch.arange(W, device="cuda", dtype=torch.float64), indexing="ij")
    cx, cy, gully = W * rng.uniform(0.4, 0.6), H * rng.uniform(0.25, 0.4), W * rng.uniform(0.45, 0.55)
    z = 2000.0 - y * CELL_M * math.tan(math.radians(35.0))
    z = z + rng.uniform(60.0, 90.0) * torch.exp(-((x - cx) ** 2 + (y - cy) ** 2) / (2.0 * 20.0 ** 2))
    return (z + (x - gully).abs() * CELL_M * math.tan(math.radians(10.0))).to(torch.float32)


def _parabola(H, W, seed):
    """A slope of 35 degrees at the top that flattens out towards +x, with a few centimetres of roughness."""
    x = torch.arange(W, device="cuda", dtype=torch.float64)
    L = 0.7 * W
    prof = math.tan(math.radians(35.0)) * L * CELL_M / 2.0 * (1.0 - x / L).clamp(min=0.0) ** 2
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rough = 0.05 * torch.rand((H, W), generator=gen, device="cuda", dtype=torch.float64)
    return (prof[None, :] + rough).to(torch.float32)


def _quantise(z):
    """Decimetres as uint16, held in an int16 tensor (the same bits)."""
    return (z * 10.0).round().clamp(0, 65535).to(torch.int32).to(torch.int16)


def _dem(case, seed, terrain=None):
    W, H = case["width"], case["height"]
    terrain = terrain or case["terrain"]
    if terrain == "plane":
        return _plane(H, W, seed)
    return _carve(_fbm(H, W, SLOPE_VALLEYS, seed)) if terrain == "valleys" else _fbm(H, W, SLOPE_FBM, seed)


def _overlay(case, seed, **more):
    """An Overlay with its DEM on the device; the release list's unused tail is zero."""
    z = _dem(case, seed)
    ov = awo.Overlay(case["width"], case["height"], CELL_M, quantised=case["u16"], want_slope=case["slope"],
                     release_log2=case["r"], **more)
    ov.load_dem(_quantise(z) if case["u16"] else z)
    ov.cells.zero_()
    return ov


def prepare(case, seed):
    kind = case["kind"]
    W, H = case.get("width"), case.get("height")
    if kind == "flow":
        ov = _overlay(case, seed, levels=case["levels"])
        p = awo.SimParams.make(mu=MU, drag_k=case["k"], persistence=case["P"], step_scale=case["s"],
                               traj_per_cell=case["N"], max_steps=case["cap"], seed=seed)
        return dict(case=case, ov=ov, p=p)
    if kind == "mask":
        ov = awo.Overlay(W, H, CELL_M, quantised=False)
        ov.load_dem(_parabola(H, W, seed))
        ov.cells.zero_()
        mask = torch.zeros((H, W), dtype=torch.uint8, device="cuda")
        rng = np.random.default_rng(seed)
        for f in (0.43, 0.5, 0.56):
            mask[int(f * H), 20 + int(rng.integers(0, 4))] = 1
        return dict(case=case, ov=ov, mask=mask,
                    p=awo.SimParams.make(mu=MU, traj_per_cell=case["N"], max_steps=case["cap"], seed=seed))
    if kind == "batch":
        rng = np.random.default_rng(case["pick"])
        dems, params = [], []
        for i in range(case["regions"]):
            side = int(rng.integers(case["side_lo"] // 64, case["side_hi"] // 64 + 1)) * 64
            mu, k = (float(v * np.exp(rng.uniform(np.log(0.5), np.log(1.5)))) for v in (MU, 1e-3))
            params.append(awo.SimParams.make(mu=mu, drag_k=k, traj_per_cell=int(rng.integers(case["N_lo"], case["N_hi"] + 1)),
                                             max_steps=case["cap"], seed=seed + i))
            dems.append(_quantise(_fbm(side, side, SLOPE_FBM, seed + 100 + i)))
        b = awo.Batch(dems, CELL_M, params, [RELEASE_FBM] * case["regions"], quantised=True)
        for ov in b.ovs:
            ov.cells.zero_()
        return dict(case=case, batch=b)
    if kind == "soft":
        q = _quantise(_dem(case, seed, "fbm")).cpu().numpy().view(np.uint16)
        prob = awo.SoftOverlay(q, CELL_M, RELEASE_FBM, traj_per_cell=case["N"], max_steps=case["cap"], seed=seed)
        gen = torch.Generator(device="cuda").manual_seed(seed)
        w = 0.5 + torch.rand(H * W, generator=gen, device="cuda")  # a map of release weights
        at = prob.cells[:prob.n_cells].to(torch.int64)
        # a fit compares the deposits with a map observed under other parameters
        target = prob.forward_raw(1.2 * MU, 0.8e-3, w[at])
        return dict(case=case, prob=prob, target=target, w=w.requires_grad_(), at=at,
                    log_mu=torch.tensor(math.log(MU), dtype=torch.float64, requires_grad=True),
                    log_k=torch.tensor(math.log(1e-3), dtype=torch.float64, requires_grad=True))
    if kind == "terrain":
        return dict(case=case, ov=_overlay(case, seed))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    g = awo.grid(W, H, CELL_M)
    if kind == "display":
        # a finished run's rasters: a third of the cells hit, counts of a few
        # to a few thousand, energies up to a few hundred metres
        hit = _fbm(H, W, SLOPE_FBM, seed)
        part = hit.reshape(-1)
        part = part[:: max(1, part.numel() // 100_000)].sort().values
        hit = (hit - part[part.numel() * 2 // 3]).clamp(min=0.0)
        maxe = (hit * (500.0 / float(hit.max()))).contiguous()
        count = (torch.rand((H, W), generator=gen, device="cuda") * 40.0 * maxe).to(torch.int32)
        base = torch.randint(0, 256, (H, W, 4), generator=gen, device="cuda", dtype=torch.uint8)
        shapes = awo.lod_shapes(g, case["levels"])[1:]
        return dict(case=case, g=g, maxe=maxe, count=count, base=base, vel=torch.empty_like(maxe),
                    rgba=torch.empty_like(base),
                    count_lv=[torch.empty(s, dtype=torch.int32, device="cuda") for s in shapes],
                    vel_lv=[torch.empty(s, dtype=torch.float32, device="cuda") for s in shapes],
                    cm=awo.Colormap.make(awo.VELOCITY_STOPS, alpha=0.7, count_min=1))
    if kind == "snow":
        h = _dem(case, seed, "fbm")
        normal = torch.empty((3, H, W), device="cuda")
        awo.awo_normals(h, g, normal)
        line = float(round(float(h.mean())))  # the snow line at half height
        return dict(case=case, g=g, h=h, nz=normal[2].contiguous(), alpha=torch.empty_like(h), line=line,
                    rgba=torch.empty((H, W, 4), dtype=torch.uint8, device="cuda"),
                    p=awo.SnowParams(line, 300.0, 36.0, 4.0))
    raise ValueError(kind)


# ----------------------------------------------------------------------------
# One pass
# ----------------------------------------------------------------------------
def _terrain_out(ov):
    out = {"tan2": ov.tan2, "cells": ov.cells, "n": ov.n_rel}
    if ov.normal is not None:
        out["normal"] = ov.normal
    if ov.slope is not None:
        out["slope"] = ov.slope
    if ov.mask is not None:
        out["mask"] = ov.mask
    if ov.quantised:
        out["h"] = ov.h
    return out


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("flow", "mask"):
        ov = state["ov"]
        if kind == "flow":
            ov.run(case["lo"], case["hi"], state["p"])
        else:
            ov.terrain_from_mask(state["mask"])
            ov.simulate(state["p"])
            ov.overlay()
        out = _terrain_out(ov)
        if kind == "mask":
            out.pop("mask")  # this path takes its mask from the caller
        out.update(count=ov.count, maxe=ov.maxe, vel=ov.vel, count_lv=list(ov.count_lv), vel_lv=list(ov.vel_lv),
                   stats=ov.stats)
        return out
    if kind == "batch":
        b = state["batch"]
        b.run()
        return {"count": [ov.count for ov in b.ovs], "maxe": [ov.maxe for ov in b.ovs],
                "vel": [ov.vel for ov in b.ovs], "cells": [ov.cells for ov in b.ovs], "stats": b.stats}
    if kind == "soft":
        D = state["prob"].deposit(state["log_mu"], state["log_k"], state["w"].index_select(0, state["at"]))
        loss = ((D - state["target"]) ** 2).sum()
        g_mu, g_k, g_w = torch.autograd.grad(loss, [state["log_mu"], state["log_k"], state["w"]])
        return {"D": D.detach(), "g_mu": g_mu, "g_k": g_k, "g_w": g_w}
    if kind == "terrain":
        state["ov"].terrain(case["lo"], case["hi"])
        return _terrain_out(state["ov"])
    if kind == "display":
        awo.awo_finalize_lod(state["maxe"], state["count"], state["g"], 9.81, case["levels"], state["vel"],
                             state["count_lv"], state["vel_lv"])
        awo.awo_compose(state["vel"], state["count"], state["g"], state["cm"], state["base"], state["rgba"])
        return {"vel": state["vel"], "count_lv": state["count_lv"], "vel_lv": state["vel_lv"], "rgba": state["rgba"]}
    awo.awo_snow_cover(state["h"], state["nz"], state["g"], state["p"], state["alpha"], state["rgba"])
    return {"alpha": state["alpha"], "rgba": state["rgba"]}


# ----------------------------------------------------------------------------
# What a pass cannot do without
# ----------------------------------------------------------------------------
def _terrain_bytes(case):
    n = case["width"] * case["height"]
    tex = n * 4.0 ** case["r"]
    per_cell = (2 + 4 if case["u16"] else 4) + 12 + 4 + (4 if case["slope"] else 0)
    return per_cell * n + tex * (1 + 4 * case["share"])


def _levels_bytes(n, levels):
    return sum(8 * n / 4.0 ** l for l in range(1, levels))


def work(case):
    kind = case["kind"]
    if kind == "batch":
        n = case["regions"] * ((case["side_lo"] + case["side_hi"]) / 2.0) ** 2
        particles = n * case["share"] * (case["N_lo"] + case["N_hi"]) / 2.0
        return {"bytes": n * (2 + 4 + 4 + 4 * case["share"] + 12), "flops": particles * case["moves"] * OPS_PER_MOVE}
    n = case["width"] * case["height"]
    if kind == "flow":
        particles = n * 4.0 ** case["r"] * case["share"] * case["N"]
        return {"bytes": _terrain_bytes(case) + 12 * n + _levels_bytes(n, case["levels"]),
                "flops": particles * (case["moves"] + 1) * OPS_PER_MOVE + 30 * n}
    if kind == "mask":
        return {"bytes": n * (1 + 4 + 12 + 4 + 12), "flops": 3 * case["N"] * case["moves"] * OPS_PER_MOVE}
    if kind == "soft":
        particles = n * 0.05 * case["N"]
        return {"bytes": n * (4 + 8 + 8 + 8), "flops": 2 * particles * case["moves"] * OPS_PER_MOVE}
    if kind == "terrain":
        return {"bytes": _terrain_bytes(case), "flops": 30 * n}
    if kind == "display":
        return {"bytes": n * (4 + 4 + 4 + 4 + 4) + _levels_bytes(n, case["levels"]), "flops": 30 * n}
    return {"bytes": n * (4 + 4 + 4 + 4), "flops": 20 * n}


# ----------------------------------------------------------------------------
# The formulas in 64 bits
# ----------------------------------------------------------------------------
def _exact_terrain(h, normal=True, slope=False):
    """Normals, tan^2 and slope of FP64 heights: central differences, one-sided at the border."""
    def diff(axis):
        n = h.shape[axis]
        i = torch.arange(n, device=h.device)
        r, l = (i + 1).clamp(max=n - 1), (i - 1).clamp(min=0)
        d = h.index_select(axis, r) - h.index_select(axis, l)
        span = ((r - l).clamp(min=1) * CELL_M).to(torch.float64)
        return d / (span[:, None] if axis == 0 else span[None, :])

    gx, gy = diff(1), diff(0)
    tan2 = gx * gx + gy * gy
    out = {"tan2": tan2}
    if normal:
        inv = 1.0 / (tan2 + 1.0).sqrt()
        out["normal"] = torch.stack([-gx * inv, -gy * inv, inv])
    if slope:
        out["slope"] = torch.rad2deg(torch.atan(tan2.sqrt()))
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "soft"):
        return None  # paths chosen by FP32 comparisons have no 64-bit counterpart
    if kind in ("flow", "mask", "terrain"):
        u16 = case.get("u16", False)
        z = _parabola(case["height"], case["width"], seed) if kind == "mask" else _dem(case, seed)
        if u16:
            z = (_quantise(z).to(torch.int32) & 0xFFFF).to(torch.float64) * float(np.float32(0.1))
        z = z.to(torch.float64)
        out = _exact_terrain(z, True, case.get("slope", False))
        if u16:
            out["h"] = z
        keys = ["cells", "n"] + ([] if kind == "mask" else ["mask"])
        if kind != "terrain":
            levels = case.get("levels", 1) - 1
            keys += ["count", "maxe", "vel", "stats"]
            out.update(count_lv=[None] * levels, vel_lv=[None] * levels)
        return {**dict.fromkeys(keys), **out}
    state = prepare(case, seed)
    if kind == "display":
        vel = (2.0 * float(np.float32(9.81)) * state["maxe"].to(torch.float64)).sqrt()
        levels, v = [], vel
        for _ in range(case["levels"] - 1):
            H, W = v.shape
            v = torch.nn.functional.pad(v, (0, W % 2, 0, H % 2))
            v = torch.maximum(torch.maximum(v[0::2, 0::2], v[0::2, 1::2]), torch.maximum(v[1::2, 0::2], v[1::2, 1::2]))
            levels.append(v)
        return {"vel": vel, "count_lv": [None] * len(levels), "vel_lv": levels, "rgba": None}

    def smooth(e0, e1, x):
        t = ((x - e0) / (e1 - e0)).clamp(0.0, 1.0)
        return t * t * (3.0 - 2.0 * t)

    alpha = smooth(state["line"] - 150.0, state["line"] + 150.0, state["h"].to(torch.float64)) * smooth(
        math.cos(math.radians(38.0)), math.cos(math.radians(34.0)), state["nz"].to(torch.float64))
    return {"alpha": alpha, "rgba": None}
