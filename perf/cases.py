"""The renders whose speed is measured: what a user of the library has it draw.

Each case is a dict of plain values; ``listed()`` gives the standing ones and ``draw(rng)``
one more of the same ranges.  ``prepare`` makes the particle set (on the GPU, or in
page-locked host memory for the out-of-core render) and what a program keeps between
frames: the resident scene, the camera, the plan.  ``run`` is one frame (or one batch of
views) through ``paper_1606_04427_gb300.render``.  ``exact`` is the same image in 64 bits
from plain torch: the decisions (projection, coverage) by the FP32 rule of the C header,
the values and sums in FP64.

The sets are drawn on the GPU from the distributions of ``synth.py``: uniform ("plain"),
200 Zipf-weighted Gaussian clusters on a uniform background ("clustered"), and gas plus
stars around the same centres ("two_species"), with smoothing lengths that follow the
local spacing.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1606_04427_gb300 import render, synth

# default values of a case's fields
DEFAULTS = {"kind": "frame", "set": "two_species", "n": 1_000_000, "width": 1024, "height": 1024, "views": 1,
            "storage": "f16", "tile": 0, "distance": 2.0, "azimuth": 0.0, "elevation": 0.0, "accum": False,
            "stable": False, "vector": False, "map": False}


def listed():
    return [
        # the smallest frame of the benchmark: launches and latency count
        {"name": "plain_100k_256", "set": "plain", "n": 100_000, "width": 256, "height": 256, "storage": "f32"},
        # an interactive preview in a window of odd size
        {"name": "preview_1m_ragged", "n": 1_000_003, "width": 637, "height": 483, "storage": "bf16"},
        # the single-species frame of the benchmark, as the accumulation a shard contributes
        {"name": "clustered_10m_1024", "set": "clustered", "n": 10_000_000, "storage": "f32", "accum": True},
        # the headline frame: 70 M gas and 30 M stars
        {"name": "two_species_100m_2048", "n": 100_000_000, "width": 2048, "height": 2048},
        # a served request at the largest image size, the camera close to the set: large particles
        {"name": "close_10m_4096", "set": "clustered", "n": 10_000_000, "width": 4096, "height": 4096,
         "distance": 0.9, "azimuth": 0.7, "elevation": 0.4},
        # a movie: orbit views in one plan, replayed as a CUDA graph
        {"name": "orbit_20m_16x1024", "kind": "plan", "set": "clustered", "n": 20_000_000, "views": 16},
        # a low-resolution preview of the whole orbit
        {"name": "orbit_300k_64x320", "kind": "plan", "set": "clustered", "n": 300_000, "views": 64, "width": 320,
         "height": 240},
        # absorption different from emission: the depth-ordered frame
        {"name": "ordered_10m_2048", "kind": "ordered", "n": 10_000_000, "width": 2048, "height": 2048},
        # one depth slab of a sharded ordered frame, as per-pixel maps, ragged image
        {"name": "ordered_map_1m_ragged", "kind": "ordered", "n": 1_000_000, "width": 1000, "height": 757,
         "storage": "f32", "map": True},
        # stars coloured from a per-particle RGB field
        {"name": "vector_10m_2048", "n": 10_000_000, "width": 2048, "height": 2048, "vector": True},
        # bitwise reproducible frame (regression images)
        {"name": "stable_10m_2048", "n": 10_000_000, "width": 2048, "height": 2048, "stable": True, "accum": True},
        # out of core: the set stays in page-locked host memory
        {"name": "streamed_20m_2048", "kind": "streamed", "n": 20_000_000, "width": 2048, "height": 2048},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "frame", "plan", "ordered", "streamed"])
    c = {"kind": kind, "set": rng.choice(["plain", "clustered", "two_species", "two_species"]),
         "storage": rng.choice(["f32", "f16", "f16", "bf16"]),
         "width": int(_log_uniform(rng, 160, 4096)), "distance": round(_log_uniform(rng, 0.8, 4.0), 3),
         "azimuth": round(rng.uniform(0.0, 6.28), 3), "elevation": round(rng.uniform(-1.2, 1.2), 3)}
    c["height"] = max(96, min(4096, int(c["width"] * rng.uniform(0.5, 1.3))))
    top = {"frame": 6e7, "plan": 4e6, "ordered": 2e7, "streamed": 2e7}[kind]
    n = int(_log_uniform(rng, 5e4, top))
    if kind == "frame":
        c["tile"] = rng.choice([0, 0, 0, 0, 12, 24, 32, 40])
        c["accum"] = rng.random() < 0.3
        c["stable"] = rng.random() < 0.15
        c["vector"] = c["set"] == "two_species" and rng.random() < 0.2
    if kind == "plan":
        c["views"] = rng.randint(2, 24)
        c["width"], c["height"] = min(c["width"], 1200), min(c["height"], 1200)
    if kind == "ordered":
        c["map"] = rng.random() < 0.3
        c["set"] = "two_species"
        if c["width"] * c["height"] > 2048 * 2048:
            c["width"] = c["height"] = 2048 - rng.randint(0, 300)
    if c.get("tile") and -(-c["width"] // c["tile"]) * -(-c["height"] // c["tile"]) > 16384:
        c["tile"] = 0
    # no more covered pixels than the headline frame's 5e9 (a sixth where an evaluation costs more)
    most = 8e8 if kind in ("ordered", "streamed") or c.get("stable") else 4e9
    each = _mean_area(c, 0) * c.get("views", 1)
    c["n"] = max(20_000, min(n, int(most / each)))
    return c


def _full(case):
    return {**DEFAULTS, **case}


def _pixels_per_length(c):
    return 0.5 * c["height"] / math.tan(math.radians(22.5)) / c["distance"]


def _mean_area(c, species):
    """Rough mean covered pixels per particle at the look-at distance (floor of one pixel)."""
    if c["set"] == "plain":
        h2 = 4.1e-5
    else:
        h2 = (0.003 if species == 0 else 0.0006) ** 2 * math.exp(2 * 0.7 ** 2)
    return 1.0 + math.pi * 0.75 ** 2 * h2 * _pixels_per_length(c) ** 2


# -----------------------------------------------------------------------------------------
# particle sets, drawn on the GPU


def _rand(g, *shape):
    return torch.rand(*shape, device="cuda", generator=g)


def _randn(g, *shape):
    return torch.randn(*shape, device="cuda", generator=g)


def _positions(g, n, centres, widths, cum, bg_frac, scale):
    cl = torch.searchsorted(cum, _rand(g, n)).clamp_(max=cum.numel() - 1)
    pos = []
    bg = _rand(g, n) < bg_frac
    for a in range(3):
        p = centres[cl, a] + _randn(g, n) * (widths[cl] * scale)
        p = torch.where(bg, _rand(g, n), p)
        p -= torch.floor(p)
        pos.append(p.clamp_(max=1.0 - 2.0 ** -24))
    return pos


def _density(centres, widths, weights, bg_frac, scale, grid=256):
    t = (torch.arange(grid, device="cuda") + 0.5) / grid
    s = (widths * scale)[:, None]
    g = []
    for a in range(3):
        e = sum(torch.exp(-0.5 * ((t[None, :] - centres[:, a][:, None] - m) / s) ** 2) for m in (-1.0, 0.0, 1.0))
        g.append(e / (math.sqrt(2.0 * math.pi) * s))
    left = ((1.0 - bg_frac) * weights)[:, None, None] * g[0][:, :, None] * g[1][:, None, :]
    rho = (left.reshape(left.shape[0], -1).T @ g[2]).reshape(grid, grid, grid)
    return rho + bg_frac


def _spacing_ranked_h(g, pos, rho, median):
    grid = rho.shape[0]
    cell = torch.zeros(pos[0].numel(), dtype=torch.int64, device="cuda")
    for p in pos:
        cell = cell * grid + (p * grid).long().clamp_(max=grid - 1)
    order = torch.argsort(rho.reshape(-1)[cell], descending=True, stable=True)
    del cell
    draws = torch.sort(torch.exp(_randn(g, pos[0].numel()) * 0.7 + math.log(median)))[0]
    h = torch.empty_like(draws)
    h[order] = draws
    return h


def _particles(case, seed):
    """Arrays of the set (CUDA tensors) and its species tables."""
    c = _full(case)
    n = int(c["n"])
    g = torch.Generator(device="cuda").manual_seed(1000 + int(seed))
    host = np.random.default_rng(int(seed))
    s = {}
    if c["set"] == "plain":
        s["x"], s["y"], s["z"] = (_rand(g, n) for _ in range(3))
        s["h"] = 0.002 + 0.008 * _rand(g, n)
        s["intensity"] = _rand(g, n)
        s["type_begin"], s["cmaps"], s["log"], s["range"] = [0, n], [synth.TWO_POINT_CMAP.copy()], 0, (0.0, 1.0)
    else:
        k = 200
        centres = _rand(g, k, 3)
        widths = torch.exp(math.log(0.005) + _rand(g, k) * math.log(10.0))
        weights = torch.arange(1, k + 1, device="cuda", dtype=torch.float32) ** -1.5
        weights /= weights.sum()
        cum = torch.cumsum(weights, 0)
        n_star = n * 3 // 10 if c["set"] == "two_species" else 0
        n_gas = n - n_star
        pos = _positions(g, n_gas, centres, widths, cum, 0.2, 1.0)
        h = _spacing_ranked_h(g, pos, _density(centres, widths, weights, 0.2, 1.0), 0.003)
        if n_star:
            star = _positions(g, n_star, centres, widths, cum, 0.0, 0.2)
            h = torch.cat([h, _spacing_ranked_h(g, star, _density(centres, widths, weights, 0.0, 0.2), 0.0006)])
            pos = [torch.cat([a, b]) for a, b in zip(pos, star)]
        s["x"], s["y"], s["z"] = pos
        s["h"] = h
        s["intensity"] = torch.exp(_randn(g, n))
        s["type_begin"] = [0, n_gas, n] if n_star else [0, n]
        s["cmaps"] = [synth.smooth_ramp_cmap(host) for _ in range(2)] if n_star else [synth.TWO_POINT_CMAP.copy()]
        s["log"], s["range"] = 1, (-3.0, 3.0)
    types = len(s["type_begin"]) - 1
    # brightness: a mean accumulation near one half per species
    s["brightness"] = np.array([0.5 * c["width"] * c["height"] /
                                max(1.0, (s["type_begin"][t + 1] - s["type_begin"][t]) * 0.25 * _mean_area(c, t))
                                for t in range(types)], np.float32)
    if c["vector"]:  # a positive RGB field with scatter, used for the last species
        s["rgb"] = torch.stack([(1.2 + torch.sin(6.0 * (a + 0.3 * b) * math.pi)) * torch.exp(0.25 * _randn(g, n))
                                for a, b in ((s["x"], s["y"]), (s["y"], s["z"]), (s["z"], s["x"]))], 1)
    return s


def _particle_set(s):
    types = len(s["type_begin"]) - 1
    ps = synth.ParticleSet(s["x"], s["y"], s["z"], s["h"], s["intensity"], np.array(s["type_begin"], np.int64),
                           s["cmaps"], s["brightness"], np.full(types, s["log"], np.int32),
                           np.full(types, s["range"][0], np.float32), np.full(types, s["range"][1], np.float32))
    if "rgb" in s:
        ps.rgb = s["rgb"]
        ps.col_vector = np.array([0] * (types - 1) + [1], np.int32)
    return ps


def _cameras(c):
    if c["kind"] == "plan":
        return synth.orbit_cameras(c["views"], c["width"], c["height"], c["distance"])
    ca, sa, ce, se = math.cos(c["azimuth"]), math.sin(c["azimuth"]), math.cos(c["elevation"]), math.sin(c["elevation"])
    d = c["distance"]
    eye = (0.5 + d * sa * ce, 0.5 + d * se, 0.5 + d * ca * ce)
    return [synth.Camera(eye, (0.5, 0.5, 0.5), (0.0, 1.0, 0.0), 45.0, 1e-3, c["width"], c["height"])]


ABSORB = [1.5, 0.3]  # absorption of gas and stars in units of their emission


# -----------------------------------------------------------------------------------------
# the measured calls


def prepare(case, seed):
    c = _full(case)
    s = _particles(case, seed)
    cams = _cameras(c)
    params = render.RenderParams(tile=c["tile"], accum=c["accum"], stable=c["stable"], map=c["map"])
    state = {"kind": c["kind"], "cam": cams[0], "params": params, "storage": c["storage"]}
    if c["kind"] == "streamed":
        for k in ("x", "y", "z", "h", "intensity"):
            pinned = torch.empty(s[k].shape, dtype=torch.float32, pin_memory=True)
            pinned.copy_(s[k])
            s[k] = pinned
            state["pinned_" + k] = pinned
        ps = _particle_set({**s, **{k: s[k].numpy() for k in ("x", "y", "z", "h", "intensity")}})
        state["set"], state["chunk"] = ps, -(-int(c["n"]) // 3)
        return state
    state["scene"] = render.Scene(_particle_set(s), c["storage"])
    if c["kind"] == "plan":
        state["plan"] = render.Plan(state["scene"], cams, params, graph=True)
        state["out"] = state["plan"].new_output()
    return state


def run(state):
    kind = state["kind"]
    if kind == "plan":
        state["plan"].launch(state["out"])
        return state["out"]
    if kind == "ordered":
        return state["scene"].render_ordered(state["cam"], ABSORB, state["params"])
    if kind == "streamed":
        return render.render_streamed(state["set"], state["cam"], state["chunk"], state["params"],
                                      storage=state["storage"])
    return state["scene"].render(state["cam"], state["params"])


def work(case):
    """Particles read once, the image written once; 40 operations per particle and view for
    the raster and 10 per covered pixel (the distance, the exponent's argument, three
    channel updates), 24 with the transfer of an ordered frame.  The covered pixels are
    those of one draw of the set: pi R^2, less the part of the support's box off the image."""
    c = _full(case)
    s = _particles(case, 0)
    covered = 0.0
    for cam in _cameras(c):
        p = _project(s, c, cam)
        for k in range(0, p["X"].numel(), 1 << 24):
            X, Y, R = (p[m][k:k + (1 << 24)] for m in ("X", "Y", "R"))
            bw = (torch.clamp(X + R, max=c["width"]) - torch.clamp(X - R, min=0.0)).clamp_(min=0.0)
            bh = (torch.clamp(Y + R, max=c["height"]) - torch.clamp(Y - R, min=0.0)).clamp_(min=0.0)
            covered += float((bw * bh).double().sum()) * math.pi / 4
        del p
    elem = 4 if c["storage"] == "f32" or c["kind"] == "streamed" else 2
    channels = 6 if c["map"] else 3
    per_particle = 5 * elem + (12 if c["vector"] else 0)
    flops = 40.0 * c["n"] * c["views"] + (24.0 if c["kind"] == "ordered" else 10.0) * covered
    return {"bytes": float(per_particle) * c["n"] + 4.0 * channels * c["views"] * c["width"] * c["height"],
            "flops": flops}


# -----------------------------------------------------------------------------------------
# the same images in 64 bits

ROUND = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}


def _camera_params(cam):
    eye, look, up = (np.array(v, np.float64) for v in (cam.eye, cam.lookat, cam.up))
    f = (look - eye) / np.sqrt(((look - eye) ** 2).sum())
    side = np.cross(f, up)
    side /= np.sqrt((side ** 2).sum())
    rows = [side, np.cross(side, f), f]
    m = [[float(np.float32(v)) for v in r] + [float(np.float32(-(r @ eye)))] for r in rows]
    focal = float(np.float32(0.5 * cam.height / math.tan(cam.fov_deg * math.pi / 360.0)))
    return m, focal


def _project(s, c, cam):
    """X, Y, R, depth and index of the particles in front of the near plane that may reach
    the image, by the FP32 rule (each operation rounded once)."""
    m, focal = _camera_params(cam)
    kind = ROUND[c["storage"]]
    got = {"X": [], "Y": [], "R": [], "z": [], "i": []}
    for k in range(0, s["x"].numel(), 1 << 24):
        x, y, z, h = (s[a][k:k + (1 << 24)].to(kind).float() for a in ("x", "y", "z", "h"))
        cc = [((x * r[0] + y * r[1]) + z * r[2]) + r[3] for r in m]
        X = (cc[0] * focal) / cc[2] + 0.5 * cam.width
        Y = 0.5 * cam.height - (cc[1] * focal) / cc[2]
        R = ((h * focal) / cc[2] * 0.75).clamp_(min=0.75)
        ok = (cc[2] > np.float32(cam.z_near).item()) & torch.isfinite(X) & torch.isfinite(Y) & torch.isfinite(R)
        ok &= (X + R > -2) & (X - R < cam.width + 2) & (Y + R > -2) & (Y - R < cam.height + 2)
        i = ok.nonzero()[:, 0]
        for name, v in (("X", X), ("Y", Y), ("R", R), ("z", cc[2])):
            got[name].append(v[i])
        got["i"].append(i + k)
    return {name: torch.cat(v) for name, v in got.items()}


def _emission(s, c, idx):
    """FP64 emission of the particles idx, and their species."""
    species = torch.zeros_like(idx)
    for b in s["type_begin"][1:-1]:
        species += idx >= b
    lo, hi = s["range"]
    v = s["intensity"][idx]
    if s["log"]:
        v = torch.log(v.clamp(min=1e-30))
    t = (((v - lo) / (hi - lo)).clamp_(0.0, 1.0)).to(ROUND[c["storage"]]).double()
    e = torch.zeros(idx.numel(), 3, dtype=torch.float64, device="cuda")
    for k, cmap in enumerate(s["cmaps"]):
        beta = float(s["brightness"][k])
        if "rgb" in s and k == len(s["cmaps"]) - 1:
            q = torch.log(s["rgb"][idx].clamp(min=1e-30)).double() if s["log"] else s["rgb"][idx].double()
            col = ((q - lo) / (hi - lo)).clamp_(0.0, 1.0)
        else:
            table = torch.from_numpy(cmap).cuda().double()
            f = t * (table.shape[0] - 1)
            j = f.long().clamp_(max=table.shape[0] - 2)
            tau = (f - j)[:, None]
            col = (1.0 - tau) * table[j] + tau * table[j + 1]
        e = torch.where((species == k)[:, None], beta * col, e)
    return e, species


def _covered(p, cam, sel):
    """Covered (particle, pixel) pairs of the particles `sel`: (position in sel, pixel, weight)."""
    X, Y, R = p["X"][sel], p["Y"][sel], p["R"][sel]
    i0 = (torch.ceil(X - R - 0.5) - 1).clamp_(min=0).long()
    i1 = (torch.floor(X + R - 0.5) + 1).clamp_(max=cam.width - 1).long()
    j0 = (torch.ceil(Y - R - 0.5) - 1).clamp_(min=0).long()
    j1 = (torch.floor(Y + R - 0.5) + 1).clamp_(max=cam.height - 1).long()
    bw, bh = (i1 - i0 + 1).clamp_(min=0), (j1 - j0 + 1).clamp_(min=0)
    cells = bw * bh
    who = torch.repeat_interleave(torch.arange(sel.numel(), device="cuda"), cells)
    k = torch.arange(who.numel(), device="cuda") - (torch.cumsum(cells, 0) - cells)[who]
    row = torch.div(k, bw[who], rounding_mode="floor")
    i, j = i0[who] + k - row * bw[who], j0[who] + row
    dx, dy = (i.float() + 0.5) - X[who], (j.float() + 0.5) - Y[who]
    d2 = dx * dx + dy * dy
    r2 = (R * R)[who]
    on = d2 < r2
    who, d2, r2 = who[on], d2[on].double(), r2[on].double()
    return who, (j * cam.width + i)[on], torch.exp(-4.0 * d2 / r2)


def _batches(p, cells=1 << 25):
    """Ranges of the projected particles with about `cells` box pixels each."""
    total = torch.cumsum(((2 * p["R"] + 3) ** 2).double(), 0)
    n = total.numel()
    if n == 0:
        return []
    parts = int(float(total[-1]) // cells) + 1
    cuts = torch.searchsorted(total, torch.arange(1, parts, device="cuda", dtype=torch.float64) * cells).tolist()
    edges = [0] + cuts + [n]
    return [(a, b) for a, b in zip(edges, edges[1:]) if b > a]


def _exact_view(s, c, cam):
    p = _project(s, c, cam)
    pixels = cam.width * cam.height
    if c["kind"] != "ordered":
        image = torch.zeros(pixels, 3, dtype=torch.float64, device="cuda")
        for a, b in _batches(p):
            sel = torch.arange(a, b, device="cuda")
            e, _ = _emission(s, c, p["i"][sel])
            who, pix, w = _covered(p, cam, sel)
            image.index_add_(0, pix, e[who] * w[:, None])
        image = image if c["accum"] else -torch.expm1(-image)
        return image.reshape(cam.height, cam.width, 3)
    # nearest first; of equal depths the higher index is in front
    order = torch.argsort(p["i"], descending=True)
    order = order[torch.argsort(p["z"][order], stable=True)]
    p = {k: v[order] for k, v in p.items()}
    absorb = torch.tensor(ABSORB, dtype=torch.float64, device="cuda")
    depth = torch.zeros(pixels, 3, dtype=torch.float64, device="cuda")   # absorption so far
    image = torch.zeros(pixels, 3, dtype=torch.float64, device="cuda")
    for a, b in _batches(p, 1 << 24):
        sel = torch.arange(a, b, device="cuda")
        e, species = _emission(s, c, p["i"][sel])
        who, pix, w = _covered(p, cam, sel)
        pix, by = torch.sort(pix, stable=True)
        who, w = who[by], w[by][:, None]
        rate = absorb[species[who]][:, None]
        x = rate * e[who] * w
        run_x = torch.cumsum(x, 0) - x
        first = torch.ones(pix.numel(), dtype=torch.bool, device="cuda")
        first[1:] = pix[1:] != pix[:-1]
        start = torch.cummax(torch.where(first, torch.arange(pix.numel(), device="cuda"), 0), 0)[0]
        before = depth[pix] + (run_x - run_x[start])
        image.index_add_(0, pix, -torch.expm1(-x) / rate * torch.exp(-before))
        depth.index_add_(0, pix, x)
    if c["map"]:
        image = torch.cat([torch.exp(-depth), image], 1)
    return image.reshape(cam.height, cam.width, -1)


def exact(case, seed):
    c = _full(case)
    s = _particles(case, seed)
    views = [_exact_view(s, c, cam) for cam in _cameras(c)]
    return torch.stack(views) if c["kind"] == "plan" else views[0]
