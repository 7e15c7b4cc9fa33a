"""The calls whose speed matters to a user of this framework, with their inputs and an FP64 restatement.

A case is a dict of plain values naming an operation and its sizes.  `prepare` makes on the GPU
what a user's program holds before the call (phantom, Poisson data, multipliers, a set-up
context, network weights), `run` makes one pass through the public entry points, `work` counts the
bytes and operations that pass cannot do without, and `exact` restates it in FP64 torch.

Scanners follow the repository's workloads: "flat" (2-D), "direct" (one plane per slice),
"mashed" (each plane also sums its two adjacent-oblique LORs), "tilted" (a direct and two oblique
segments) and "span11" (eleven segments with the mMR ring differences).
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

import paper_1808_07150_gb300 as pkg
from paper_1808_07150_gb300 import learned

CHANNELS = (16, 32, 64, 128)
SPAN11 = ((0, 0), (6, 11), (6, -11), (17, 22), (17, -22), (28, 33), (28, -33), (39, 44), (39, -44), (50, 55), (50, -55))
RHO = 0.99


# ------------------------------------------------------------------------------------------
# cases
# ------------------------------------------------------------------------------------------

def listed():
    flat = dict(kind="flat", n=64, nz=1, voxel=2.0, radial=95, views=90, radius=200.0)
    cyl = dict(n=128, nz=64, voxel=2.0, radial=128, views=180, radius=300.0, subsets=21)
    mmr = dict(kind="span11", n=344, nz=127, voxel=2.08, radial=344, views=252, radius=380.0, subsets=252)
    return [
        # one epoch of the 2-D reconstruction: short kernels in a chain, launch latency
        dict(name="epoch_2d_tv", op="iterate", prior="tv", subsets=10, data=10, priors=10, mult=False, **flat),
        # one epoch of the 3-D scanner with its adjacent-oblique LORs summed
        dict(name="epoch_3d_mashed_tv", op="iterate", kind="mashed", prior="tv", data=21, priors=21, mult=False, **cyl),
        # a tenth of an epoch of the mMR-scale reconstruction with the anatomical prior
        dict(name="iterate_mmr_dtv", op="iterate", prior="dtv", data=24, priors=24, mult=True, **mmr),
        # one epoch of an odd-sized oblique problem with TGV
        dict(name="epoch_tilted_tgv", op="iterate", kind="tilted", n=171, nz=92, voxel=2.0, radial=171, views=185,
             radius=252.0, subsets=15, prior="tgv", data=15, priors=14, mult=True),
        # the two operators alone, as a user's own algorithm calls them, on one mMR-scale subset
        dict(name="project_mmr", op="project", subset=37, mult=True, **mmr),
        dict(name="backproject_mmr", op="backproject", subset=37, mult=True, **mmr),
        # all bins of a test-sized scanner: the smallest call
        dict(name="project_small", op="project", kind="direct", n=32, nz=16, voxel=2.0, radial=32, views=48, radius=60.0,
             subsets=8, subset=-1, mult=False),
        # an epoch of the OSEM baseline
        dict(name="osem_3d", op="osem", kind="direct", mult=True, epochs=1, **cyl),
        # the stopping rule's objective: a full projection and the FP64 sums
        dict(name="objective_3d_tv", op="objective", kind="tilted", n=187, nz=83, voxel=2.0, radial=187, views=193,
             radius=275.0, subsets=16, prior="tv", mult=True),
        # uneven reconstructions side by side, one graph launch per epoch, set-up included
        dict(name="batch_uneven", op="batch", problems=6, n=72, nz=37, views=84, epochs=2, mult=True),
        # learned warm start: inference, and the gradients of a mini-batch of four
        dict(name="unet_forward", op="unet_forward", ny=128, nx=128, nz=64),
        dict(name="unet_train", op="unet_train", ny=128, nx=128, nz=64, batch=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_scanner(rng, kind):
    if kind == "flat":
        n = _log_int(rng, 24, 256)
        c = dict(n=n, nz=1, voxel=2.0, radial=n + rng.randrange(0, n // 2 + 1), views=rng.randrange(24, 181))
    elif kind == "span11":
        n = rng.randrange(128, 321)
        c = dict(n=n, nz=rng.randrange(41, 128), voxel=2.08, radial=n, views=rng.randrange(28, 169))
    else:
        n = _log_int(rng, 24, 200)
        nz = min(128, max(12, int(n * rng.uniform(0.3, 1.0))))
        c = dict(n=n, nz=nz, voxel=2.0, radial=n, views=rng.randrange(max(24, n // 2), max(49, n + n // 4)))
    half = 0.5 * c["voxel"] * max(c["n"], c["radial"])
    c["radius"] = 380.0 if kind == "span11" else float(math.ceil(math.hypot(half, half)) + 10)
    c["kind"] = kind
    c["subsets"] = c["views"] if kind == "span11" else max(1, c["views"] // rng.choice((4, 8, 12)))
    c["mult"] = rng.random() < 0.7
    return c


def draw(rng):
    op = rng.choice(("iterate", "iterate", "iterate", "project", "backproject", "osem", "objective", "batch",
                     "unet_forward", "unet_train"))
    if op == "batch":
        return dict(op=op, problems=rng.randrange(2, 7), n=rng.randrange(24, 73), nz=rng.randrange(12, 38),
                    views=rng.randrange(24, 85), epochs=rng.randrange(1, 3), mult=rng.random() < 0.5)
    if op in ("unet_forward", "unet_train"):
        c = dict(op=op, ny=8 * _log_int(rng, 2, 16), nx=8 * _log_int(rng, 2, 16), nz=8 * rng.randrange(1, 9))
        return dict(c, batch=rng.randrange(1, 4)) if op == "unet_train" else c
    kinds = ("direct", "mashed", "tilted") if op in ("osem", "objective") else ("flat", "direct", "mashed", "tilted", "span11")
    c = dict(op=op, **_draw_scanner(rng, rng.choice(kinds)))
    if op == "iterate":
        c["prior"] = rng.choice(("tv", "dtv", "atv", "tgv"))
        c["data"] = c["priors"] = min(c["subsets"], 16)
    elif op in ("project", "backproject"):
        c["subset"] = rng.randrange(-1, c["subsets"]) if c["kind"] != "span11" else rng.randrange(c["subsets"])
    elif op == "osem":
        c["epochs"] = 1
    else:
        c["prior"] = rng.choice(("tv", "dtv", "atv"))
    return c


# ------------------------------------------------------------------------------------------
# scanners and inputs
# ------------------------------------------------------------------------------------------

@dataclasses.dataclass(frozen=True)
class Scanner:
    """The geometry fields Context reads; `components` per segment as (dz, first plane, end, step)."""
    nx: int
    ny: int
    nz: int
    vx: float
    vy: float
    vz: float
    n_radial: int
    d_radial: float
    n_views: int
    radius: float
    seg_n: tuple
    seg_zmid0: tuple
    seg_dzmid: tuple
    seg_dz: tuple
    n_subsets: int
    components: tuple = ()

    @property
    def planes(self):
        return sum(self.seg_n)

    @property
    def voxels(self):
        return self.nx * self.ny * self.nz

    @property
    def bins(self):
        return self.n_views * self.n_radial * self.planes

    def lors(self):
        """(dz, z of the mid-points, sinogram planes) of every family of parallel-shifted LORs."""
        out, p0 = [], 0
        for k, n in enumerate(self.seg_n):
            for dz, lo, hi, step in (self.components[k] if self.components else ((self.seg_dz[k], 0, n, 1),)):
                q = torch.arange(lo, hi, step)
                out.append((float(dz), self.seg_zmid0[k] + q.double() * self.seg_dzmid[k], p0 + q))
            p0 += n
        return out


def _scanner(c):
    n, nz, v = c["n"], c["nz"], c["voxel"]
    z0, comps = -(nz - 1) * v / 2, ()
    if c["kind"] == "tilted":
        off = 4 if nz > 24 else 2
        segs = [(0, nz, 0.0), (off, nz - 2 * off, 6 * v), (off, nz - 2 * off, -6 * v)]
    elif c["kind"] == "span11":
        segs = [(first, nz - 2 * first, 2 * v * rd) for first, rd in SPAN11 if nz - 2 * first > 0]
    else:
        segs = [(0, nz, 0.0)]
        if c["kind"] == "mashed":
            comps = (((0.0, 0, nz, 1), (2 * v, 1, nz - 1, 1), (-2 * v, 1, nz - 1, 1)),)
    return Scanner(n, n, nz, v, v, v, c["radial"], v, c["views"], c["radius"], tuple(s[1] for s in segs),
                   tuple(z0 + s[0] * v for s in segs), (v,) * len(segs), tuple(s[2] for s in segs), c["subsets"], comps)


def _problems(c):
    """The uneven reconstructions of a batch case: sizes, views and priors differ."""
    out = []
    for k in range(c["problems"]):
        n, nz, views = c["n"] + 7 * k, c["nz"] + (5 * k) % 11, c["views"] + 9 * k
        out.append(dict(kind="tilted", n=n, nz=nz, voxel=2.0, radial=n, views=views, mult=c["mult"],
                        radius=float(math.ceil(math.sqrt(2.0) * n) + 10), subsets=max(1, views // 12),
                        prior="tgv" if k % 2 else "tv", epochs=c["epochs"]))
    return out


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _ellipsoids(g, seed, count=7):
    """A body and inner ellipsoids: (centre, semi-axes, value), in mm."""
    r = np.random.default_rng(seed)
    hx, hz = 0.5 * g.nx * g.vx, 0.5 * g.nz * g.vz
    out = [((0.0, 0.0, 0.0), (0.7 * hx, 0.6 * hx, 2.0 * hz), r.uniform(0.2, 0.3))]
    for _ in range(count - 1):
        z, az = (0.0, 2.0 * hz) if g.nz == 1 else (r.uniform(-0.6, 0.6) * hz, r.uniform(0.2, 0.9) * hz)
        out.append(((*(r.uniform(-0.35, 0.35, 2) * hx), z), (*(r.uniform(0.06, 0.25, 2) * hx), az), r.uniform(0.2, 1.0)))
    return out


def _image(g, ells, seed, texture=0.1):
    """Phantom at the voxel centres with a multiplicative texture, flat [iy][ix][iz]."""
    ax = [(torch.arange(n, device="cuda", dtype=torch.float64) - 0.5 * (n - 1)) * v
          for n, v in ((g.ny, g.vy), (g.nx, g.vx), (g.nz, g.vz))]
    img = torch.zeros(g.ny, g.nx, g.nz, device="cuda")
    for (cx, cy, cz), (ax_, ay_, az_), value in ells:
        q = (((ax[0] - cy) / ay_) ** 2)[:, None, None] + (((ax[1] - cx) / ax_) ** 2)[None, :, None]
        img += (value * ((q + (((ax[2] - cz) / az_) ** 2)[None, None, :]) <= 1.0)).float()
    noise = torch.rand(img.shape, device="cuda", generator=_generator(seed))
    return (img * (1.0 + texture * (noise - 0.5))).reshape(-1)


def _sinogram_data(g, ells, seed, mult, counts_per_bin=5.0):
    """Poisson counts of the phantom's analytic line integrals, background and multipliers."""
    v = torch.arange(g.n_views, device="cuda", dtype=torch.float64)[:, None, None] * math.pi / g.n_views
    s = (torch.arange(g.n_radial, device="cuda", dtype=torch.float64)[None, :, None] - 0.5 * (g.n_radial - 1)) * g.d_radial
    h = (g.radius ** 2 - s * s).sqrt()
    zm = torch.zeros(g.planes, dtype=torch.float64)
    tilt = torch.zeros(g.planes, dtype=torch.float64)
    for dz, z, planes in reversed(g.lors()):
        zm[planes], tilt[planes] = z, dz
    zm, tilt = zm.cuda()[None, None, :], tilt.cuda()[None, None, :]
    lam = torch.empty(g.n_views, g.n_radial, g.planes, device="cuda")
    for v0 in range(0, g.n_views, 16):
        c, sn = v[v0:v0 + 16].cos(), v[v0:v0 + 16].sin()
        acc = 0.0
        for (cx, cy, cz), (a, b, e), value in ells:
            px, py, pz = (s * c - cx) / a, (s * sn - cy) / b, (zm - cz) / e
            dx, dy, dz = -sn / a, c / b, tilt / (2 * h) / e
            A, B = dx * dx + dy * dy + dz * dz, px * dx + py * dy + pz * dz
            disc = B * B - A * (px * px + py * py + pz * pz - 1.0)
            acc = acc + value * 2.0 * disc.clamp_min(0).sqrt() / A / g.vx
        lam[v0:v0 + 16] = acc.float()
    m = None
    if mult:
        r = torch.arange(g.n_radial, device="cuda")[None, :, None] / g.n_radial
        p = torch.arange(g.planes, device="cuda")[None, None, :] / g.planes
        att = torch.exp(-1.8 * (1.0 - (2.2 * (r - 0.5)) ** 2).clamp_min(0) * (0.9 + 0.1 * torch.cos(2 * v).float()))
        m = ((1.0 + 0.1 * torch.cos(2 * math.pi * 3 * r) + 0.1 * torch.cos(2 * math.pi * 2 * p + seed % 7)) * att).float().contiguous()
        lam *= m
    scale = counts_per_bin / float(lam.mean())
    lam *= scale
    back = 0.1 * counts_per_bin
    lam += back
    b = torch.poisson(lam, generator=_generator(seed + 1))
    return b.reshape(-1), torch.full_like(b, back).reshape(-1), None if m is None else m.reshape(-1), scale


def _problem(c, seed):
    """Scanner and input arrays of a case: counts, background, multipliers, side image, start image."""
    g = _scanner(c)
    ells = _ellipsoids(g, seed)
    b, r, mult, scale = _sinogram_data(g, ells, seed, c["mult"])
    side = _image(g, ells[::2] + _ellipsoids(g, seed + 5, 4)[1:], seed + 2, 0.02) if c.get("prior") == "dtv" else None
    return g, dict(b=b, r=r, mult=mult, side=side, x=_image(g, ells, seed + 3) * scale)


def _params(c, **more):
    return pkg.make_params(c["prior"], alpha=0.05, alpha0=0.2, alpha1=0.1, seed=1808, **more)


def _sequence(c, seed):
    """Block indices of an iterate case: distinct data subsets and the prior blocks, shuffled."""
    r, m = np.random.default_rng(seed), c["subsets"]
    prior = [m + (k % 2 if c["prior"] == "tgv" else 0) for k in range(c["priors"])]
    return r.permutation(np.concatenate([r.permutation(m)[:c["data"]], prior])).astype(np.int32)


def _states(c):
    names = ["x", "z", "y", "q"]
    return names + ["w", "zw", "q2"] if c["prior"] == "tgv" else names


def _state_size(g, name):
    return {"x": g.voxels, "z": g.voxels, "y": g.bins, "q2": 6 * g.voxels}.get(name, 3 * g.voxels)


def _network_layers():
    """(input channels, output channels, taps, level of the output voxels) in the order of the public
    parameter vector; taps 8 is a transposed convolution, taps 1 the head."""
    out, cin, ch = [], 1, CHANNELS
    for l, c in enumerate(ch):
        out += [(cin, c, 27, l), (c, c, 27, l)]
        cin = c
    for l in range(len(ch) - 2, -1, -1):
        out += [(ch[l + 1], ch[l], 8, l + 1), (2 * ch[l], ch[l], 27, l), (ch[l], ch[l], 27, l)]
    return out + [(ch[0], 1, 1, 0)]


def _network_vector(seed):
    """Weights of He-normal size and small biases: a network in training."""
    r, out = np.random.default_rng(seed), []
    for ci, co, taps, _ in _network_layers():
        out += [r.standard_normal(ci * co * taps) * math.sqrt((2.0 if taps > 1 else 0.1) / (ci * taps)), r.standard_normal(co) * 0.02]
    return np.concatenate(out).astype(np.float32)


def _volume(c, seed):
    g = Scanner(c["nx"], c["ny"], c["nz"], 2.0, 2.0, 2.0, 1, 1.0, 1, 1e3, (1,), (0.0,), (2.0,), (0.0,), 1)
    return _image(g, _ellipsoids(g, seed), seed + 1, 0.5) + 0.05


def prepare(case, seed):
    op = case["op"]
    if op.startswith("unet"):
        shape = (case["ny"], case["nx"], case["nz"])
        net = learned.UNet(shape, CHANNELS)
        net.set_params(_network_vector(seed))
        count = case.get("batch", 1)
        s = dict(case=case, net=net, x=[_volume(case, seed + 10 * k) for k in range(count)])
        if op == "unet_train":
            s["target"] = [_volume(case, seed + 10 * k + 5) for k in range(count)]
        else:
            s["pred"], s["x0"] = torch.empty_like(s["x"][0]), torch.empty_like(s["x"][0])
        return s
    if op == "batch":
        s = dict(case=case, contexts=[], params=[], start=[], x=[])
        for k, c in enumerate(_problems(case)):
            g, d = _problem(c, seed + 100 * k)
            ctx = pkg.Context(g)
            ctx.spdhg_set_data(d["b"], d["r"], d["mult"])
            s["contexts"].append(ctx)
            s["params"].append(_params(c, epochs=c["epochs"], graph=True))
            s["start"].append(d["x"])
            s["x"].append(torch.empty_like(d["x"]))
        return s
    g, d = _problem(case, seed)
    ctx = pkg.Context(g)
    ctx.spdhg_set_data(d["b"], d["r"], d["mult"], d["side"])
    s = dict(case=case, g=g, ctx=ctx)
    if op == "project":
        s["x"], s["y"] = d["x"], torch.zeros(g.bins, device="cuda")
    elif op == "backproject":
        s["y"], s["x"] = d["b"] - d["r"], torch.empty(g.voxels, device="cuda")
    elif op == "osem":
        s["params"] = pkg.make_params("none", epochs=case["epochs"])
        s["start"], s["x"] = d["x"] + 1e-3, torch.empty_like(d["x"])
        s["x"].copy_(s["start"])
        ctx.spdhg_osem(pkg.make_params("none", epochs=0), s["x"])  # the sensitivities, kept by the context
    else:
        ctx.spdhg_setup(_params(case), d["x"])
        if op == "iterate":
            s["blocks"] = _sequence(case, seed)
            s["out"] = {k: torch.empty(_state_size(g, k), device="cuda") for k in _states(case)}
    return s


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "iterate":
        ctx = state["ctx"]
        ctx.spdhg_iterate(state["blocks"])
        for name, t in state["out"].items():
            ctx.spdhg_get(name, t)
        return state["out"]
    if op == "project":
        g, subset = state["g"], case["subset"]
        state["ctx"].spdhg_project(state["x"], state["y"], subset)
        y = state["y"].view(g.n_views, g.n_radial, g.planes)
        return y if subset < 0 else y[subset::g.n_subsets]
    if op == "backproject":
        state["ctx"].spdhg_backproject(state["y"], state["x"], case["subset"])
        return state["x"]
    if op == "osem":
        state["x"].copy_(state["start"])
        state["ctx"].spdhg_osem(state["params"], state["x"])
        return state["x"]
    if op == "objective":
        return state["ctx"].spdhg_objective()
    if op == "batch":
        for x, x0 in zip(state["x"], state["start"]):
            x.copy_(x0)
        pkg.spdhg_run_batch(state["contexts"], state["params"], state["x"])
        return state["x"]
    net = state["net"]
    if op == "unet_forward":
        net.forward(state["x"][0], 0.0, state["pred"], state["x0"])
        return state["pred"], state["x0"]
    loss = 0.0
    for k, (x, t) in enumerate(zip(state["x"], state["target"])):
        net.forward(x, 0.0)
        loss += net.backward(t, accumulate=k > 0)
    return net.get_grads(), loss


# ------------------------------------------------------------------------------------------
# the work of one pass
# ------------------------------------------------------------------------------------------

def _iteration_bytes(c, g, count_data, count_prior):
    """Bytes of `count_data` data and `count_prior` prior iterations: inputs read once, outputs
    written once.  Data: x; b, r, mult, sigma, y; y written; x, z, T; x, z written.  Priors: x, z, T
    and the duals read, x, z and the duals written."""
    N, Mi = g.voxels, g.bins // g.n_subsets
    data = 4 * (N + 6 * Mi + 5 * N) + (36 * N if c["prior"] == "tgv" else 0)
    prior = {"tv": 44, "atv": 44, "dtv": 48, "tgv": 102}[c["prior"]] * N  # TGV: 92 and 112 in turn
    return count_data * data + count_prior * prior


def _crossings(g):
    """Pixels a line crosses, averaged over views and radial bins, times the LORs' number per view line."""
    per_line = 4.0 / math.pi * g.nx * g.ny * g.vx / (g.n_radial * g.d_radial)
    return per_line * sum(len(p) for _, _, p in g.lors())


def work(case):
    op = case["op"]
    if op.startswith("unet"):
        V = case["ny"] * case["nx"] * case["nz"]
        flops = 2.0 * sum((V >> 3 * level) * ci * co * taps for ci, co, taps, level in _network_layers())
        weights = 4.0 * sum(ci * co * taps for ci, co, taps, _ in _network_layers())
        if op == "unet_forward":
            return {"bytes": 12.0 * V + weights, "flops": flops}
        return {"bytes": case["batch"] * 8.0 * V + 2 * weights, "flops": case["batch"] * 3 * flops}
    if op == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for c in _problems(case):
            g = _scanner(c)
            e, per = c["epochs"], 2.0 * _crossings(g) * g.n_views * g.n_radial
            total["bytes"] += _iteration_bytes(c, g, e * g.n_subsets, e * g.n_subsets) + 12.0 * g.bins + 16.0 * g.voxels
            total["flops"] += (2 * e + 2) * per  # set-up: the projection and backprojections of ones
        return total
    g = _scanner(case)
    N, M, view = g.voxels, g.bins, 2.0 * _crossings(g) * g.n_radial  # operations of one view's projection
    m_read = 4.0 if case["mult"] else 0.0
    if op in ("project", "backproject"):
        part = 1.0 if case["subset"] < 0 else len(range(case["subset"], g.n_views, g.n_subsets)) / g.n_views
        return {"bytes": 4.0 * N + (4.0 + m_read) * M * part, "flops": view * g.n_views * part}
    if op == "osem":
        return {"bytes": case["epochs"] * (16.0 * N * g.n_subsets + (8.0 + m_read) * M), "flops": case["epochs"] * 2 * view * g.n_views}
    if op == "objective":
        return {"bytes": 4.0 * N * (2 if case["prior"] == "dtv" else 1) + (8.0 + m_read) * M, "flops": view * g.n_views}
    outputs = 8.0 * sum(_state_size(g, k) for k in _states(case))
    return {"bytes": _iteration_bytes(case, g, case["data"], case["priors"]) + outputs,
            "flops": 2 * view * g.n_views / g.n_subsets * case["data"] + 60.0 * N * case["priors"]}


# ------------------------------------------------------------------------------------------
# FP64 restatement: exact line integrals, SPDHG, EM and the network in plain torch
# ------------------------------------------------------------------------------------------

def _pixel_pieces(g, view):
    """(line, pixel, ta, tb) of every transaxial pixel that the lines of a view cross."""
    c, sn = math.cos(math.pi * view / g.n_views), math.sin(math.pi * view / g.n_views)
    c, sn = (0.0 if abs(u) < 1e-12 else u for u in (c, sn))
    dev = dict(device="cuda", dtype=torch.float64)
    s = (torch.arange(g.n_radial, **dev) - 0.5 * (g.n_radial - 1)) * g.d_radial
    h = (g.radius ** 2 - s * s).sqrt()
    x0, y0 = -0.5 * g.nx * g.vx, -0.5 * g.ny * g.vy
    cuts = [-h[:, None], h[:, None]]
    if sn:
        cuts.append(((s * c)[:, None] - (x0 + torch.arange(g.nx + 1, **dev) * g.vx)) / sn)
    if c:
        cuts.append(((y0 + torch.arange(g.ny + 1, **dev) * g.vy) - (s * sn)[:, None]) / c)
    t = torch.cat(cuts, 1)
    t = torch.minimum(torch.maximum(t, -h[:, None]), h[:, None]).sort(1).values
    ta, tb = t[:, :-1], t[:, 1:]
    mid = 0.5 * (ta + tb)
    ix = ((s * c)[:, None] - mid * sn - x0).div(g.vx).floor().long()
    iy = ((s * sn)[:, None] + mid * c - y0).div(g.vy).floor().long()
    ok = (tb - ta > 1e-12) & (ix >= 0) & (ix < g.nx) & (iy >= 0) & (iy < g.ny)
    line = torch.arange(g.n_radial, device="cuda")[:, None].expand_as(ta)[ok]
    return line, (iy * g.nx + ix)[ok], ta[ok], tb[ok], h


def _pieces(g, view, room=1 << 26):
    """Yields (lines, planes, voxel [pieces][planes], length [pieces][planes]) covering every
    intersection of the view's LORs with the voxels; lengths are 0 outside the volume."""
    line, pixel, ta, tb, h = _pixel_pieces(g, view)
    low = -0.5 * g.nz * g.vz
    for dz, zmid, planes in g.lors():
        f, planes = ((zmid - low) / g.vz).cuda()[None, :], planes.cuda()
        step = max(1, room // len(planes))
        for e in range(0, len(line), step):
            L = line[e:e + step]
            kappa = (dz / (2 * h[L] * g.vz))[:, None]
            scale = (1.0 + (dz / (2 * h[L])) ** 2).sqrt()[:, None] / g.vx
            a, b = ta[e:e + step, None], tb[e:e + step, None]
            za, zb = f + kappa * a, f + kappa * b
            lo, hi = torch.minimum(za, zb), torch.maximum(za, zb)
            first = lo.floor()
            reach = int((hi - first).max().item()) + 1 if dz else 1
            per_slab = (b - a) / (hi - lo).clamp_min(1e-300) if dz else None
            for k in range(reach):
                slab = first + k
                if dz:
                    length = (torch.minimum(hi, slab + 1) - torch.maximum(lo, slab)).clamp_min(0) * per_slab * scale
                else:
                    length = ((b - a) * scale).expand_as(slab)
                inside = (slab >= 0) & (slab < g.nz)
                voxel = pixel[e:e + step, None] * g.nz + slab.clamp(0, g.nz - 1).long()
                yield L, planes, voxel, length * inside


def _project(g, x, view):
    out = torch.zeros(g.n_radial, g.planes, device="cuda", dtype=torch.float64)
    for line, planes, voxel, length in _pieces(g, view):
        part = torch.zeros(g.n_radial, len(planes), device="cuda", dtype=torch.float64)
        out[:, planes] += part.index_add_(0, line, length * x[voxel])
    return out


def _backproject(g, y, view, out):
    for line, planes, voxel, length in _pieces(g, view):
        out.index_add_(0, voxel.reshape(-1), (length * y[line][:, planes]).reshape(-1))


def _differences(u):
    """Forward differences with a zero last row, components x, y, z of an [iy][ix][iz] array."""
    d = torch.zeros(3, *u.shape, device="cuda", dtype=torch.float64)
    d[0][:, :-1] = u[:, 1:] - u[:, :-1]
    d[1][:-1] = u[1:] - u[:-1]
    d[2][:, :, :-1] = u[:, :, 1:] - u[:, :, :-1]
    return d


def _differences_t(p):
    """Transpose of one forward difference each: components x, y, z of p, not summed."""
    out = torch.zeros_like(p)
    out[0][:, 1:] += p[0][:, :-1]
    out[0][:, :-1] -= p[0][:, :-1]
    out[1][1:] += p[1][:-1]
    out[1][:-1] -= p[1][:-1]
    out[2][:, :, 1:] += p[2][:, :, :-1]
    out[2][:, :, :-1] -= p[2][:, :, :-1]
    return out


def _symmetrised(w):
    """E w (xx, yy, zz, xy, xz, yz) from backward differences d- = -D^T."""
    d = [-_differences_t(w[k].expand(3, *w[k].shape).contiguous()) for k in range(3)]
    return torch.stack([d[0][0], d[1][1], d[2][2], 0.5 * (d[1][0] + d[0][1]), 0.5 * (d[2][0] + d[0][2]), 0.5 * (d[2][1] + d[1][2])])


def _symmetrised_t(p):
    d = [-_differences(p[k]) for k in range(6)]
    return torch.stack([d[0][0] + d[3][1] + d[4][2], d[1][1] + d[3][0] + d[5][2], d[2][2] + d[4][0] + d[5][1]])


def _dtv_field(side, frac=0.01):
    d = _differences(side)
    eta = frac * float((d * d).sum(0).sqrt().max())
    return d / ((d * d).sum(0) + eta * eta).sqrt()


class _Solver:
    """SPDHG with preconditioned data steps, scalar prior steps and balanced sampling."""

    def __init__(self, c, g, d, x0):
        self.c, self.g = c, g
        shape = (g.ny, g.nx, g.nz)
        f64 = {k: None if v is None else v.double() for k, v in d.items()}
        sino = (g.n_views, g.n_radial, g.planes)
        self.b, self.r = f64["b"].view(sino), f64["r"].view(sino)
        self.mult = torch.ones(1, 1, 1, device="cuda", dtype=torch.float64).expand(sino) if f64["mult"] is None else f64["mult"].view(sino)
        zeros = lambda *n: torch.zeros(*n, device="cuda", dtype=torch.float64)  # noqa: E731
        self.x, self.z, self.y = x0.double().view(shape).clamp_min(0), zeros(shape), zeros(sino)
        self.q, self.q2, self.w, self.zw = zeros(3, *shape), zeros(6, *shape), zeros(3, *shape), zeros(3, *shape)
        tgv = c["prior"] == "tgv"
        blocks = 2 if tgv else 1
        self.p_data, self.p_prior = 0.5 / g.n_subsets, 0.5 / blocks
        norm = math.sqrt(sum(4.0 * math.sin(math.pi * (n - 1) / (2.0 * n)) ** 2 for n in shape))
        norms = [math.sqrt(norm * norm + 1.0), norm] if tgv else [norm]
        self.sigma_prior = [RHO / n for n in norms]
        self.Tw = min(RHO * self.p_prior / n for n in norms)
        self.xi = _dtv_field(f64["side"].view(shape)) if c["prior"] == "dtv" else None
        T = torch.full(shape, RHO * self.p_prior / norms[0], device="cuda", dtype=torch.float64).view(-1)
        seen = torch.zeros_like(T, dtype=torch.bool)
        for i in range(g.n_subsets):
            sens = zeros(g.voxels)
            for v in range(i, g.n_views, g.n_subsets):
                _backproject(g, self.mult[v], v, sens)
            seen |= sens > 0
            T = torch.where(sens > 0, torch.minimum(T, RHO * self.p_data / sens.clamp_min(1e-300)), T)
        self.T = T.view(shape)

    def primal(self, dz, p):
        self.z = self.z + dz
        self.x = (self.x - self.T * (self.z + dz / p)).clamp_min(0)

    def data(self, i):
        g, dz = self.g, torch.zeros(self.g.voxels, device="cuda", dtype=torch.float64)
        ones = torch.ones(g.voxels, device="cuda", dtype=torch.float64)
        for v in range(i, g.n_views, g.n_subsets):
            a1 = self.mult[v] * _project(g, ones, v)
            sigma = torch.where(a1 > 0, RHO / a1.clamp_min(1e-300), torch.zeros_like(a1))
            w = self.y[v] + sigma * (self.mult[v] * _project(g, self.x.view(-1), v) + self.r[v])
            yn = 0.5 * (w + 1.0 - ((w - 1.0) ** 2 + 4.0 * sigma * self.b[v]).sqrt())
            _backproject(g, self.mult[v] * (yn - self.y[v]), v, dz)
            self.y[v] = yn
        self.primal(dz.view_as(self.x), self.p_data)
        if self.c["prior"] == "tgv":
            self.w = self.w - self.Tw * self.zw

    def tgv(self, k):
        first = k == 0
        q, alpha = (self.q, 0.2) if first else (self.q2, 0.1)
        a = q + self.sigma_prior[k] * (_differences(self.x) - self.w if first else _symmetrised(self.w))
        n2 = (a[:3] ** 2).sum(0) + (0 if first else 2.0 * (a[3:] ** 2).sum(0))
        new = a / (n2.sqrt() / alpha).clamp_min(1.0)
        b = new - q
        dzw = -b if first else _symmetrised_t(b)
        self.zw = self.zw + dzw
        self.w = self.w - self.Tw * (self.zw + dzw / self.p_prior)
        if first:
            self.q = new
            self.primal(_differences_t(b).sum(0), self.p_prior)
        else:
            self.q2 = new
            self.x = (self.x - self.T * self.z).clamp_min(0)

    def tv(self):
        kind = self.c["prior"]
        across = (lambda v: v - 0.995 * self.xi * (self.xi * v).sum(0)) if kind == "dtv" else (lambda v: v)
        a = self.q + self.sigma_prior[0] * across(_differences(self.x))
        new = a.clamp(-0.05, 0.05) if kind == "atv" else a / ((a * a).sum(0).sqrt() / 0.05).clamp_min(1.0)
        dz = _differences_t(across(new - self.q)).sum(0)
        self.q = new
        self.primal(dz, self.p_prior)

    def iterate(self, blocks):
        m = self.g.n_subsets
        for i in blocks:
            if i < m:
                self.data(int(i))
            elif self.c["prior"] == "tgv":
                self.tgv(int(i) - m)
            else:
                self.tv()

    def prior_value(self):
        d = _differences(self.x)
        if self.c["prior"] == "atv":
            return 0.05 * float(d.abs().sum())
        if self.xi is not None:
            d = d - 0.995 * self.xi * (self.xi * d).sum(0)
        return 0.05 * float((d * d).sum(0).sqrt().sum())


def _exact_osem(c, g, d):
    sino = (g.n_views, g.n_radial, g.planes)
    b, r = d["b"].double().view(sino), d["r"].double().view(sino)
    mult = torch.ones(sino, device="cuda", dtype=torch.float64) if d["mult"] is None else d["mult"].double().view(sino)
    u = (d["x"] + 1e-3).double()
    for i in list(range(g.n_subsets)) * c["epochs"]:
        sens, ratio = torch.zeros_like(u), torch.zeros_like(u)
        for v in range(i, g.n_views, g.n_subsets):
            _backproject(g, mult[v], v, sens)
            back = mult[v] * _project(g, u, v) + r[v]
            _backproject(g, torch.where(b[v] > 0, mult[v] * b[v] / back, torch.zeros_like(back)), v, ratio)
        u = torch.where(sens > 0, u * ratio / sens.clamp_min(1e-300), torch.zeros_like(u))
    return u


def _exact_objective(c, g, d):
    s = dataclasses.replace(g, n_views=1, n_subsets=1)  # the prior's value needs no step sizes
    solver = _Solver.__new__(_Solver)
    solver.c, solver.g = c, s
    solver.x = d["x"].double().view(g.ny, g.nx, g.nz).clamp_min(0)
    solver.xi = _dtv_field(d["side"].double().view_as(solver.x)) if c["prior"] == "dtv" else None
    sino = (g.n_views, g.n_radial, g.planes)
    total = 0.0
    for v in range(g.n_views):
        ax = _project(g, solver.x.view(-1), v)
        if d["mult"] is not None:
            ax *= d["mult"].view(sino)[v]
        e, b = ax + d["r"].view(sino)[v], d["b"].double().view(sino)[v]
        total += float((e - b + torch.special.xlogy(b, b / e)).sum())
    prior = solver.prior_value()
    return total, prior, total + prior


def _conv3(x, w, b):
    """3x3x3 convolution with zero padding of x [ci][y][x][z], as 27 matrix products."""
    ci, *n = x.shape
    pad = torch.nn.functional.pad(x, (1, 1, 1, 1, 1, 1))
    out = b[:, None].expand(len(b), n[0] * n[1] * n[2])
    for t in range(27):
        ky, kx, kz = t // 9, t // 3 % 3, t % 3
        part = pad[:, ky:ky + n[0], kx:kx + n[1], kz:kz + n[2]].reshape(ci, -1)
        out = out + w[:, :, ky, kx, kz] @ part
    return out.view(len(b), *n)


def _exact_network(vector, shape, x):
    """The network's prediction (units of the mean) from the public parameter vector, FP64."""
    at = 0

    def take(*n):
        nonlocal at
        k = math.prod(n)
        at += k
        return vector[at - k:at].view(*n)

    L, ch = len(CHANNELS), CHANNELS
    xn = (x / x.mean()).view(1, *shape)
    h, skips, cin = xn, [], 1
    for l in range(L):
        if l:
            h = torch.nn.functional.max_pool3d(h[None], 2)[0]
        for ci in (cin, ch[l]):
            w, b = take(ch[l], ci, 3, 3, 3), take(ch[l])
            h = _conv3(h, w, b).relu()
        cin = ch[l]
        skips.append(h)
    for l in range(L - 2, -1, -1):
        w, b = take(ch[l + 1], ch[l], 2, 2, 2), take(ch[l])
        n = h.shape[1:]
        up = torch.einsum("iv,iot->otv", h.reshape(ch[l + 1], -1), w.reshape(ch[l + 1], ch[l], 8)) + b[:, None, None]
        up = up.view(ch[l], 2, 2, 2, *n).permute(0, 4, 1, 5, 2, 6, 3).reshape(ch[l], *(2 * k for k in n))
        h = torch.cat([up, skips[l]])
        for ci in (2 * ch[l], ch[l]):
            w, b = take(ch[l], ci, 3, 3, 3), take(ch[l])
            h = _conv3(h, w, b).relu()
    w, b = take(ch[0]), take(1)
    return (xn[0] + torch.einsum("c,cyxz->yxz", w, h) + b).reshape(-1)


def _exact_unet(case, seed):
    shape = (case["ny"], case["nx"], case["nz"])
    vector = torch.from_numpy(_network_vector(seed)).cuda().double()
    if case["op"] == "unet_forward":
        x = _volume(case, seed).double()
        pred = _exact_network(vector, shape, x)
        return pred, pred * x.mean()
    vector.requires_grad_()
    total = 0.0
    for k in range(case["batch"]):
        x, t = _volume(case, seed + 10 * k).double(), _volume(case, seed + 10 * k + 5).double()
        loss = ((_exact_network(vector, shape, x) - t / x.mean()) ** 2).mean()
        loss.backward()
        total += float(loss.detach())
    return vector.grad, total


def _sampled(seed, count, m, priors):
    """Balanced sampling from the SplitMix64 stream: the first block whose cumulative probability exceeds u."""
    mask, cumulative, out = (1 << 64) - 1, np.cumsum([0.5 / m] * m + [0.5 / priors] * priors), []
    for k in range(count):
        u = (seed + (k + 1) * 0x9E3779B97F4A7C15) & mask
        u = ((u ^ u >> 30) * 0xBF58476D1CE4E5B9) & mask
        u = ((u ^ u >> 27) * 0x94D049BB133111EB) & mask
        u = ((u ^ u >> 31) >> 11) / 9007199254740992.0
        out.append(min(int(np.searchsorted(cumulative, u, side="right")), m + priors - 1))
    return out


def exact(case, seed):
    op = case["op"]
    if op.startswith("unet"):
        return _exact_unet(case, seed)
    if op == "batch":
        out = []
        for k, c in enumerate(_problems(case)):
            g, d = _problem(c, seed + 100 * k)
            solver = _Solver(c, g, d, d["x"])
            solver.iterate(_sampled(1808, 2 * g.n_subsets * c["epochs"], g.n_subsets, 2 if c["prior"] == "tgv" else 1))
            out.append(solver.x.reshape(-1))
        return out
    g, d = _problem(case, seed)
    if op == "project":
        views = range(g.n_views) if case["subset"] < 0 else range(case["subset"], g.n_views, g.n_subsets)
        y = torch.stack([_project(g, d["x"].double(), v) for v in views])
        return y if d["mult"] is None else y * d["mult"].view(g.n_views, g.n_radial, g.planes)[list(views)]
    if op == "backproject":
        views = range(g.n_views) if case["subset"] < 0 else range(case["subset"], g.n_views, g.n_subsets)
        y = (d["b"] - d["r"]).double() * (1.0 if d["mult"] is None else d["mult"].double())
        out = torch.zeros(g.voxels, device="cuda", dtype=torch.float64)
        for v in views:
            _backproject(g, y.view(g.n_views, g.n_radial, g.planes)[v], v, out)
        return out
    if op == "osem":
        return _exact_osem(case, g, d)
    if op == "objective":
        return _exact_objective(case, g, d)
    solver = _Solver(case, g, d, d["x"])
    solver.iterate(_sequence(case, seed))
    return {k: getattr(solver, k).reshape(-1) for k in _states(case)}
