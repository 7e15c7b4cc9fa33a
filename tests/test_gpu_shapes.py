"""Edge sizes of the kernels against the FP64 oracle: remainders and limits of their tiles.

* Projectors: one warp word of slices and its neighbours (32, 33, 65, 97, 129, 130 slices), one and
  four columns per backprojector warp, tap counts 1 to 4, stages of several views, several component
  batches, more plane tasks than one block takes, mashed components of step 2, flat images around
  32, 64, 128, and an image that does not start on 16 bytes.  Single operators agree to 1e-5
  relative L2 and of the largest entry (FP32 rounding of sums of some hundred terms).
* Backprojection from the tap-item table equals the one that computes its items bit for bit.
* Priors: ragged rows, one to four words of slices, flat images either side of 256 columns; a short
  sequence agrees to 1e-4 in every state array.
* Objective of the zero image: the bins' expectations are the background exactly, so the FP64 data
  term agrees to 1e-12 for ratios from 1e-12 to 1e12 and zero counts.
* U-Net: every channel count of the convolutions on ragged volumes; bars 3e-2 (output) and 6e-2 (gradients),
  those of BF16 activations over at least 300 voxels per level.
"""
import numpy as np
import pytest

import synth
from oracle import algorithms as O
from oracle import unet as U

from gpu_helpers import dev, host, maxerr, problem, rel, upload

pytestmark = pytest.mark.gpu


def _scanner(n, nz, segments=1, taps=1, views=6, subsets=2, mash=False, kind="views", name=""):
    """nx x ny x nz voxels of 1 mm; `segments` segments, the steepest with the tilt that needs `taps` taps."""
    nx, ny = n
    radial = max(nx, ny) + 3
    radius = 1.5 * radial
    h = np.sqrt(radius ** 2 - (0.5 * radial) ** 2)
    dz = (taps - 1.5) * 2.0 * h / np.sqrt(2.0) if taps > 1 else 0.0
    tilt = [dz * (1.0 - 0.5 * (k // 2) / segments) * (1 if k % 2 else -1) for k in range(segments)]
    if segments > 1:
        tilt[0] = 0.0
    sizes = [max(1, nz - (k + 1) // 2) for k in range(segments)]
    z0 = [-0.5 * (s - 1) for s in sizes]
    comps = None
    if mash:  # every plane its own LOR; every second plane two more, of other tilts and ranges
        comps = tuple(((t, 0, s, 1), (0.5 * t, s > 1, s, 2), (0.8 * t, 0, max(1, s - 2), 2)) if k % 2 == 0 else
                      ((t, 0, s, 2), (0.7 * t, s > 1, s, 2), (0.9 * t, 0, max(1, s - 1), 2))
                      for k, (t, s) in enumerate(zip(tilt, sizes)))
    sc = synth.Scanner(nx=nx, ny=ny, nz=nz, vx=1.0, vy=1.0, vz=1.0, n_radial=radial, d_radial=1.0, n_views=views,
                       radius=radius, seg_n=tuple(sizes), seg_zmid0=tuple(z0), seg_dzmid=(1.0,) * segments,
                       seg_dz=tuple(tilt), n_subsets=subsets,
                       name=name or f"{nx}x{ny}x{nz}-s{segments}t{taps}v{views}m{subsets}{'-mash' if mash else ''}-{kind}",
                       **({"components": comps} if comps else {}))
    return sc.with_subsets(subsets, kind)


GEOMS = [
    _scanner((21, 13), 32), _scanner((21, 13), 33, 3, 2), _scanner((20, 14), 65, 3, 3, kind="bins"),
    _scanner((13, 21), 97, 2, 4), _scanner((14, 9), 129, 13, 2), _scanner((14, 9), 130, 15, 3, subsets=6),
    _scanner((102, 99), 9, 3, 2, views=7), _scanner((101, 100), 33, 3, 3), _scanner((100, 103), 5, 5, 4, subsets=6),
    _scanner((101, 100), 64, 1, 1, subsets=6),
    _scanner((21, 13), 33, 3, 2, mash=True), _scanner((20, 14), 65, 3, 3, mash=True), _scanner((21, 13), 40, 5, 4, mash=True),
    _scanner((102, 99), 12, 3, 2, mash=True), _scanner((100, 103), 34, 3, 3, mash=True), _scanner((100, 103), 7, 1, 1, mash=True),
    _scanner((33, 31), 1), _scanner((64, 65), 1, views=9, subsets=9), _scanner((129, 97), 1, kind="bins"), _scanner((130, 128), 1),
]


@pytest.mark.parametrize("sc", GEOMS, ids=lambda s: s.name)
def test_projectors_match_oracle(sc):
    import paper_1808_07150_gb300 as pkg
    import torch
    mult = synth.smooth_multipliers(sc, 9)
    x = synth.random_image(sc, 1)
    yv = synth.random_sinogram(sc, 2)
    ones = np.ones(sc.sino_shape, np.float32)
    shifted = torch.zeros(sc.n_voxels + 1, device="cuda")[1:]
    shifted.copy_(dev(x))
    last = sc.n_subsets - 1
    with pkg.Context(sc) as ctx:
        ctx.spdhg_set_data(dev(ones), dev(ones * 0.1), dev(mult))
        computed = {}
        for subset in (-1, 0, last):
            y, y1 = torch.zeros(sc.n_bins, device="cuda"), torch.zeros(sc.n_bins, device="cuda")
            bp = torch.zeros(sc.n_voxels, device="cuda")
            ctx.spdhg_project(dev(x), y, subset)
            ctx.spdhg_project(shifted, y1, subset)
            ctx.spdhg_backproject(dev(yv), bp, subset)
            torch.cuda.synchronize()
            computed[subset] = bp
            mask = O.subset_mask(sc, subset)
            y_ref = O.project(sc, x.astype(np.float64), subset, mult.astype(np.float64))
            assert rel(host(y)[mask.ravel()], y_ref[mask]) < 1e-5
            assert maxerr(host(y)[mask.ravel()], y_ref[mask]) < 1e-5
            assert torch.equal(y, y1)
            bp_ref = O.backproject(sc, yv.astype(np.float64) * mask, subset, mult.astype(np.float64))
            assert rel(host(bp), bp_ref) < 1e-5
            assert maxerr(host(bp), bp_ref) < 1e-5
        ctx.spdhg_setup(pkg.make_params("none"))  # builds the table where the geometry can have one
        for subset in (0, last):
            bp = torch.zeros(sc.n_voxels, device="cuda")
            ctx.spdhg_backproject(dev(yv), bp, subset)
            torch.cuda.synchronize()
            assert torch.equal(bp, computed[subset])


PRIOR_GEOMS = [_scanner((37, 35), 7), _scanner((35, 33), 33), _scanner((9, 70), 65), _scanner((33, 6), 129),
               _scanner((32, 33), 1), _scanner((256, 9), 1), _scanner((257, 9), 1), _scanner((97, 66), 1)]


@pytest.mark.parametrize("kind", ["tv", "dtv", "atv", "tgv"])
@pytest.mark.parametrize("sc", PRIOR_GEOMS, ids=lambda s: s.name)
def test_priors_match_oracle(sc, kind):
    import paper_1808_07150_gb300 as pkg
    import torch
    d, prob = problem(sc, side=(kind == "dtv"))
    if kind == "tgv":
        prior = O.Prior("tgv", alpha0=0.2, alpha1=0.1)
    else:
        prior = O.Prior(kind, alpha=0.08, side=d["side"].astype(np.float64) if kind == "dtv" else None)
    probs = O.probabilities(sc.n_subsets, prior)
    seq = O.sample(77, 14, probs)
    x0 = synth.random_image(sc, 17) * float(d["x_true"].max())
    sizes = {"x": 1, "z": 1, "q": 3, **({"w": 3, "zw": 3, "q2": 6} if kind == "tgv" else {})}
    got = {k: torch.zeros(n * sc.n_voxels, device="cuda") for k, n in sizes.items()}
    with pkg.Context(sc) as ctx:
        upload(ctx, d)
        ctx.spdhg_setup(pkg.make_params(kind, alpha=0.08, alpha0=0.2, alpha1=0.1), dev(x0))
        ctx.spdhg_iterate(seq)
        for k in got:
            ctx.spdhg_get(k, got[k])
        torch.cuda.synchronize()
    st, steps = O.spdhg(prob, prior, seq, probs, x0=x0.astype(np.float64))
    assert rel(host(got["x"]), O.next_primal(st, steps)) < 1e-4
    assert rel(host(got["z"]), st.z) < 1e-4
    assert rel(host(got["q"]), st.q[0]) < 1e-4
    if kind == "tgv":
        assert rel(host(got["w"]), st.w - steps["T"][1] * st.zbar_w) < 1e-4
        assert rel(host(got["zw"]), st.zw) < 1e-4
        assert rel(host(got["q2"]), st.q[1]) < 1e-4


def test_data_term_over_extreme_ratios():
    import paper_1808_07150_gb300 as pkg
    sc = _scanner((21, 13), 5)
    rng = np.random.default_rng(5)
    b = (10.0 ** rng.uniform(-6, 6, sc.sino_shape)).astype(np.float32)
    r = (10.0 ** rng.uniform(-6, 6, sc.sino_shape)).astype(np.float32)
    near = rng.random(sc.sino_shape) < 0.3
    r[near] = b[near] * (1 + rng.uniform(-1e-3, 1e-3, near.sum())).astype(np.float32)
    b[rng.random(sc.sino_shape) < 0.2] = 0.0
    with pkg.Context(sc) as ctx:
        ctx.spdhg_set_data(dev(b), dev(r))
        ctx.spdhg_setup(pkg.make_params("none"))
        got = ctx.spdhg_objective(dev(np.zeros(sc.image_shape)))[0]
    ref = O.data_fidelity(np.zeros(sc.sino_shape), b.astype(np.float64), r.astype(np.float64))
    assert got == pytest.approx(ref, rel=1e-12)


@pytest.mark.parametrize("channels,shape", [((16, 32), (20, 14, 10)), ((32, 64), (14, 18, 12)),
                                            ((64, 128), (18, 12, 14)), ((128, 16), (18, 12, 14))],
                         ids=lambda v: "x".join(map(str, v)))
def test_unet_channel_counts_match_oracle(channels, shape):
    import torch
    from paper_1808_07150_gb300 import learned
    spec = U.UNetSpec(channels)
    rng = np.random.default_rng(4)
    bf = lambda a: torch.from_numpy(np.asarray(a, np.float32)).bfloat16().float().numpy().astype(np.float64)
    p = U.init_params(spec, 4)
    for k in p:
        if k.endswith(".b"):
            p[k] = 0.05 * rng.standard_normal(p[k].shape)
    p["head.W"] = 0.3 * rng.standard_normal(p["head.W"].shape)
    p = {k: bf(v) for k, v in p.items()}
    x, t = bf(rng.random(shape) + 0.2), rng.random(shape)
    pred_o, cache = U.forward(spec, p, x)
    _, gpred = U.mse_loss(pred_o, t)
    g_o, _ = U.backward(spec, p, cache, gpred)
    names = [name for name, _ in U.layer_shapes(spec)]
    pred = torch.zeros(x.size, device="cuda")
    with learned.UNet(shape, channels) as net:
        net.set_params(np.concatenate([p[k].ravel() for k in names]))
        net.forward(dev(x), 1.0, pred)
        net.backward(dev(t))
        grads, q = net.get_grads().astype(np.float64), 0
        assert learned.device_error() == 0
    assert rel(host(pred).reshape(shape) - x, pred_o - x) < 3e-2
    for k, s in U.layer_shapes(spec):
        n = int(np.prod(s))
        assert rel(grads[q:q + n], g_o[k]) < 6e-2, k
        q += n
