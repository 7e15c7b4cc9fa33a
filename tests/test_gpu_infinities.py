"""Infinite values go where plain arithmetic takes them, and nowhere else."""
import numpy as np
import pytest

import synth

from gpu_helpers import dev, host, problem, upload

pytestmark = pytest.mark.gpu


def _flat():
    return synth.Scanner(nx=40, ny=37, nz=1, vx=1.0, vy=1.0, vz=1.0, n_radial=43, d_radial=1.0, n_views=9, radius=70.0,
                         seg_n=(1,), seg_zmid0=(0.0,), seg_dzmid=(1.0,), seg_dz=(0.0,), n_subsets=3, name="flat")


def test_flat_projections_of_an_infinite_value():
    """Sums that meet it are infinite, the others keep their bits."""
    import paper_1808_07150_gb300 as pkg
    import torch
    sc = _flat()
    ones = np.ones(sc.sino_shape, np.float32)
    x = torch.rand(sc.n_voxels, generator=torch.Generator().manual_seed(1)).cuda()
    y = torch.rand(sc.n_bins, generator=torch.Generator().manual_seed(2)).cuda()
    with pkg.Context(sc) as ctx:
        ctx.spdhg_set_data(dev(ones), dev(ones * 0.1))
        for call, src, n_out, at in ((ctx.spdhg_project, x, sc.n_bins, 19 * 40 + 21), (ctx.spdhg_backproject, y, sc.n_voxels, 4 * 43 + 20)):
            run = lambda v: (call(v, out := torch.zeros(n_out, device="cuda"), -1), out)[1]
            spike, holed, unit = src.clone(), src.clone(), torch.zeros_like(src)
            spike[at], holed[at], unit[at] = float("inf"), 0.0, 1.0
            got, rest, meets = run(spike), run(holed), run(unit) > 0
            torch.cuda.synchronize()
            assert bool(meets.any()) and bool((got[meets] == float("inf")).all())
            assert torch.equal(got[~meets], rest[~meets])


@pytest.mark.parametrize("sc", [_flat(), synth.tiny_3d(n_subsets=2)], ids=lambda s: s.name)
@pytest.mark.parametrize("kind", ["tv", "dtv", "atv", "tgv"])
def test_prior_duals_beyond_the_last_voxel(sc, kind):
    """The last voxel has no neighbour in any direction: its gradient is 0 whatever it holds."""
    import paper_1808_07150_gb300 as pkg
    import torch
    d, _ = problem(sc, side=kind == "dtv")
    x0 = np.ones(sc.image_shape, np.float32)
    x0[-1, -1, -1] = np.inf
    q = torch.full((3 * sc.n_voxels,), 7.0, device="cuda")
    with pkg.Context(sc) as ctx:
        upload(ctx, d)
        ctx.spdhg_setup(pkg.make_params(kind, alpha=0.08, alpha0=0.2, alpha1=0.1), dev(x0))
        ctx.spdhg_iterate(np.array([sc.n_subsets], np.int32))  # the (first) prior block
        ctx.spdhg_get("q", q)
        torch.cuda.synchronize()
    assert (host(q).reshape(3, -1)[:, -1] == 0.0).all()


def test_first_convolution_of_an_infinite_voxel():
    """Through one weight of 1 at tap (dy, dx, dz) the voxel at that distance becomes infinite, and the identity
    layers behind it carry it to the prediction; every other tap's weight of 0 turns it into NaN, which ReLU clears."""
    import torch
    from oracle import unet as U
    from paper_1808_07150_gb300 import learned
    spec, shape, at = U.UNetSpec((16, 16)), (6, 20, 12), (3, 9, 6)
    for tap in [(0, 0, 0), (1, 1, 1), (2, 2, 0), (2, 2, 1), (2, 2, 2)]:
        p = {k: np.zeros(s, np.float32) for k, s in U.layer_shapes(spec)}
        p["enc0a.W"][(0, 0) + tap] = 1.0
        p["enc0b.W"][0, 0, 1, 1, 1] = 1.0
        p["dec0a.W"][0, 16, 1, 1, 1] = 1.0
        p["dec0b.W"][0, 0, 1, 1, 1] = 1.0
        p["head.W"].flat[0] = 1.0
        x = np.full(shape, 0.5, np.float32)
        x[at] = np.inf
        pred = torch.zeros(x.size, device="cuda")
        with learned.UNet(shape, spec.channels) as net:
            net.set_params(np.concatenate([p[k].ravel() for k, _ in U.layer_shapes(spec)]))
            net.forward(dev(x), 1.0, pred)
            out = host(pred).reshape(shape)
        assert out[tuple(a - (t - 1) for a, t in zip(at, tap))] == np.inf, tap
