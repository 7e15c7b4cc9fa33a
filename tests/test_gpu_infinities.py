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
