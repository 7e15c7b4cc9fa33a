"""Several radial bins per pixel: set-up, projections and OSEM on geometries whose pair lists are long.

With d_radial = vx / 3 and vx / 9 a pixel has 5 and 13 candidate bins per view, and short rows let many
views share a stage.  Projections agree with the FP64 oracle to 1e-5 (relative L2 and of the largest
entry, FP32 rounding of sums of some hundred terms), with and without the tap-item table in the same bits.
"""
import numpy as np
import pytest

import synth
from oracle import algorithms as O

from gpu_helpers import dev, host, maxerr, rel

pytestmark = pytest.mark.gpu


def _scanner(nx, ny, nz, planes, per_pixel, views, subsets):
    radial = per_pixel * max(nx, ny) + 3
    return synth.Scanner(nx=nx, ny=ny, nz=nz, vx=1.0, vy=1.0, vz=1.0, n_radial=radial, d_radial=1.0 / per_pixel, n_views=views,
                         radius=1.5 * max(nx, ny), seg_n=(planes,), seg_zmid0=(-0.5 * (planes - 1),), seg_dzmid=(1.0,),
                         seg_dz=(0.0,), n_subsets=subsets, name=f"{nx}x{ny}x{nz}-{per_pixel}bins-{views // subsets}views")


GEOMS = [_scanner(104, 100, 12, 12, 3, 26, 2),    # the pair lists of 13 views would take 49,920 bytes
         _scanner(100, 103, 4, 4, 9, 32, 2),      # 159,744 bytes at 16 views a stage
         _scanner(100, 103, 130, 7, 9, 32, 2),    # eight words of slices
         _scanner(33, 30, 4, 4, 9, 32, 2)]        # one column per warp


@pytest.mark.parametrize("sc", GEOMS, ids=lambda s: s.name)
def test_projections_and_setup(sc):
    import paper_1808_07150_gb300 as pkg
    import torch
    x, yv = synth.random_image(sc, 1), synth.random_sinogram(sc, 2)
    ones = np.ones(sc.sino_shape, np.float32)
    with pkg.Context(sc) as ctx:
        ctx.spdhg_set_data(dev(ones), dev(ones * 0.1))
        y, bp, bt = torch.zeros(sc.n_bins, device="cuda"), *(torch.zeros(sc.n_voxels, device="cuda") for _ in range(2))
        ctx.spdhg_project(dev(x), y, 1)
        ctx.spdhg_backproject(dev(yv), bp, 1)
        ctx.spdhg_setup(pkg.make_params("none"))
        ctx.spdhg_backproject(dev(yv), bt, 1)
        torch.cuda.synchronize()
        mask = O.subset_mask(sc, 1)
        y_ref = O.project(sc, x.astype(np.float64), 1)
        bp_ref = O.backproject(sc, yv.astype(np.float64) * mask, 1)
        assert rel(host(y)[mask.ravel()], y_ref[mask]) < 1e-5
        assert rel(host(bp), bp_ref) < 1e-5 and maxerr(host(bp), bp_ref) < 1e-5
        assert torch.equal(bp, bt)


def test_osem_is_accepted_at_the_first_call():
    import paper_1808_07150_gb300 as pkg
    import torch
    sc = GEOMS[0]
    ones = np.ones(sc.sino_shape, np.float32)
    u = torch.ones(sc.n_voxels, device="cuda")
    with pkg.Context(sc) as ctx:
        ctx.spdhg_set_data(dev(ones), dev(ones * 0.1))
        ctx.spdhg_osem(pkg.make_params("none", epochs=1), u)
        torch.cuda.synchronize()
    assert bool(torch.isfinite(u).all())
