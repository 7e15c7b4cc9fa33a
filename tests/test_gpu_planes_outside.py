"""Mashed components whose planes lie far above or below the image's slices.

Their items have no voxel in any lane; the backprojector must neither count nor read anything for them.
Projections agree with the FP64 oracle to 1e-5 (relative L2 and of the largest entry).
"""
import numpy as np
import pytest

import synth
from oracle import algorithms as O

from gpu_helpers import dev, host, maxerr, rel

pytestmark = pytest.mark.gpu


def _scanner(nx, ny, nz, taps):
    radial = max(nx, ny) + 3
    radius = 1.5 * radial
    h = np.sqrt(radius ** 2 - (0.5 * radial) ** 2)
    t = (taps - 1.5) * 2.0 * h / np.sqrt(2.0) if taps > 1 else 0.0
    above, below = 340, 330           # planes from the lowest slice up, and from the highest slice down
    comps = (((t, 0, above, 1), (0.5 * t, 290, above, 1), (0.8 * t, 301, above, 2), (-t, 0, above, 2)),
             ((-t, 0, below, 1), (0.5 * t, 0, 20, 1), (0.7 * t, 1, 30, 2), (t, 0, below, 2)))
    return synth.Scanner(nx=nx, ny=ny, nz=nz, vx=1.0, vy=1.0, vz=1.0, n_radial=radial, d_radial=1.0, n_views=5,
                         radius=radius, seg_n=(above, below), seg_zmid0=(-0.5 * (nz - 1), 0.5 * (nz - 1) - (below - 1)),
                         seg_dzmid=(1.0, 1.0), seg_dz=(t, -t), n_subsets=2, components=comps,
                         name=f"{nx}x{ny}x{nz}-t{taps}")


@pytest.mark.parametrize("sc", [_scanner(14, 9, 12, 1), _scanner(14, 9, 12, 2), _scanner(14, 9, 40, 3), _scanner(14, 9, 130, 4),
                                _scanner(102, 99, 12, 3), _scanner(102, 99, 130, 2)], ids=lambda s: s.name)
def test_projections_match_oracle(sc):
    import paper_1808_07150_gb300 as pkg
    import torch
    x, yv = synth.random_image(sc, 1), synth.random_sinogram(sc, 2)
    ones = np.ones(sc.sino_shape, np.float32)
    with pkg.Context(sc) as ctx:
        ctx.spdhg_set_data(dev(ones), dev(ones * 0.1))
        for subset in (-1, 1):
            y, bp = torch.zeros(sc.n_bins, device="cuda"), torch.zeros(sc.n_voxels, device="cuda")
            ctx.spdhg_project(dev(x), y, subset)
            ctx.spdhg_backproject(dev(yv), bp, subset)
            torch.cuda.synchronize()
            mask = O.subset_mask(sc, subset)
            y_ref = O.project(sc, x.astype(np.float64), subset)
            bp_ref = O.backproject(sc, yv.astype(np.float64) * mask, subset)
            assert rel(host(y)[mask.ravel()], y_ref[mask]) < 1e-5
            assert rel(host(bp), bp_ref) < 1e-5 and maxerr(host(bp), bp_ref) < 1e-5
        ctx.spdhg_setup(pkg.make_params("none"))
        bt = torch.zeros(sc.n_voxels, device="cuda")
        ctx.spdhg_backproject(dev(yv), bt, 1)
        torch.cuda.synchronize()
        assert torch.equal(bp, bt)
