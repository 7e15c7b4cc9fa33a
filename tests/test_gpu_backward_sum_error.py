"""Rounding error of a backprojected column of many records against the FP64 oracle.

Records of several taps are summed twelve at a time and the sums added in order.  With u = 2^-24 a rounding
has an rms of about 0.4 u of the partial sum it rounds; n equal terms in one running sum give 0.4 u sqrt(n / 3)
of the total, so the 230 records of these columns (60 views and three tilted segments) would have 3.5 u
and more in one chain, and have 0.4 u sqrt(19 / 3) = 1.0 u in 19 sums of twelve, whose own roundings and
those of the lengths add less than 0.3 u.  The bar is 2 u (relative L2 over the image).
"""
import numpy as np
import pytest

import synth
from oracle import algorithms as O

from gpu_helpers import dev, host, rel

pytestmark = pytest.mark.gpu


def _scanner(n, nz, views, tilts):
    radial = n + 3
    S = len(tilts)
    return synth.Scanner(nx=n, ny=n, nz=nz, vx=1.0, vy=1.0, vz=1.0, n_radial=radial, d_radial=1.0, n_views=views,
                         radius=1.5 * radial, seg_n=(nz,) * S, seg_zmid0=(-0.5 * (nz - 1),) * S, seg_dzmid=(1.0,) * S,
                         seg_dz=tuple(tilts), n_subsets=1, name=f"{n}x{n}x{nz}-{views}v-{S}s")


@pytest.mark.parametrize("sc", [_scanner(24, 33, 60, (0.0, 60.0, -60.0)), _scanner(104, 33, 60, (0.0, 250.0, -250.0))],
                         ids=lambda s: s.name)
def test_columns_of_many_records(sc):
    import paper_1808_07150_gb300 as pkg
    import torch
    yv = np.random.default_rng(4).random(sc.sino_shape).astype(np.float32)
    ones = np.ones(sc.sino_shape, np.float32)
    bp = torch.zeros(sc.n_voxels, device="cuda")
    with pkg.Context(sc) as ctx:
        ctx.spdhg_set_data(dev(ones), dev(ones * 0.1))
        ctx.spdhg_backproject(dev(yv), bp, -1)
        torch.cuda.synchronize()
    assert rel(host(bp), O.backproject(sc, yv.astype(np.float64))) < 2 * 2.0 ** -24
