"""Launches whose dynamic shared memory just fits 48 KB.

The kernel's static shared memory counts against the same 48 KB, so such a launch has to ask for more.  The forward
projector of the geometry below takes 49,136 bytes beside 136 static ones; its neighbours in size are on either side.
Projections agree with the FP64 oracle to 1e-5.
"""
import numpy as np
import pytest

import synth
from oracle import algorithms as O

from gpu_helpers import dev, host, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [6, 8, 12, 13])
@pytest.mark.parametrize("z", [40.4, 41.4, 42.4, 43.4, 46.4])
def test_project(nx, z):
    import paper_1808_07150_gb300 as pkg
    import torch
    sc = synth.Scanner(nx=nx, ny=12, nz=111, vx=1.0, vy=1.0, vz=1.0, n_radial=25, d_radial=1.0 / 6.0, n_views=5, radius=8.24,
                       seg_n=(55, 111), seg_zmid0=(z, -55.0), seg_dzmid=(1.0, 1.0), seg_dz=(12.25, 11.22), n_subsets=2,
                       name="edge")
    x = synth.random_image(sc, 1)
    ones = np.ones(sc.sino_shape, np.float32)
    y = torch.zeros(sc.n_bins, device="cuda")
    with pkg.Context(sc) as ctx:
        ctx.spdhg_set_data(dev(ones), dev(ones * 0.1))
        ctx.spdhg_project(dev(x), y, -1)
        torch.cuda.synchronize()
    assert rel(host(y), O.project(sc, x.astype(np.float64))) < 1e-5
