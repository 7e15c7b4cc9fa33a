"""Rounding error of a bin that sums many components against the FP64 oracle.

A chunk's component sums are added to each other before they join the bin's sum.  With u = 2^-24 a rounding has
an rms of about 0.4 u of the partial sum it rounds, n equal terms in one running sum 0.4 u sqrt(n / 3) of the
total.  A line of 200 rows has some 250 pixel entries, eight chunks of 32; with nine components, 72 additions
to one sum would have 2.0 u.  Eight additions have 0.65 u, the nine of a chunk 0.25 u, the entries' own 0.2 u,
together 0.7 u, and the lengths add less than 0.3 u.  The bar is 1.4 u (relative L2 over the bins).
"""
import numpy as np
import pytest

import synth
from oracle import algorithms as O

from gpu_helpers import dev, host, rel

pytestmark = pytest.mark.gpu


def test_bins_of_nine_components():
    import paper_1808_07150_gb300 as pkg
    import torch
    n, nz, radial = 200, 8, 203
    comps = (tuple((t, 0, nz, 1) for t in np.linspace(-6.0, 6.0, 9)),)
    sc = synth.Scanner(nx=n, ny=n, nz=nz, vx=1.0, vy=1.0, vz=1.0, n_radial=radial, d_radial=1.0, n_views=7, radius=310.0,
                       seg_n=(nz,), seg_zmid0=(-0.5 * (nz - 1),), seg_dzmid=(1.0,), seg_dz=(0.0,), n_subsets=1,
                       components=comps, name="nine-components")
    x = (np.random.default_rng(4).random(sc.image_shape) + 0.5).astype(np.float32)
    ones = np.ones(sc.sino_shape, np.float32)
    y = torch.zeros(sc.n_bins, device="cuda")
    with pkg.Context(sc) as ctx:
        ctx.spdhg_set_data(dev(ones), dev(ones * 0.1))
        ctx.spdhg_tune("fwd_groups", 1)
        ctx.spdhg_tune("fwd_split", 1)
        ctx.spdhg_project(dev(x), y, -1)
        torch.cuda.synchronize()
    assert rel(host(y), O.project(sc, x.astype(np.float64))) < 1.4 * 2.0 ** -24
