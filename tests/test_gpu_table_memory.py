"""The backprojector's table yields its memory to what a call needs.

OSEM builds the table wherever it fits the context's memory limit; a set-up and an objective that fit beside
the sensitivities alone have to succeed afterwards, and give the same bits as without a table.
"""
import numpy as np
import pytest

import synth
from oracle import algorithms as O

from gpu_helpers import host, problem, upload

pytestmark = pytest.mark.gpu


def test_setup_and_objective_after_osem_within_a_limit():
    import torch
    import paper_1808_07150_gb300 as pkg
    sc = synth.Scanner(nx=40, ny=38, nz=16, vx=1.0, vy=1.0, vz=1.0, n_radial=43, d_radial=1.0, n_views=20, radius=70.0,
                       seg_n=(16, 15), seg_zmid0=(-7.5, -7.0), seg_dzmid=(1.0, 1.0), seg_dz=(0.0, 6.0), n_subsets=4, name="limit")
    d, _ = problem(sc)
    params = pkg.make_params("tgv", alpha0=0.2, alpha1=0.1)
    seq = O.sample(3, 12, O.probabilities(sc.n_subsets, O.Prior("tgv", alpha0=0.2, alpha1=0.1)))
    after_osem, held, x, psi = [], [], [], []
    for table_off in (1, 0):
        with pkg.Context(sc) as ctx:
            ctx.spdhg_tune("bwd_table", table_off)
            upload(ctx, d)
            if held:
                ctx.spdhg_set_memory_limit(held[0])
            ctx.spdhg_osem(pkg.make_params("none", epochs=1))
            after_osem.append(ctx.spdhg_set_memory_limit(held[0] if held else 0))
            ctx.spdhg_setup(params)
            ctx.spdhg_iterate(seq)
            psi.append(ctx.spdhg_objective())
            out = torch.zeros(sc.n_voxels, device="cuda")
            ctx.spdhg_get("x", out)
            torch.cuda.synchronize()
            x.append(host(out))
            held.append(ctx.spdhg_set_memory_limit(0))
    assert after_osem[1] > after_osem[0]  # the table was there
    assert held[1] <= held[0]
    np.testing.assert_array_equal(x[1], x[0])
    assert tuple(psi[1]) == tuple(psi[0])
