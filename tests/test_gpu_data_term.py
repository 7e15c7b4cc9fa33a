"""One bin of the FP64 data term, b log(b / e) + e - b, against exact arithmetic.

All bins but one have b = r = 1 and an image of zero, whose terms are exactly 0, so the objective is
the remaining bin's term.  The term rounds the logarithm, e - b and its result once each (2^-53 of b |log|, |e - b|
and the term; 1 % for the roundings inside the logarithm's small part, which carry a factor of 2^-8.9) and log1p's
series ends at r^7 / 7 < 2^-62, which 2^-58 b covers with the rounding of r.
"""
from decimal import Decimal, getcontext

import numpy as np
import pytest

import synth

from gpu_helpers import dev

pytestmark = pytest.mark.gpu


def test_one_bin_within_three_roundings():
    import paper_1808_07150_gb300 as pkg
    getcontext().prec = 60
    sc = synth.tiny_2d()
    rng = np.random.default_rng(8)
    pairs = [(b, e) for b in (1.0, 3.0, 700.5, 1e-6) for e in (b, 0.999 * b, 1.002 * b, 0.6 * b, 37.0 * b, 1e-5 * b, 1e9 * b)]
    pairs += list(zip(10.0 ** rng.uniform(-12, 12, 60), 10.0 ** rng.uniform(-12, 12, 60)))
    pairs += [(b, b * f) for b, f in zip(10.0 ** rng.uniform(-3, 6, 60), rng.uniform(0.5, 2.0, 60))]
    zero = dev(np.zeros(sc.image_shape))
    worst = 0.0
    with pkg.Context(sc) as ctx:
        for b, e in pairs:
            bs, rs = np.ones(sc.sino_shape, np.float32), np.ones(sc.sino_shape, np.float32)
            bs.flat[5], rs.flat[5] = b, e
            ctx.spdhg_set_data(dev(bs), dev(rs))
            ctx.spdhg_setup(pkg.make_params("none"))
            got = ctx.spdhg_objective(zero)[0]
            B, E = Decimal(float(bs.flat[5])), Decimal(float(rs.flat[5]))
            L = (B / E).ln()
            ref = B * L + E - B
            bound = (abs(B * L) + abs(E - B) + abs(ref)) * Decimal(1.01 * 2.0 ** -53) + B * Decimal(2.0 ** -58)
            worst = max(worst, float(abs(Decimal(float(got)) - ref) / bound))
    assert worst <= 1.0
