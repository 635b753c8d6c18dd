"""pipeline_stages = 3 asked for by number (256 velocities, eight consumer warps): two
groups of four warps up to degree 3, one group of eight with one velocity per thread above,
on more elements than the CTAs hold, so that the ring wraps and, with two groups, a stage
passes from one group to the other; against the FMA kernel with the same moment sums.

Both do the same FP32 arithmetic in another order: a value is a sum of about 5 Np
products of relative rounding 2^-24, five stages per step, so they differ by at most 5 Np
2^-24 per stage of the largest value; BF16 by a few storage units of the element's
largest deviation."""
import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("p,red", [(0, "default"), (1, "comp"), (1, "default"), (2, "fp64"), (3, "comp"), (4, "default"),
                                   (4, "fp64"), (5, "comp")])
def test_by_number_matches_fma_kernel(prec, p, red):
    c = cases.couette(30, 29, p, velset=("nc", 16), kn=1.0, eq_order=3 if p % 2 else 2)
    s, ref = cases.solver(c, prec, red, stages=3), cases.solver(c, prec, red, stages=1, epc=1, tpb=128)
    assert s.info.pipeline_stages == 3 and s.info.threads_per_cta == 288 and s.info.grid < s.info.K
    out = []
    for x in (s, ref):
        x.set_equilibrium(1.0, 0.02, -0.01, 0.05, 9)
        x.step(2)
        out.append(x.state())
        x.close()
    Np = (p + 1) * (p + 2) // 2
    if prec == "fp32":
        assert np.abs(out[0] - out[1]).max() <= 10 * 5 * Np * 2.0 ** -24 * np.abs(out[1]).max()
    else:
        w = cases.oracle_problem(c).w
        md = np.abs(out[1] / w - 1).max(axis=(1, 2), keepdims=True)
        assert (np.abs(out[0] - out[1]) <= 4 * 2.0 ** -8 * w * md).all()
