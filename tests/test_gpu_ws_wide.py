"""The wide warp-specialised stage kernel (any velocity count from 512 up, neighbour
traces read from global memory): counts that leave the last pass over the velocities
partly empty (1,089 padded to 1,120; 24 x 24 = 576), every face kind, more and fewer
elements than CTAs, against the FMA or the velocity-split kernel.

Tolerances as for the grouped forms: the FP32 forms do the same arithmetic in
another order, a value a sum of about 5 Np products of relative rounding 2^-24 per
stage; BF16 within a few storage units of the element's largest deviation."""
import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n,p,nx,ny,kind", [("fp32", 33, 5, 13, 12, "cavity"), ("fp32", 33, 3, 2, 3, "couette"),
                                                 ("fp32", 24, 2, 14, 11, "cavity"), ("bf16", 33, 4, 3, 2, "cavity"),
                                                 ("bf16", 24, 3, 15, 13, "couette"), ("fp32", 32, 4, 1, 1, "cavity")])
def test_wide_form_matches_other_forms(prec, n, p, nx, ny, kind):
    from paper_2012_13487_gb300 import fedbm as fb
    c = (cases.cavity if kind == "cavity" else cases.couette)(nx, ny, p, velset=("nc", n), kn=1.0)
    s = cases.solver(c, prec)
    ref = cases.solver(c, prec, vsplit=4) if n == 33 and p == 5 else cases.solver(c, prec, stages=1, epc=1, tpb=128)
    assert s.info.pipeline_stages == 3 and s.info.velocity_split == 1 and ref.info.pipeline_stages != 3
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
        w = fb.fedbm_velset(fb.velset_desc(fb.VELSET_NC, n))[2]
        md = np.abs(out[1] / w - 1).max(axis=(1, 2), keepdims=True)
        assert (np.abs(out[0] - out[1]) <= 4 * 2.0 ** -8 * w * md).all()


def test_few_elements_keep_the_velocity_split():
    s = cases.solver(cases.cavity(2, 2, 5, velset=("nc", 33), kn=1.0), "fp32")
    assert s.info.velocity_split >= 2
