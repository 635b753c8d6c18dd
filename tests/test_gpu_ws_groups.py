"""The warp-specialised stage kernel with several consumer groups on one ring: its
1,024-velocity form (three groups; two ring stages at degree 3 in FP32, up to
twelve at degree 1) and the two-group form of 256 velocities, on fewer and more
elements than the CTAs hold, against the FMA kernel.

Both do the same FP32 arithmetic in another order: a value is a sum of about 5 Np
products of relative rounding 2^-24 (contractions, lift, collision), five stages
per step, so they differ by at most 5 Np 2^-24 per stage of the largest value; BF16
to a few storage units of the element's largest deviation (2^-8 each), since an
encode that rounds the other way carries into the next stage."""
import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("n,p,nx,ny", [(32, 1, 3, 5), (32, 2, 16, 15), (32, 3, 1, 1), (32, 3, 17, 19),
                                       (16, 4, 1, 1), (16, 4, 21, 23), (16, 5, 19, 12)])
def test_groups_match_fma_kernel(prec, n, p, nx, ny):
    c = cases.cavity(nx, ny, p, velset=("nc", n), kn=1.0)
    # 1,024 velocities: the automatic choice; 256: two groups, asked for by number
    s = cases.solver(c, prec, stages=3 if n == 16 else 0)
    ref = cases.solver(c, prec, stages=1, epc=1, tpb=128)
    assert s.info.pipeline_stages == 3 and ref.info.pipeline_stages == 1
    out = []
    for x in (s, ref):
        x.set_equilibrium(1.0, 0.02, -0.01, 0.05, 9)
        x.step(3)
        out.append(x.state())
        x.close()
    Np = (p + 1) * (p + 2) // 2
    if prec == "fp32":
        assert np.abs(out[0] - out[1]).max() <= 15 * 5 * Np * 2.0 ** -24 * np.abs(out[1]).max()
    else:
        from paper_2012_13487_gb300 import fedbm as fb
        w = fb.fedbm_velset(fb.velset_desc(fb.VELSET_NC, n))[2]
        md = np.abs(out[1] / w - 1).max(axis=(1, 2), keepdims=True)
        assert (np.abs(out[0] - out[1]) <= 4 * 2.0 ** -8 * w * md).all()
