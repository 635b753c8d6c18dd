"""The warp-specialised forms that the automatic choice takes (one consumer group with 256
velocities, three with 1,024, the wide form above): every option of the stage against the
FMA kernel, and the bounded waits.

Both kernels do the same FP32 arithmetic in another order: a value is a sum of about 5 Np
products of relative rounding 2^-24, five stages per step, so they differ by at most 5 Np
2^-24 per stage of the largest value; BF16 by a few storage units of the element's largest
deviation (also with stochastic rounding, whose draws depend on the value's index, the
step and the stage only)."""
import time

import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu

ADVECTION = dict(bc=("periodic",) * 4, wall_u=((0, 0),) * 4, collision=False)
#          set           p  more
FORMS = [(("nc", 16), 3), (("nc", 32), 2), (("nc", 24), 3)]
OPTIONS = {"third order": lambda v, p: cases.couette(4, 5, p, velset=v, eq_order=3, kn=0.5),
           "advection": lambda v, p: dict(nx=4, ny=5, p=p, velset=v, **ADVECTION),
           "eq walls": lambda v, p: dict(cases.cavity(5, 4, p, velset=v), bc=("eq",) * 4),
           "central": lambda v, p: dict(cases.couette(4, 5, p, velset=v), beta=0.5),
           "unstructured": lambda v, p: cases.unstructured(cases.cavity(0, 0, p, velset=v, kn=2.0), 5, 4),
           "fp64": lambda v, p: cases.cavity(5, 4, p, velset=v),
           "comp": lambda v, p: cases.cavity(5, 4, p, velset=v),
           "rounding": lambda v, p: cases.cavity(5, 4, p, velset=v)}


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("option", list(OPTIONS))
@pytest.mark.parametrize("velset,p", FORMS)
def test_options_match_fma_kernel(velset, p, option, prec):
    if option == "rounding" and prec == "fp32":
        pytest.skip("FP32 state has no stochastic rounding")
    c = OPTIONS[option](velset, p)
    red = option if option in ("fp64", "comp") else "default"
    kw = dict(rounding=1) if option == "rounding" else {}
    out = []
    for tile in ({}, dict(stages=1, epc=1, tpb=128)):
        s = cases.solver(c, prec, red, **tile, **kw)
        assert (s.info.pipeline_stages == 3) == (not tile)
        s.set_equilibrium(1.0, 0.02, -0.01, 0.05, 9)
        s.step(2)
        out.append(s.state())
        s.close()
    Np = (p + 1) * (p + 2) // 2
    if prec == "fp32":
        assert np.abs(out[0] - out[1]).max() <= 10 * 5 * Np * 2.0 ** -24 * np.abs(out[1]).max()
    else:
        w = cases.oracle_problem(c).w
        md = np.abs(out[1] / w - 1).max(axis=(1, 2), keepdims=True)
        assert (np.abs(out[0] - out[1]) <= 4 * 2.0 ** -8 * w * md).all()


@pytest.mark.parametrize("prec,velset,p", [("fp32", ("nc", 16), 2), ("bf16", ("nc", 16), 4), ("fp32", ("nc", 32), 1),
                                           ("fp32", ("nc", 32), 3),   # two ring stages for three groups
                                           ("bf16", ("nc", 32), 3), ("fp32", ("nc", 33), 4), ("bf16", ("nc", 24), 3)])
def test_wait_timeout_is_reported_and_the_context_usable(prec, velset, p):
    """16 expected bytes that never arrive: every group's bounded wait runs out (on the
    copies, or on its element's number in the stage), the producer's on the release too, all
    leave, and the host reads FEDBM_ETIMEOUT.  The next solver steps as usual."""
    from paper_2012_13487_gb300 import fedbm as fb
    c = cases.cavity(20, 20, p, velset=velset, kn=1.0)
    s = cases.solver(c, prec, test_wait_timeout=1)
    assert s.info.pipeline_stages == 3
    s.set_equilibrium(1.0, 0.0, 0.0, 1e-3, 5)
    t0 = time.time()
    s.stage(0)
    with pytest.raises(fb.FedbmError) as e:
        s.mass()
    assert e.value.code == fb.FEDBM_ETIMEOUT and time.time() - t0 < 30.0
    s.close()
    g = cases.solver(c, prec)
    g.set_equilibrium(1.0, 0.0, 0.0, 1e-3, 5)
    m = g.mass()
    g.step(2)
    assert abs(g.mass() - m) <= 1e-4 * abs(m) * (1 if prec == "fp32" else 10)
    g.close()
