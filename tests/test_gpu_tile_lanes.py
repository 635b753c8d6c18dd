"""The FMA kernel with one velocity per thread (tiles that have a thread for every value)
against its form with two: every operation rounds a value the same way in both, and below
128 velocities the sums over a row have one order whatever the tile, so the states agree bit
for bit.  From 128 up the moment sums of 256 and 128 threads differ in order: FP32 within
15 5 Np 2^-24 of the largest value over three steps (a value is a sum of about 5 Np products a
stage), the 16-bit forms within a few storage units of the element's largest deviation."""
import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu

# 338 elements: more than two per SM, so that one-element tiles take one velocity per thread
CASES = [(cases.couette(13, 13, 2, velset=("gh", 4)), (1, 32), (2, 32)),
         (cases.cavity(13, 13, 5, velset=("gh", 4), kn=0.5), (1, 64), (4, 32)),
         (cases.cavity(13, 13, 3, velset=("gh", 6), eq_order=3), (1, 64), (3, 32)),
         (dict(cases.cavity(13, 13, 1, velset=("gh", 5)), bc=("eq",) * 4, beta=0.5), (1, 32), (4, 64)),
         (dict(nx=13, ny=13, p=4, velset=("gh", 6), bc=("periodic",) * 4, wall_u=((0, 0),) * 4, collision=False),
          (1, 96), (2, 32)),
         (cases.unstructured(cases.cavity(0, 0, 2, velset=("gh", 4), kn=2.0), 13, 13), (1, 32), (8, 64)),
         (cases.couette(36, 35, 3, velset=("gh", 4)), (8, 128), (8, 64)),
         (cases.cavity(13, 13, 0, velset=("nc", 16)), (1, 256), (1, 128)),
         (cases.cavity(13, 13, 3, velset=("nc", 16)), (1, 256), (1, 128)),
         (cases.couette(13, 13, 6, velset=("gh", 4)), (1, 32), (2, 32))]


@pytest.mark.parametrize("prec,rounding", [("fp32", 0), ("bf16", 0), ("bf16", 1), ("fp16", 0)])
@pytest.mark.parametrize("j", range(len(CASES)))
def test_one_and_two_velocities_per_thread_agree(j, prec, rounding):
    c, one, two = CASES[j]
    out = []
    for stages, (epc, tpb) in ((1, one), (1, two), (2, one)):
        s = cases.solver(c, prec, epc=epc, tpb=tpb, stages=stages, rounding=rounding)
        s.set_equilibrium(1.0, 0.02, -0.01, 0.05, 9)
        s.step(3)
        out.append(s.state())
        Q = s.info.Q_padded
        s.close()
    assert np.array_equal(out[0], out[2])  # one or two tile buffers
    if Q < 128:
        assert np.array_equal(out[0], out[1])
    elif prec == "fp32":
        Np = (c["p"] + 1) * (c["p"] + 2) // 2
        assert np.abs(out[0] - out[1]).max() <= 15 * 5 * Np * 2.0 ** -24 * np.abs(out[1]).max()
    else:
        w = cases.oracle_problem(c).w
        md = np.abs(out[1] / w - 1).max(axis=(1, 2), keepdims=True)
        u = 2.0 ** -8 if prec == "bf16" else 2.0 ** -11
        assert (np.abs(out[0] - out[1]) <= 4 * u * w * md).all()


@pytest.mark.parametrize("c", [cases.couette(13, 13, 2, velset=("gh", 4)), cases.cavity(13, 13, 3, velset=("gh", 4))])
def test_one_velocity_per_thread_matches_the_oracle(c):
    pr = cases.oracle_problem(c)
    f0 = cases.initial_state(pr, amp=0.05, seed=31)
    s = cases.solver(c, "fp32", epc=1, tpb=32, stages=1)
    s.set_state(f0)
    s.step(4)
    assert cases.rel_max_err(s.state(), pr.run(f0, 4)) <= 4.0 * pr.Np * 2.0 ** -24 * np.sqrt(20) + 2.0 ** -24
