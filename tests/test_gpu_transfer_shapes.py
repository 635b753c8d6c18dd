"""Loads, read-outs and moments where their kernels change: the direct and the staged ones
(few values, tiny elements, elements of 1,024 to 1,536 values, many values), elements by warps
and by CTAs, one and four nodes per group of lanes, and cases of different element counts in
one batch.  FP64 and FP32 state round-trip exactly; a deviation code is within half its
spacing, 2^-8 (BF16) or 2^-11 (FP16) of the value, plus 2^-14 of that; the moments are the sums
of the stored state to Q + 4 roundings of the state's compute precision."""
import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu

#         set           p  cells (2 cells^2 elements each side of a line)
SHAPES = [(("gh", 3), 0, 5), (("gh", 3), 0, 60), (("gh", 4), 0, 35), (("gh", 4), 2, 20), (("gh", 4), 5, 3),
          (("gh", 4), 5, 40), (("gh", 6), 3, 24), (("gh", 5), 6, 8), (("nc", 16), 2, 5), (("nc", 16), 2, 60),
          (("nc", 16), 4, 9), (("nc", 16), 4, 28), (("nc", 32), 3, 4), (("nc", 33), 5, 2)]


def check(pr, prec, f, g, rho, ux, uy):
    if prec in ("fp64", "fp32"):
        assert np.array_equal(g, f)
    else:
        d = f / pr.w - 1
        md = np.abs(d).max(axis=(1, 2), keepdims=True)
        u = 2.0 ** -8 if prec == "bf16" else 2.0 ** -11
        floor = 0.0 if prec == "bf16" else 2.0 ** -39 * md  # half the smallest FP16 code of the scale
        assert (np.abs(g / pr.w - 1 - d) <= np.maximum(np.abs(d) * u * (1 + 2.0 ** -13), floor) + 1e-15).all()
    u, q = 2.0 ** -53 if prec == "fp64" else 2.0 ** -24, pr.Q + 4
    r0 = g.sum(-1)
    assert (np.abs(rho - r0) <= q * u * np.abs(g).sum(-1)).all()
    for v, e in ((ux, pr.ex), (uy, pr.ey)):
        jx, ja = g @ e, np.abs(g) @ np.abs(e)
        assert (np.abs(v * r0 - jx) <= 2 * q * u * (ja + np.abs(jx))).all()


@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16", "fp16"])
@pytest.mark.parametrize("velset,p,n", SHAPES)
def test_round_trip_and_moments(velset, p, n, prec):
    if prec == "fp64" and velset == ("nc", 33):
        pytest.skip("no FP64 tile of one CTA at this size")
    c = cases.cavity(n, n, p, velset=velset, nc_sqrt2=velset[1] == 33)
    pr = cases.oracle_problem(c)
    f = cases.initial_state(pr, amp=2e-2, seed=5, ux0=0.05)
    if prec != "fp64":
        f = f.astype(np.float32).astype(np.float64)
    s = cases.solver(c, prec)
    s.set_state(f)
    check(pr, prec, f, s.state(), *s.moments())
    s.close()


@pytest.mark.parametrize("prec", ["bf16", "fp32"])
def test_cases_of_one_group_with_few_and_many_elements(prec):
    """One group (same sizes, so the same kernels' limits), element counts on both sides of the
    line between a warp and a CTA per element."""
    cs = [cases.cavity(n, n, 2, velset=("nc", 16), kn=1.0) for n in (40, 4, 30, 2)]
    b = cases.batch(cs, prec)
    assert len({b.info(j).group for j in range(4)}) == 1
    prs = [cases.oracle_problem(c) for c in cs]
    fs = [cases.initial_state(pr, amp=2e-2, seed=j).astype(np.float32).astype(np.float64) for j, pr in enumerate(prs)]
    for j, f in enumerate(fs):
        b.set_state(j, f)
    for j, (pr, f) in enumerate(zip(prs, fs)):
        check(pr, prec, f, b.state(j), *b.moments(j))
    b.close()
