"""Encode, decode and moment kernels at the edges of their work split: elements
of one warp and of one CTA, rows staged in several passes, padded and odd
velocity counts, groups of 1 to 32 lanes per node, device pointers with only
the alignment of one value.

Bounds: FP64 and FP32 state round-trip exactly.  A deviation code of t
significant bits (8 for BF16, 11 for FP16) is the exact deviation d = (f - w)/w
rounded to within half its spacing, 2^(floor(log2 |d|) + 1 - t) / 2 whatever the
power-of-two scale (FP16 codes below 2^-14, 2^-29 of the element's largest, have
the spacing 2^-24 of the scale); the FP32 difference and product in front of the
rounding add at most 3 2^-24 |d|, less than 2^-10 of a spacing.  A sum of
Q products in a precision of unit roundoff u is off by at most Q u times the
sum of their magnitudes, whatever the order."""
import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu

#        set           p  precisions
SHAPES = [(("gh", 3), 0, ("fp64", "fp32", "bf16", "fp16")),   # 9 velocities padded to 16, one node
          (("gh", 4), 5, ("fp64", "fp32", "bf16", "fp16")),   # a warp per element
          (("gh", 5), 4, ("fp32", "bf16")),                   # 25 padded to 32
          (("nc", 16), 2, ("fp32", "bf16")),                  # the largest element of a warp
          (("nc", 16), 3, ("fp64", "fp32", "fp16")),          # a CTA per element
          (("nc", 33), 5, ("fp32", "bf16", "fp16"))]          # rows in several passes


@pytest.mark.parametrize("velset,p,prec", [(v, p, x) for v, p, ps in SHAPES for x in ps])
def test_round_trip_and_moments(velset, p, prec):
    import torch

    from paper_2012_13487_gb300 import fedbm as fb
    c = cases.cavity(5, 3, p, velset=velset, nc_sqrt2=velset[1] == 33)
    pr = cases.oracle_problem(c)
    f = cases.initial_state(pr, amp=2e-2, seed=5, ux0=0.05)
    wide = prec == "fp64"
    if not wide:
        f = f.astype(np.float32)
    s = cases.solver(c, prec)
    src = torch.zeros(f.size + 1, dtype=torch.float64 if wide else torch.float32, device="cuda")
    src[1:] = torch.from_numpy(f.ravel())
    out = torch.zeros(f.size + 1, dtype=torch.float64, device="cuda")
    (fb.fedbm_set_state if wide else fb.fedbm_set_state_f32)(s.h, src[1:], True)
    fb.fedbm_get_state(s.h, out[1:], True)
    g = out[1:].cpu().numpy().reshape(f.shape)
    f = f.astype(np.float64)
    if prec in ("fp64", "fp32"):
        assert np.array_equal(g, f)
    else:
        d = f / pr.w - 1
        t = 8 if prec == "bf16" else 11
        spacing = 2.0 ** (np.floor(np.log2(np.maximum(np.abs(d), 1e-300))) + 1 - t)
        if prec == "fp16":
            scale = 2.0 ** (np.floor(np.log2(np.abs(d).max(axis=(1, 2), keepdims=True))) + 1 - 15)
            spacing = np.maximum(spacing, scale * 2.0 ** -24)
        assert (np.abs(g / pr.w - 1 - d) <= (0.5 + 2.0 ** -10) * spacing + 1e-15).all()
    # the moments are those of the stored state
    rho, ux, uy = s.moments()
    u = 2.0 ** -53 if wide else 2.0 ** -24
    q = pr.Q + 4
    r0, j = g.sum(-1), [(g @ e, np.abs(g) @ np.abs(e)) for e in (pr.ex, pr.ey)]
    assert (np.abs(rho - r0) <= q * u * np.abs(g).sum(-1)).all()
    for v, (jx, ja) in zip((ux, uy), j):
        assert (np.abs(v * r0 - jx) <= 2 * q * u * (ja + np.abs(jx))).all()
