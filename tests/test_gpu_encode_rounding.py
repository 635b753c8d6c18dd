"""The 16-bit deviation codes are rounded from (f - w) / w in at least FP32: near the ties of
the code grid, where an error in front of the rounding shows, a code is off by at most
half a spacing plus what rounding the exact quotient to FP32 first adds.

Bound: with t significant bits (8 BF16, 11 FP16) and 2^e <= |d| < 2^(e+1), the spacing is
2^(e+1-t); an FP32 rounding of d moves it by at most 2^(e-24), which is 2^(t-25) spacings
(FP16 codes below 2^-14 of the scale are spaced 2^-24 of it).  The decoded value carries
one FP64 FMA: below 2^-30 spacings here.  The FP64 quotient rounded to FP32 keeps the
bound; a difference and a product in plain FP32 (3 to 4 units of 2^-24) did not."""
import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,t", [("bf16", 8), ("fp16", 11)])
@pytest.mark.parametrize("velset,p", [(("gh", 4), 3), (("nc", 16), 2), (("nc", 16), 4), (("nc", 33), 5),
                                      (("gh", 40), 1)])  # the last: weights below 2^-96 take the FP64 quotient
@pytest.mark.parametrize("wide", [False, True])
def test_codes_near_ties(prec, t, velset, p, wide):
    import torch

    from paper_2012_13487_gb300 import fedbm as fb
    c = cases.cavity(6, 5, p, velset=velset, nc_sqrt2=velset[1] == 33)
    s = cases.solver(c, prec)
    K, Np, Q = s.shape
    w = fb.fedbm_velset(s_vd(fb, c))[2]
    rng = np.random.default_rng(7 + p)
    # ties of the grid of elements whose largest deviation lies in [0.5, 1): odd multiples of half
    # a spacing, some octaves below the largest as well
    e = rng.integers(-4, 0, (K, Np, Q))
    d = (2.0 ** (t - 1) + rng.integers(0, 2 ** (t - 1), e.shape) + 0.5) * 2.0 ** (e + 1.0 - t)
    d *= rng.choice([-1.0, 1.0], e.shape)
    d[:, 0, 0] = 0.75
    f = w * (1.0 + d * (1.0 + (2.0 ** -24 * rng.uniform(-4, 4, e.shape) if wide else 0.0)))
    if not wide:
        f = f.astype(np.float32)
    ok = np.broadcast_to(w > (0.0 if wide else 2.0 ** -100), f.shape)  # FP32 holds the value to 24 bits
    src = torch.from_numpy(f).cuda()
    (fb.fedbm_set_state if wide else fb.fedbm_set_state_f32)(s.h, src, True)
    out = torch.empty(f.shape, dtype=torch.float64, device="cuda")
    fb.fedbm_get_state(s.h, out, True)
    g, f = out.cpu().numpy().astype(np.longdouble), f.astype(np.longdouble)
    wl = w.astype(np.longdouble)
    exact, got = (f - wl) / wl, (g - wl) / wl
    m = np.abs(np.where(ok, exact, 0)).max(axis=(1, 2), keepdims=True).astype(np.float64)
    spacing = 2.0 ** (np.floor(np.log2(np.maximum(np.abs(exact), 1e-300).astype(np.float64))) + 1 - t)
    if prec == "fp16":
        spacing = np.maximum(spacing, 2.0 ** (np.floor(np.log2(m)) + 1 - 15) * 2.0 ** -24)
    worst = float(np.where(ok, np.abs(got - exact) / spacing, 0).max())
    print("%s %s p=%d wide=%d: %.7f spacings" % (prec, velset, p, wide, worst))
    assert worst <= 0.5 + 2.0 ** (t - 25) * (1 + 2.0 ** -10) + 2.0 ** -30
    s.close()


def s_vd(fb, c):
    kind, n = c["velset"]
    return fb.velset_desc(fb.VELSET_GH if kind == "gh" else fb.VELSET_NC, n, nc_sqrt2=int(c.get("nc_sqrt2", False)))
