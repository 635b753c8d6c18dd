"""The even-odd operator tables of the FMA stage kernels (csrc/stage_eo.cuh):
the committed FP32 tables equal the library's operators split and rounded, bit
for bit, and the split contraction reproduces Dr, Ds and LIFT.

Rounding each coefficient to FP32 moves a sum of n products by at most 2^-24
times the sum of their magnitudes; halving and adding the parts takes at most
four roundings more, in FP64 here."""
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
INC = os.path.join(ROOT, "paper_2012_13487_gb300", "csrc", "ops_tables.inc")


def committed(p):
    text = open(INC).read()
    m = re.search(r"FEDBM_P == %d\n.*?#define FEDBM_EO32_TABLE \\\n(.*?)(?=\n#)" % p, text, re.S)
    return np.array([float.fromhex(v) for v in re.findall(r"(-?0x[0-9a-f.]+p[+-]\d+)f", m.group(1))],
                    dtype=np.float32)


@pytest.mark.parametrize("p", range(6))
def test_table_and_split(p):
    from paper_2012_13487_gb300 import fedbm as fb
    from paper_2012_13487_gb300.csrc import gen_ops_tables as gen
    t = committed(p)
    assert np.array_equal(t, np.array(gen.eo_table(p), dtype=np.float32))
    o = fb.fedbm_ref_operators(p)
    pr, n, Np = gen.pairs(p), p + 1, (p + 1) * (p + 2) // 2
    assert sorted({x for ab in pr for x in ab}) == list(range(Np))
    ne, no = len(pr), sum(a != b for a, b in pr)
    f1e, f1o = p // 2 + 1, (p + 1) // 2
    nle, nlo = n + f1e, n + f1o
    sizes = [(ne, ne), (no, no), (no, ne), (ne, no), (ne, nle), (no, nlo)]
    parts = np.split(t.astype(np.float64), np.cumsum([a * b for a, b in sizes])[:-1])
    se, so, de, do, le, lo = (x.reshape(s) for x, s in zip(parts, sizes))
    # the kernel leaves out what D reads from off the face r + s = 0 at that face's nodes
    hyp = np.array([a in o["fmask"][1] for a, _ in pr])
    do[np.ix_(hyp, ~hyp[:no])] = 0.0
    de[np.ix_(hyp[:no], ~hyp)] = 0.0
    rng = np.random.default_rng(p)
    f, flux, ar, as_ = rng.standard_normal(Np), rng.standard_normal(3 * n), 0.7, -1.3
    a, b = np.array(pr).T
    E = np.where(a == b, f[a], f[a] + f[b])
    O = (f[a] - f[b])[:no]
    g = np.concatenate([flux[:n] + flux[2 * n:], [flux[n + j] + (flux[n + p - j] if j != p - j else 0) for j in range(f1e)]])
    h = np.concatenate([flux[:n] - flux[2 * n:], [flux[n + j] - flux[n + p - j] for j in range(f1o)]])
    oe = -0.5 * (ar + as_) * (se @ E) + 0.5 * (ar - as_) * (do @ O) + le @ g
    oo = -0.5 * (ar + as_) * (so @ O) + 0.5 * (ar - as_) * (de @ E) + lo @ h
    got = np.zeros(Np)
    got[a] = oe
    got[a[:no]] = oe[:no] + oo
    got[b[:no]] = oe[:no] - oo
    want = -(ar * o["Dr"] + as_ * o["Ds"]) @ f + o["LIFT"] @ flux
    size = (abs(ar) + abs(as_)) * (np.abs(o["Dr"]) + np.abs(o["Ds"])).max() * np.abs(f).sum() \
        + np.abs(o["LIFT"]).max() * np.abs(flux).sum()
    assert np.abs(got - want).max() <= (2.0 ** -24 + 8 * 2.0 ** -53) * 2 * size
