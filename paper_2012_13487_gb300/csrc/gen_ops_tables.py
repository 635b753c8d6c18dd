"""Writes ops_tables.inc: the FP32 Dr, Ds and LIFT operators of degrees 0..5 and
their even and odd parts (stage_eo.cuh) as compile-time tables for the FMA
stage kernels.

The nodal Lagrange basis of Sec. II.B.1 lives on one reference triangle, so
Dr, Ds and LIFT depend only on the degree (and on the node set, which the paper
leaves open: warp & blend nodes with alpha = 0 here).  The FP32 kernels can
therefore take them as instruction immediates instead of loading them from
constant memory.  The values are the library's own operators
(``fedbm_ref_operators``) rounded to FP32 exactly as the runtime upload rounds
them; a CPU test checks that the committed file still matches.  Every kernel of
degree <= 5 that computes in FP32 takes the even and odd parts; degree 6 (784
entries per derivative matrix) keeps constant memory.  Run as
``python -m paper_2012_13487_gb300.csrc.gen_ops_tables`` after a build.
"""
import os

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
OUT = os.path.join(HERE, "ops_tables.inc")
MAX_P = 5


def table(p):
    from paper_2012_13487_gb300 import fedbm as fb
    o = fb.fedbm_ref_operators(p)
    vals = np.concatenate([o["Dr"].ravel(), o["Ds"].ravel(), o["LIFT"].ravel()])
    return [float(np.float32(v)) for v in vals]


def pairs(p):
    """Nodes exchanged by r <-> s as (a, b), those off the axis first (eo_pairs in stage_eo.cuh)."""
    def node(row, col):
        return row * (p + 1) - row * (row - 1) // 2 + col
    ij = [(i, j) for j in range(p + 1) for i in range(j + 1) if i + j <= p]
    return [(node(j, i), node(i, j)) for i, j in ij if i != j] + [(node(i, i), node(i, i)) for i, j in ij if i == j]


def eo_table(p):
    """Se, So, De, Do, Le, Lo in the order and with the arithmetic of eo_coefficients."""
    from paper_2012_13487_gb300 import fedbm as fb
    o = fb.fedbm_ref_operators(p)
    pr = pairs(p)
    n = p + 1
    no = sum(a != b for a, b in pr)
    ne = len(pr)
    nle, nlo = n + p // 2 + 1, n + (p + 1) // 2
    se, so, de, do = np.zeros((ne, ne)), np.zeros((no, no)), np.zeros((no, ne)), np.zeros((ne, no))
    le, lo = np.zeros((ne, nle)), np.zeros((no, nlo))
    for q, (a, _) in enumerate(pr):
        s, d, lift = o["Ds"][a] + o["Dr"][a], o["Ds"][a] - o["Dr"][a], o["LIFT"][a]
        for m, (x, y) in enumerate(pr):
            se[q, m] = s[x] if x == y else 0.5 * (s[x] + s[y])
            if q < no:
                de[q, m] = d[x] if x == y else 0.5 * (d[x] + d[y])
            if m < no:
                do[q, m] = 0.5 * (d[x] - d[y])
                if q < no:
                    so[q, m] = 0.5 * (s[x] - s[y])
        for j in range(n):
            le[q, j] = 0.5 * (lift[j] + lift[2 * n + j])
            if q < no:
                lo[q, j] = 0.5 * (lift[j] - lift[2 * n + j])
        for j in range(p // 2 + 1):
            k = p - j
            le[q, n + j] = lift[n + j] if j == k else 0.5 * (lift[n + j] + lift[n + k])
            if q < no and j < (p + 1) // 2:
                lo[q, n + j] = 0.5 * (lift[n + j] - lift[n + k])
    return [float(np.float32(v)) for v in np.concatenate([x.ravel() for x in (se, so, de, do, le, lo)])]


def macro(name, vals):
    lines = ["#define %s \\" % name]
    for i in range(0, len(vals), 4):
        chunk = ", ".join(v.hex() + "f" for v in vals[i:i + 4])
        lines.append("  %s%s \\" % (chunk, "," if i + 4 < len(vals) else ""))
    lines[-1] = lines[-1][:-2]
    return lines


def render():
    lines = ["// Generated by gen_ops_tables.py from the library's operators: FP32 Dr, Ds",
             "// (row-major Np x Np) and LIFT (row-major Np x 3(p+1)) of the FEDBM_P of the",
             "// including translation unit, and Se, So, De, Do, Le, Lo of stage_eo.cuh, in the",
             "// order of the runtime upload.  The kernels take the second table; the first is the",
             "// one a test holds against the library's operators.  Do not edit."]
    for p in range(MAX_P + 1):
        lines.append("#%s FEDBM_P == %d" % ("if" if p == 0 else "elif", p))
        lines += macro("FEDBM_OPS32_TABLE", table(p)) + macro("FEDBM_EO32_TABLE", eo_table(p))
    lines.append("#endif")
    return "\n".join(lines) + "\n"


if __name__ == "__main__":
    with open(OUT, "w") as f:
        f.write(render())
    print(OUT)
