"""The tile rules (csrc/tile_rule.h) are functions of the sizes and the device's SM count:
on 152 SMs they give the tiles that were measured there, on another count the tiles of
the same elements per SM.  Automatic tiles take two velocities per thread."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2012_13487_gb300", "csrc")
PROGRAM = r"""
#include "tile_rule.h"
#include <cstdio>
int main() {
  int p, store, Qp, nsm, epc, tpb;
  long long K;
  while (std::scanf("%d %d %d %lld %d %d %d", &p, &store, &Qp, &K, &nsm, &epc, &tpb) == 7) {
    fedbm::TileShape s;
    s.p = p; s.store = store; s.Qp = Qp; s.K = K; s.nsm = nsm;
    if (tpb == 0) fedbm::auto_tile(s, &epc, &tpb);
    std::printf("%d %d %d\n", epc, tpb, fedbm::stage_lanes(s, epc, tpb));
  }
}
"""
F64, F32, BF16, F16 = 0, 1, 2, 3


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("rule")
    (d / "rule.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-Wall", "-I" + CSRC, str(d / "rule.cpp"), "-o", str(d / "rule")], check=True)

    def run(rows):
        text = "\n".join(" ".join(str(v) for v in r) for r in rows)
        out = subprocess.run([str(d / "rule")], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(int(v) for v in line.split()) for line in out.splitlines()]
    return run


def measured(p, store, Qp, K):
    """The rule as it was measured on 152 SMs."""
    f64, few, spread = store == F64, K < 2432, min(4, (K + 303) // 304)
    if Qp == 16 and f64:
        return (8 if not few else 1 if K <= 304 else 2), (128 if not few or K <= 608 else 64 if K <= 1216 else 32)
    if Qp == 16:
        epc = spread if few else 4 if K < 32768 else 8 if p <= 3 else 4
        if K >= 32768 and p == 1 and store >= BF16:
            epc = 16
        return epc, 32 * spread if few else 32
    epc = max(1, 128 // Qp)
    if Qp < 128 and not f64:
        epc = min(epc, spread) if few else epc
        return epc, min(128, 64 * epc) if few else 32 if p <= 2 and K >= 9728 else 64
    items = epc * Qp // (1 if f64 else 2)
    if not f64 and items >= 512 and (p >= 3 or (p == 2 and items > 512)):
        return epc, 256
    return epc, min(128, max(32, (items + 31) // 32 * 32))


SIZES = [1, 2, 151, 303, 304, 305, 607, 608, 609, 912, 1215, 1216, 1217, 2431, 2432, 2433, 9727, 9728, 32767, 32768,
         400000]


def test_rule_on_152_sms(rule):
    rows = [(p, st, Qp, K, 152, 0, 0) for p in range(7) for st in (F64, F32, BF16, F16)
            for Qp in (8, 16, 24, 32, 40, 64, 72, 88, 120, 128, 144, 256, 576, 1024, 1120, 1600) for K in SIZES]
    for r, (epc, tpb, lanes) in zip(rows, rule(rows)):
        assert (epc, tpb) == measured(*r[:4]), r
        assert lanes == 2, r  # FP64 has one by its own kernel; the number is not used there


def test_rule_follows_the_sm_count(rule):
    """Twice the SMs and twice the elements: the same tile (below the size where more
    elements per tile pay whatever the device)."""
    rows = [(p, st, Qp, K, 152, 0, 0) for p in (1, 4) for st in (F64, F32, F16) for Qp in (16, 40, 256)
            for K in SIZES if K < 16000]
    twice = [(p, st, Qp, 2 * K, 304, e, t) for p, st, Qp, K, _, e, t in rows]
    assert rule(rows) == rule(twice)
    assert not re.search(r"\b(152|304|608|1216|303)\b", re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "tile_rule.h")).read()))


@pytest.mark.parametrize("store", [F32, BF16, F16])
def test_one_velocity_per_thread_where_threads_would_idle(rule, store):
    got = rule([(5, store, 256, 5000, 152, 1, 256), (5, store, 256, 5000, 152, 1, 128),  # a thread per value, per pair
                (5, store, 16, 5000, 152, 8, 128), (5, store, 16, 5000, 152, 8, 64),
                (3, store, 40, 5000, 152, 4, 128), (3, store, 40, 5000, 152, 3, 64),      # a warp without a pair; none
                (3, store, 40, 500, 152, 4, 128), (3, store, 40, 500, 152, 1, 64),        # few elements
                (3, store, 40, 300, 152, 1, 64)])
    assert [g[2] for g in got] == [1, 2, 1, 2, 1, 2, 2, 1, 2]
