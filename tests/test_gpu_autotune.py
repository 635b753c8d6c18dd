"""The tile autotuner never loses to the library's own choice: that choice is timed among
the candidates of the same run, so the kept time is at most its time, on shapes whose
automatic tile is not in the candidates' grid (one-warp CTAs at 16 velocities, FP64
elements split over four warps, the warp-specialised form)."""
import json

import pytest

import cases

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c,prec", [(cases.couette(8, 8, 2, velset=("gh", 4)), "fp64"),
                                    (cases.couette(40, 40, 3, velset=("gh", 4)), "fp32"),
                                    (cases.couette(40, 40, 1, velset=("gh", 4)), "fp16"),
                                    (cases.cavity(6, 5, 3, velset=("gh", 6)), "fp32"),
                                    (cases.cavity(6, 5, 3, velset=("nc", 16)), "bf16")])
def test_kept_tile_is_no_slower_than_the_default(tmp_path, c, prec):
    s = cases.solver(c, prec)
    path = tmp_path / "tune.json"
    s.set_equilibrium(1.0, 0.01, 0.0, 1e-3, 3)
    s.autotune(str(path), 4)
    (entry,) = json.loads(path.read_text()).values()
    assert 0 < entry["us"] <= entry["auto_us"]
    kept = (s.info.elems_per_cta, s.info.threads_per_cta, s.info.pipeline_stages)
    # a second solver takes the entry from the file
    t = cases.solver(c, prec)
    before = path.read_text()
    t.autotune(str(path), 4)
    assert (t.info.elems_per_cta, t.info.threads_per_cta, t.info.pipeline_stages) == kept
    assert path.read_text() == before


def test_entries_of_other_kernels_are_timed_again(tmp_path):
    """A cache written by an earlier generation of the kernels (no such tag in its keys)
    is kept in the file but not used."""
    c = cases.couette(8, 8, 2, velset=("gh", 4))
    s = cases.solver(c, "fp64")
    path = tmp_path / "tune.json"
    s.autotune(str(path), 2)
    (key,) = json.loads(path.read_text())
    gen = next(x for x in key.split("|") if x.startswith("gen"))
    old = key.replace(gen + "|", "")
    path.write_text('{\n"%s": {"epc": 32, "tpb": 64, "stages": 1, "tc": 0, "ncl": 0, "us": 1.000}\n}\n' % old)
    t = cases.solver(c, "fp64")
    t.autotune(str(path), 2)
    entries = json.loads(path.read_text())
    assert set(entries) == {old, key} and t.info.elems_per_cta != 32
