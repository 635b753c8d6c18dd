"""Consecutive stages of a small mesh are on the GPU together (programmatic launch): the
state after many steps equals, bit for bit, the state of the same stages run one launch
at a time with the stream drained between them.  FP16 deviation state forms new element
scales at every stage, so a stale scale would decode a whole element or face wrongly;
BF16 goes through the warp-specialised (256 velocities), the wide (576), the FMA (16) and the
velocity-split forms."""
import numpy as np
import pytest

import cases

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,velset,p,tile", [("fp16", ("gh", 4), 2, {}), ("fp16", ("nc", 16), 3, {}),
                                                ("fp16", ("gh", 6), 1, {}), ("bf16", ("gh", 4), 3, {}),
                                                ("bf16", ("nc", 16), 2, {}), ("bf16", ("nc", 24), 3, {}),
                                                ("bf16", ("nc", 16), 3, dict(vsplit=2)),
                                                ("fp32", ("nc", 16), 2, {}), ("fp64", ("gh", 4), 2, {})])
def test_overlapped_stages_equal_separate_ones(prec, velset, p, tile):
    import torch
    c = cases.couette(5, 4, p, velset=velset, kn=0.5)
    out = []
    for overlapped in (True, False):
        s = cases.solver(c, prec, **tile)
        # far enough from equilibrium that the FP16 scales move by powers of two
        s.set_equilibrium(1.0, 0.05, -0.02, 0.2, 17)
        if overlapped:
            s.step(40)
        else:
            for n in range(200):
                s.stage(n % 5)
                torch.cuda.synchronize()
        out.append(s.state())
        s.close()
    assert np.isfinite(out[0]).all()
    assert np.array_equal(out[0], out[1])
