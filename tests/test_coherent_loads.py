"""A stage kernel launched programmatically is resident while the stage before it still
writes the state, the residual and the element scales (stage_impl.cuh), so none of the
three may be read through the non-coherent path: __ldg and ld.global.nc are specified
only for data that nothing writes during the kernel's lifetime."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2012_13487_gb300", "csrc")
WRITTEN = r"scale_in|scale_out|res|f_in|f_out"  # StageArgs members that a stage kernel writes


def code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


@pytest.mark.parametrize("name", ["stage_impl.cuh", "stage_ws.cuh", "stage_cluster.cuh", "stage_eo.cuh"])
def test_no_non_coherent_load_of_what_a_stage_writes(name):
    text = code(name)
    # the pointers a kernel derives from those members
    derived = re.findall(r"\*\s*(\w+)\s*=\s*static_cast<[^>]*>\(a\.(?:%s)\)" % WRITTEN, text)
    names = r"a\.(?:%s)\b" % WRITTEN + "".join(r"|\b%s\b" % d for d in derived)
    assert not re.findall(r"__ldg\(\s*(?:reinterpret_cast<[^>]*>\()?(?:%s)" % names, text)
    assert "ld.global.nc" not in text
    assert "__restrict__" not in text  # which would let the compiler take that path by itself


def test_the_step_counter_is_written_between_steps_only():
    """The stage kernels read the counter with __ldg: its one writer among the kernels is
    an ordinary launch (no programmatic edge), which never lets the next stage start early."""
    text = code("capi.cu")
    assert len(re.findall(r"sr_step_kernel<<<1, 1, 0, st>>>", text)) == 1
    body = re.search(r"__global__ void sr_step_kernel\(uint32_t\* step\) \{(.*?)\}", text).group(1)
    assert "launch_dependents" not in body
