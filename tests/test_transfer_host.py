"""Loads and read-outs last a few microseconds on the GPU: what does not change from call to
call (device attributes, the kernels' shared-memory limit) is asked for when a solver is
created, in transfer::prepare and the batch, not in every call."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2012_13487_gb300", "csrc")


def code(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def test_no_device_query_per_call():
    text = code("transfer.cu")
    assert "cudaDeviceGetAttribute" not in text and "cudaGetDevice" not in text
    assert text.count("cudaFuncSetAttribute") == 1
    # its one caller
    assert len(re.findall(r"\ballow_smem\(\)", text)) == 1 + text[text.index("prepare_as(const Shape"):].split(
        "\n}\n")[0].count("allow_smem()")


def test_the_batch_asks_once():
    text = code("capi.cu")
    body = text[text.index("int create_batch("):text.index("int check_batch(")]
    assert body.count("cudaDeviceGetAttribute") == 2 and "transfer::prepare(" in body
    rest = text.replace(body, "")
    assert rest.count("cudaDeviceGetAttribute") == 1  # sm_count, once per device
