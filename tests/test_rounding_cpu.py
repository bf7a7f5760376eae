"""The streaming and the on-chip time steps are to give the same bits, so every float operation that
both share says how it rounds (fmaf, __fmul_rn, packed intrinsics): a plain product inside a sum would
leave that to what the compiler contracts in each of them.  Checked in their sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1804_01184_gb300", "csrc")
# a product added in place, or to an accessed element; index arithmetic (no element, no name of a weight) is not matched
SUM = re.compile(r"(?:\+=|-=)[^;]*(?:\]|\))\s*\*|(?:\+=|-=)[^;]*\*\s*[\w.]+\[|(?:\+=|-=)[^;]*\*\s*w\b")


def code(name):
    src = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", src, flags=re.S)


@pytest.mark.parametrize("name", ["fwi_stream.cuh", "fwi_warp.cuh", "fwi_resident.cuh"])
def test_no_product_in_a_sum_is_left_to_contraction(name):
    bad = [line.strip() for line in code(name).splitlines() if SUM.search(line)]
    assert not bad, bad


def test_sampling_kernel():
    src = code("fwi_kernels.cuh")
    body = src[src.index("void k_sample("):]
    body = body[:body.index("\n}")]
    assert not SUM.search(body), body


def test_injection_is_written_out():
    """The source terms go through one function, whose roundings are explicit."""
    for name, n in (("fwi_warp.cuh", 3), ("fwi_resident.cuh", 3)):
        src = code(name)
        calls = re.findall(r"add_source<(?:true|false)>\(([^;]*)\);", src)
        assert len(calls) == n, (name, calls)
        assert all("__fmul_rn(" in c for c in calls), calls
    for name in ("fwi_warp.cuh", "fwi_stream.cuh"):
        assert "addc(" not in code(name)
