"""Host-only check of what the library sets up once per device (csrc/fwi_device.h): compiles and
runs tests/native/device_check.cpp; and in the source, that no launch attribute of a kernel is
set in a process-wide static, which would hold for the first device alone."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1804_01184_gb300", "csrc")


def test_per_device_cache(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "device_check")
    subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, os.path.join(HERE, "native", "device_check.cpp"),
                    "-o", exe], check=True, capture_output=True, text=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "device ok" in r.stdout, r.stdout + r.stderr


def test_no_function_attribute_in_a_process_wide_static():
    found = 0
    for f in sorted(os.listdir(CSRC)):
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        # initialisers of function-local statics: static T x = [] { ... }();
        for m in re.finditer(r"static const \w+ \w+ = \[\]\s*\{(.*?)\}\(\);", src, flags=re.S):
            assert "cudaFuncSetAttribute" not in m.group(1) and "cudaOccupancy" not in m.group(1), f
        found += "cudaFuncAttributeNonPortableClusterSizeAllowed" in src
    assert found == 1
