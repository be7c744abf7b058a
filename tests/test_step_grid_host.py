"""Which launches are element-major, without a GPU: step launches up to blocks of 2047
elements, no-allocation launches only while their blocks or all their elements are few."""

import os
import re
import shutil
import subprocess

import pytest

from paper_2004_09362_gb300 import build

TESTS = os.path.dirname(os.path.abspath(__file__))
#        block, P, ops, no allocation, element-major
CASES = [(2047, 64, 64, 0, 1), (2048, 64, 64, 0, 0), (2047, 64, 64, 1, 0), (512, 64, 64, 1, 0), (511, 64, 64, 1, 1),
         (2047, 5, 5, 1, 1), (2048, 5, 5, 1, 0), (1024, 16, 15, 1, 1), (1024, 16, 16, 1, 0), (1024, 16, 16, 0, 1), (1, 64, 1, 1, 1)]


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_element_major_launches(tmp_path):
    text = open(os.path.join(build.CSRC, "step_kernels.cu")).read()
    consts = "\n".join(re.findall(r"^constexpr .*?;", text, re.M))
    rules = re.search(r"^uint32_t pick_chunk\(.*?^\}\n", text, re.S | re.M).group(0)
    rules += re.search(r"^int pick_group\(.*?^\}\n", text, re.S | re.M).group(0)
    rules += re.search(r"^template <int MAXP>\nint step_grid\(.*?^\}\n", text, re.S | re.M).group(0)
    (tmp_path / "step_rules.inc").write_text(consts + "\n" + rules)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    exe = str(tmp_path / "check")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-I", str(tmp_path), "-I", build.INCLUDE, "-I", build.CSRC, "-isystem", cuda,
                    os.path.join(TESTS, "step_grid_check.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], input="".join("%d %d %d %d\n" % c[:4] for c in CASES), capture_output=True, text=True, check=True)
    assert [int(v) for v in r.stdout.split()] == [c[4] for c in CASES]
