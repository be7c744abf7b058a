"""The step kernels' byte counts, without a GPU: range_work, compiled for the host and run
thread by thread, returns for every thread what that thread read from its partner, in every
kind of loop (a count taken from the range's ends would hide a loop that skips elements)."""

import os
import shutil
import subprocess

import pytest

from paper_2004_09362_gb300 import build

TESTS = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_every_thread_counts_what_it_reads(tmp_path):
    text = open(os.path.join(build.CSRC, "step_kernels.cu")).read()
    device, rest = text.split("// Launches a step kernel with programmatic stream serialisation")
    assert "range_work" in device and "launch_step" in rest
    (tmp_path / "step_device.inc").write_text(device + "}  // namespace\n}  // namespace gar\n")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    exe = str(tmp_path / "check")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-I", str(tmp_path), "-I", build.INCLUDE, "-I", build.CSRC, "-isystem", cuda,
                    os.path.join(TESTS, "step_count_check.cpp"), "-L", build._cuda_lib_dir(build._nvcc()), "-lcudart",
                    "-o", exe, f"-Wl,-rpath,{build._cuda_lib_dir(build._nvcc())}"], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[:2000] + r.stderr[:2000]
