"""Host code of the library on a fake CUDA runtime (no GPU, no CUDA libraries): what it asks
of the runtime for several devices, plans, threads and settings.  fake_cuda_check.cpp holds
the checks, fake_cuda.hpp the runtime."""

import concurrent.futures as cf
import os
import shutil
import subprocess

import pytest

from paper_2004_09362_gb300 import build

TESTS = os.path.dirname(os.path.abspath(__file__))
SOURCES = ["api.cpp", "codegen.cpp", "jit.cpp", "plan.cpp"]


def _cuda_include():
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")


def _program(out, flags):
    cmd = ["g++", "-std=c++17", *flags, "-I", build.INCLUDE, "-I", build.CSRC, "-I", TESTS, "-isystem", _cuda_include()]
    sources = [os.path.join(build.CSRC, s) for s in SOURCES] + [os.path.join(TESTS, "fake_cuda_check.cpp")]

    def compile_one(src):
        obj = str(out / (os.path.basename(src) + ".o"))
        subprocess.run([*cmd, "-c", src, "-o", obj], check=True)
        return obj

    with cf.ThreadPoolExecutor(len(sources)) as ex:
        objs = list(ex.map(compile_one, sources))
    subprocess.run([*cmd, *objs, "-pthread", "-o", str(out / "check")], check=True)
    return str(out / "check")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    return _program(tmp_path_factory.mktemp("fake_cuda"), ["-O1"])


def _run(program, check, **env):
    r = subprocess.run([program, check], capture_output=True, text=True, timeout=30, env={**os.environ, **env})
    assert r.returncode == 0, r.stdout + r.stderr


def test_equal_plans_on_two_devices(program):
    _run(program, "two_devices")


def test_failed_waits_of_plans_that_share_a_kernel(program):
    _run(program, "wait_status")


@pytest.mark.parametrize("forced", ["", "3", "4"])
def test_groups_of_a_streaming_kernel_that_spills(program, forced):
    _run(program, "stream_groups", **({"GAR_TUNE_ST_GROUPS": forced} if forced else {}))


def test_threads_that_batch_over_shared_plans(tmp_path):
    """Under the thread sanitizer (exit code 66 of a race)."""
    (tmp_path / "t.cpp").write_text("int main() {}")
    flags = ["-O1", "-g", "-fsanitize=thread"]
    probe = f"g++ {' '.join(flags)} {tmp_path}/t.cpp -o {tmp_path}/t && {tmp_path}/t"
    if subprocess.run(probe, shell=True, capture_output=True).returncode != 0:
        pytest.skip("no thread sanitizer here")
    _run(_program(tmp_path, flags), "batched_threads")


def test_tuning_knobs_reach_the_kernels_they_shape(program):
    _run(program, "knobs")


def test_a_plan_compiled_ahead_prepares_the_same_kernel(program):
    _run(program, "compiled_ahead")


def test_the_cooperative_form_follows_the_sm_count(program):
    _run(program, "sm_count")


def test_ranks_from_which_short_vectors_take_the_cooperative_form(program):
    _run(program, "cooperative_ranks")


def test_host_memory_has_its_own_width(program):
    _run(program, "host_width")


def test_host_memory_calls_run_in_whole_rounds(program):
    _run(program, "host_grid")
