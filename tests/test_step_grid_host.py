"""Launch rules of the step kernels, without a GPU: which launches are element-major (step
launches up to blocks of 2047 elements, no-allocation launches only while their blocks or all
their elements are few), the persistent kernel's CTAs per SM and the pieces of its blocks."""

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


@pytest.fixture(scope="module")
def rules_program(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    tmp_path = tmp_path_factory.mktemp("step_rules")
    text = open(os.path.join(build.CSRC, "step_kernels.cu")).read()
    consts = "\n".join(re.findall(r"^constexpr .*?;", text, re.M))
    rules = re.search(r"^uint32_t pick_chunk\(.*?^\}\n", text, re.S | re.M).group(0)
    rules += re.search(r"^int pick_group\(.*?^\}\n", text, re.S | re.M).group(0)
    rules += re.search(r"^template <int MAXP>\nint step_grid\(.*?^\}\n", text, re.S | re.M).group(0)
    rules += re.search(r"^int persist_per_sm\(.*?^\}\n", text, re.S | re.M).group(0)
    (tmp_path / "step_desc.inc").write_text(re.search(r"^LaunchDesc launch_desc\(.*?^\}\n", text, re.S | re.M).group(0))
    (tmp_path / "step_rules.inc").write_text(consts + "\n" + rules)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    exe = str(tmp_path / "check")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-I", str(tmp_path), "-I", build.INCLUDE, "-I", build.CSRC, "-isystem", cuda,
                    os.path.join(TESTS, "step_grid_check.cpp"), "-o", exe], check=True)
    return exe


def _ask(exe, what, lines):
    text = "".join(" ".join(map(str, x)) + "\n" for x in lines)
    r = subprocess.run([exe, what], input=text, capture_output=True, text=True, check=True)
    return [[int(v) for v in line.split()] for line in r.stdout.splitlines()]


def test_element_major_launches(rules_program):
    assert _ask(rules_program, "flat", [c[:4] for c in CASES]) == [[c[4]] for c in CASES]


F32, BF16 = 0, 1


#        elements, P, ops of the largest step, result copies, type, CTAs per SM
PERSIST = [(1 << 20, 24, 3, 1, F32, 2), (1 << 20, 24, 4, 1, F32, 3), (1 << 20, 24, 12, 1, BF16, 2), (1 << 22, 24, 4, 1, BF16, 3),
           (1 << 20, 24, 4, 3, BF16, 3), (80000, 18, 34, 18, F32, 3), (80000, 18, 33, 18, F32, 2), (40000, 64, 32, 2, F32, 2)]


def test_persistent_ctas_and_pieces(rules_program):
    assert [r[0] for r in _ask(rules_program, "pieces", [c[:5] for c in PERSIST])] == [c[5] for c in PERSIST]
    lines = [(n, P, nops, K, t) for P in (2, 3, 13, 18, 64, 127) for n in (2048 * P, 2049 * P - 1, 13331 * P, 120000 * P + 1)
             for nops in (1, P // 2 + 1, 2 * P) for K in (1, P) for t in (F32, BF16)] + [(1 << 34, 2, 1, 1, F32)]
    batch = lambda piece: -(-piece // 2048) + 1
    for (n, P, nops, K, _t), (per_sm, pieces, piece) in zip(lines, _ask(rules_program, "pieces", lines)):
        blk, blocks, grid = -(-n // P), P * nops, 152 * per_sm
        assert piece >= 2048 and (pieces - 1) * piece < blk <= pieces * piece       # every element, no empty piece
        cost = -(-blocks * pieces // grid) * batch(piece)
        assert cost <= -(-blocks // grid) * batch(blk)                              # no worse than whole blocks
