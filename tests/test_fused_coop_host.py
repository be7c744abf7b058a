"""Host-side checks of the cooperative fused kernel (GAR_FORM_COOP, no GPU): its table of the
program, run level by level in numpy, gives the oracle's bits for every rank; a level only
reads values of earlier ones; NVRTC compiles the kernels for sm_103a."""

import re

import numpy as np
import pytest

from oracle import gar_oracle as O
from paper_2004_09362_gb300 import gar as G


def _plan(monkeypatch, P, n, dtype, op, S, group="cyclic"):
    monkeypatch.setenv("GAR_TUNE_FUSED_FORM", "4")
    pl = G.gar_plan_create_group(P, n, dtype, op, S, group)
    assert G.gar_plan_get_info(pl)["fused_form"] == G.GAR_FORM_COOP
    return pl


def _table(src, name):
    return [int(x) for x in re.search(name + r"\[\d+\] = \{([\du,]*)\}", src).group(1).replace("u", "").split(",") if x]


def _combine(dtype, op, a, b):
    if op == "sum":
        return (a.astype(np.int64) + b).astype(np.int32) if dtype == "i32" else a + b
    return np.maximum(a, b) if op == "max" else np.minimum(a, b)


CASES = [(P, "f32", "sum", S, "cyclic") for P in (2, 3, 5, 6, 13, 24)
         for S in [*range((P - 1).bit_length(), 2 * (P - 1).bit_length() + 1), G.GAR_STEPS_RING]]
CASES += [(24, "bf16", "sum", 6, "cyclic"), (24, "i32", "sum", 7, "cyclic"), (40, "bf16", "max", 9, "cyclic"),
          (24, "f32", "min", 14, "cyclic"), (127, "bf16", "sum", 14, "cyclic"), (127, "bf16", "sum", 10, "cyclic"),
          (8, "f32", "sum", 4, "xor"), (64, "bf16", "sum", 12, "xor")]


@pytest.mark.parametrize("P,dtype,op,S,group", CASES)
def test_table_reproduces_the_oracle(P, dtype, op, S, group, monkeypatch):
    n = 3 * P + 2
    pl = _plan(monkeypatch, P, n, dtype, op, S, group)
    src = G.gar_plan_fused_source(pl)
    rng = np.random.default_rng(P + n)
    if dtype == "i32":
        x = [rng.integers(-2 ** 31, 2 ** 31, n).astype(np.int32) for _ in range(P)]
    else:
        x = [(rng.standard_normal(n) * np.exp2(rng.integers(-9, 10, n))).astype(np.float32) for _ in range(P)]
        x = [O.round_to_bf16(r) for r in x] if dtype == "bf16" else x
    want = O.allreduce(x, S if S > 0 else "ring", op, dtype, **({"group": "xor"} if group == "xor" else {}))
    q, rem = divmod(n, P)
    block = np.repeat(np.arange(P), [q + (b < rem) for b in range(P)])
    rotate = G.gar_plan_get_info(pl)["K"] != P
    rank = (lambda j: (block ^ j if group == "xor" else (block + j) % P)) if rotate else (lambda j: np.full(n, j))
    at, xs = np.arange(n), np.stack(x)
    v = [xs[rank(j), at] for j in range(P)]
    ops, outs = _table(src, "gar_ops"), _table(src, "gar_outs")
    k = 0
    for k0, k1 in re.findall(r"gar_level\(v, s_ops, (\d+), (\d+), row, c\);", src):
        assert int(k0) == k < int(k1)
        k = int(k1)
        for o in ops[int(k0): k]:
            assert max(o & 0xffff, o >> 16) < P + int(k0)
            v.append(_combine(dtype, op, v[o & 0xffff], v[o >> 16]))
    assert k == len(ops) == G.gar_plan_get_info(pl)["fused_combines"]
    got = np.empty_like(xs)
    for p in range(P):
        got[rank(p), at] = O.round_to_bf16(v[outs[p]]) if dtype == "bf16" else v[outs[p]]
    for r in range(P):
        w = np.asarray(want[r], got.dtype)
        assert np.array_equal(got[r].view(np.uint32), w.view(np.uint32)), r


@pytest.mark.parametrize("P,n,dtype,op,S", [(2, 1, "f32", "sum", 1), (127, 212, "bf16", "sum", 14), (24, 4608, "i32", "max", 7)])
def test_kernel_compiles(P, n, dtype, op, S, monkeypatch):
    G.gar_plan_compile(_plan(monkeypatch, P, n, dtype, op, S), "fused")
