"""The step kernels at the edges of their launch shapes, bit for bit against the oracle:
block lengths around the element-major limit (2048 elements) and around one and two
chunks, op counts that leave a remainder in a group of ops per thread, one element; the
per-step, persistent and no-allocation calls, the counters of the first two when the calls
alternate on one plan."""

import numpy as np
import pytest
import torch

import gar_inputs
from oracle import gar_oracle as G

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2004_09362_gb300 import gar

SHAPES = [
    (2, 1, "f32", 1), (3, 2, "bf16", 4), (7, 7 * 2047 + 3, "bf16", 5), (7, 7 * 2048, "i32", 6),
    (5, 5 * 2049 + 2, "f32", 3), (4, 4 * 4096 + 1, "bf16", 2), (3, 3 * 16384 + 2, "f32", 4),
    (3, 3 * 33000 + 1, "bf16", 4), (61, 61 * 700 + 5, "bf16", 8), (64, 64 * 40 + 1, "i32", 6),
    (13, 13 * 2060 + 12, "f32", 24),
]


def _same(got, want, what):
    view = np.uint16 if got.dtype == torch.bfloat16 else np.uint32
    raw = got.view(torch.int16) if got.dtype == torch.bfloat16 else got.view(torch.int32)
    raw = raw.cpu().numpy().view(view)
    for x, w in enumerate(want):
        bits = w.astype(np.float32).view(np.uint32) if view is np.uint16 else np.ascontiguousarray(w).view(np.uint32)
        bits = (bits >> 16).astype(np.uint16) if view is np.uint16 else bits
        assert np.array_equal(raw[x], bits), f"{what}: rank {x} differs"


@pytest.mark.parametrize("P,n,dtype,S", SHAPES)
def test_step_kernels_at_shape_edges(P, n, dtype, S):
    dist = ("int", -1000, 1000) if dtype == "i32" else ("normal", 0.0, 1.0)
    t = gar_inputs.rank_inputs(P, n, dtype, dist, 7 * P + n)
    host = [r.float().numpy() if dtype == "bf16" else r.numpy() for r in t]
    want = G.allreduce([h.copy() for h in host], S, "sum", dtype)
    pad = -n % 8
    plan = gar.gar_plan_create(P, n, dtype, "sum", S)
    _ws, per_step, _S = gar.gar_plan_bytes(plan)
    for mode in ("step", "persistent", "step", "step", "persistent", "persistent", "noalloc", "step"):
        x = torch.zeros(P, n + pad, dtype=t.dtype, device="cuda")[:, :n]
        x.copy_(t)
        if mode == "noalloc":
            gar.gar_allreduce_noalloc(plan, x)
        else:
            gar.gar_allreduce(plan, x, mode)
            assert gar.gar_last_step_bytes(plan) == list(per_step), mode
        if mode == "persistent":
            assert gar.gar_plan_status(plan) == gar.GAR_OK
        _same(x, want, f"{mode} P={P} n={n} {dtype} S={S}")
