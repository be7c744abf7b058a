"""No-allocation Allreduces on both sides of the lines between element-major and chunked
launches, and calls that mix the two, bit for bit against the oracle."""

import numpy as np
import pytest
import torch

import gar_inputs
from oracle import gar_oracle as G

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2004_09362_gb300 import gar

# 16 ranks x 1024 elements: launches of 16 and more ops are chunked, fewer element-major
CASES = [(16, 1023, "f32", "sum"), (16, 1024, "f32", "sum"), (20, 511, "f32", "sum"), (20, 513, "bf16", "sum"), (33, 700, "i32", "max"),
         (48, 1300, "bf16", "min"), (64, 2000, "f32", "sum"), (5, 2047, "bf16", "sum"), (7, 2049, "f32", "sum")]


@pytest.mark.parametrize("P,blk,dtype,op", CASES)
def test_every_step_count(P, blk, dtype, op):
    L = G.ceil_log2(P)
    n = blk * P - P // 3
    dist = ("int", -1000, 1000) if dtype == "i32" else ("normal", 0.0, 1.0)
    t = gar_inputs.rank_inputs(P, n, dtype, dist, P + blk, device="cpu")
    pos = np.unique(np.concatenate([np.arange(300), np.arange(n - 300, n), np.random.default_rng(P).integers(0, n, 1500)]))
    host = np.zeros((P, n), np.int32 if dtype == "i32" else np.float32)
    host[:, pos] = t[:, pos].numpy() if dtype == "i32" else t[:, pos].float().numpy()
    for S in (L, L + 1, L + 2, 2 * L):
        store = torch.zeros((P, n + -n % 8), dtype=t.dtype, device="cuda")
        store[:, :n] = t.cuda()
        plan = gar.gar_plan_create(P, n, dtype, op, S)
        gar.gar_allreduce_noalloc(plan, gar.rank_pointer_array([store[x] for x in range(P)]))
        torch.cuda.synchronize()
        got = store[:, :n].cpu()[:, pos]
        got = got.numpy() if dtype == "i32" else got.float().numpy()
        for x, w in enumerate(G.allreduce(list(host), S, op, dtype, elements=pos)):
            assert np.array_equal(got[x].view(np.uint32), np.asarray(w, got.dtype).view(np.uint32)), (P, blk, S, x)
        assert not store[:, n:].any()
