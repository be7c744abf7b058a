"""Positions per thread of the single-thread fused kernel on both sides of the lines where
blocks that vectors would straddle are read one position at a time: the width that is chosen
(no GPU), and the results, bit for bit against the oracle (GPU)."""

import numpy as np
import pytest
import torch

import gar_inputs
from oracle import gar_oracle as G
from paper_2004_09362_gb300 import gar

CASES = [(24, (1 << 18) - 1, "f32", 10, 1), (24, (1 << 18) + 1, "f32", 10, 4), (24, 24 * 4096, "f32", 10, 4),
         (24, 24 * 4096 + 4, "f32", 10, 1), (7, (1 << 17) - 3, "f32", 6, 1), (7, (1 << 17) + 3, "f32", 6, 4),
         (12, 200001, "f32", 4, 4), (16, 16 * 4098, "f32", 8, 1), (16, 16 * 4098, "bf16", 8, 4)]


@pytest.mark.parametrize("P,n,dtype,S,width", CASES)
def test_width(P, n, dtype, S, width):
    plan = gar.gar_plan_create(P, n, dtype, "sum", S)
    gar.gar_plan_compile(plan, "fused")
    assert gar.gar_plan_get_info(plan)["fused_width"] == width


@pytest.mark.gpu
@pytest.mark.parametrize("P,n,dtype,S,width", CASES)
def test_results(P, n, dtype, S, width):
    t = gar_inputs.rank_inputs(P, n, dtype, ("normal", 0.0, 1.0), P + n, device="cpu")
    store = torch.zeros((P, n + -n % 8), dtype=t.dtype, device="cuda")
    store[:, :n] = t.cuda()
    gar.gar_allreduce(gar.gar_plan_create(P, n, dtype, "sum", S), gar.rank_pointer_array([store[x] for x in range(P)]), "fused")
    torch.cuda.synchronize()
    q, rem = divmod(n, P)
    starts = np.array([b * q + min(b, rem) for b in range(P)])
    pos = np.unique(np.concatenate([(starts[:, None] + np.arange(-9, 10)).ravel(), np.arange(300), np.arange(n - 20, n)]))
    pos = pos[(pos >= 0) & (pos < n)]
    want = G.allreduce([r.float().numpy() for r in t], S, "sum", dtype, elements=pos)
    got = store[:, :n].cpu()[:, pos].float().numpy()
    for x in range(P):
        assert np.array_equal(got[x].view(np.uint32), np.asarray(want[x], np.float32).view(np.uint32)), x
    assert not store[:, n:].any()
