"""The persistent kernel on plans whose steps have more blocks than the device has CTAs, which
run more CTAs per SM, and just below that line; bit for bit against the oracle, with the bytes
of every step and the status."""

import numpy as np
import pytest
import torch

import gar_inputs
from oracle import gar_oracle as G

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2004_09362_gb300 import gar

CASES = [(17, 17 * 2051 + 4, "f32", "sum", 5), (17, 17 * 2051 + 4, "bf16", "sum", 6), (18, 18 * 2101 + 1, "bf16", "max", 5),
         (24, 24 * 2500 + 3, "i32", "sum", 6), (33, 33 * 2048 + 7, "f32", "sum", 6), (33, 33 * 5003, "bf16", "sum", 6),
         (18, 18 * 9001 + 2, "f32", "sum", 7), (130, 130 * 2060 + 9, "f32", "min", 9)]


@pytest.mark.parametrize("P,n,dtype,op,S", CASES)
def test_many_blocks(P, n, dtype, op, S):
    dist = ("int", -1000, 1000) if dtype == "i32" else ("normal", 0.0, 1.0)
    t = gar_inputs.rank_inputs(P, n, dtype, dist, P + n, device="cpu")
    q, rem = divmod(n, P)
    starts = np.array([b * q + min(b, rem) for b in range(P)])
    pos = np.unique(np.concatenate([(starts[:, None] + np.arange(-9, 10)).ravel(), np.arange(n - 50, n),
                                    np.random.default_rng(n).integers(0, n, 2000)]))
    pos = pos[(pos >= 0) & (pos < n)]
    host = np.zeros((P, n), np.int32 if dtype == "i32" else np.float32)
    host[:, pos] = t[:, pos].numpy() if dtype == "i32" else t[:, pos].float().numpy()
    want = G.allreduce(list(host), S, op, dtype, elements=pos)
    plan = gar.gar_plan_create(P, n, dtype, op, S)
    for mode in ("persistent", "persistent", "step", "persistent"):
        x = torch.zeros((P, n + -n % 8), dtype=t.dtype, device="cuda")
        x[:, :n] = t.cuda()
        gar.gar_allreduce(plan, x[:, :n], mode)
        assert gar.gar_last_step_bytes(plan) == gar.gar_plan_bytes(plan)[1], mode
        if mode == "persistent":
            assert gar.gar_plan_status(plan) == gar.GAR_OK
        got = x.cpu()[:, pos]
        got = got.numpy() if dtype == "i32" else got.float().numpy()
        for r in range(P):
            assert np.array_equal(got[r].view(np.uint32), np.asarray(want[r], got.dtype).view(np.uint32)), (mode, r)
        assert not x[:, n:].any()
