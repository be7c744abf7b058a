"""Fused Allreduces of pinned host vectors that block boundaries cut, which run wider vectors
than on the device: called directly, captured before the host kernel is there and after, and
the device call of the same plan; bit for bit against the oracle."""

import numpy as np
import pytest
import torch

import gar_inputs
from oracle import gar_oracle as G

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2004_09362_gb300 import gar


@pytest.mark.parametrize("P,n,dtype,op,S", [(6, 79063, "i32", "sum", 5), (8, 200003, "f32", "sum", 6), (24, 100001, "f32", "max", 10),
                                            (13, 93001, "f32", "sum", 24), (40, 70001, "f32", "sum", 8)])
@pytest.mark.parametrize("first", ["direct", "captured", "device"])
def test_host_vectors(P, n, dtype, op, S, first):
    dist = ("int", -1000, 1000) if dtype == "i32" else ("normal", 0.0, 1.0)
    t = gar_inputs.rank_inputs(P, n, dtype, dist, P + n, device="cpu")
    pad = -n % 8
    hin = torch.zeros((P, n + pad), dtype=t.dtype).pin_memory()
    hin[:, :n] = t
    out = torch.zeros_like(hin).pin_memory()
    dev = torch.zeros((P, n + pad), dtype=t.dtype, device="cuda")
    q, rem = divmod(n, P)
    starts = np.array([b * q + min(b, rem) for b in range(P)])
    pos = np.unique(np.concatenate([(starts[:, None] + np.arange(-5, 6)).ravel(), np.arange(n - 20, n), np.arange(200)]))
    pos = pos[(pos >= 0) & (pos < n)]
    want = G.allreduce(list(t.numpy()), S, op, dtype, elements=pos)
    plan = gar.gar_plan_create(P, n, dtype, op, S)
    rows = lambda x: gar.rank_pointer_array([x[r] for r in range(P)])

    def check(x):
        torch.cuda.synchronize()
        got = x.cpu()[:, pos].numpy()
        for r in range(P):
            assert np.array_equal(got[r].view(np.uint32), np.asarray(want[r], got.dtype).view(np.uint32)), r
        assert not x[:, n:].any()

    def host():
        out.zero_()
        gar.gar_allreduce_host(plan, rows(hin), rows(out), rows(dev), "fused")
        check(out)

    def captured():
        gar.gar_plan_prepare(plan, "fused")
        side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            gar.gar_allreduce_host(plan, rows(hin), rows(out), rows(dev), "fused", side)
        out.zero_()
        graph.replay()
        check(out)

    def device():
        dev[:, :n] = t.cuda()
        gar.gar_allreduce(plan, rows(dev), "fused")
        check(dev)

    for step in {"direct": (host, captured, device), "captured": (captured, host, captured), "device": (device, host, device)}[first]:
        step()
    assert gar.gar_plan_get_info(plan)["fused_width"] == 1
