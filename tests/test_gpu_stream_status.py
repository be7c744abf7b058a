"""A streaming kernel whose wait for its tile runs out (an arrival too many is expected, and
the limit is short): it ends by itself, every plan that ran it reports GAR_ETIMEOUT once, a
graph replay does too, and plans of the normal kernel run on correctly."""

import numpy as np
import pytest
import torch

import gar_inputs
from oracle import gar_oracle as G

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2004_09362_gb300 import gar


def test_wait_that_gives_up(monkeypatch):
    P, n, S = 5, 5 * 4001 + 3, 4
    t = gar_inputs.rank_inputs(P, n, "bf16", ("normal", 0.0, 1.0), 11, device="cpu")
    store = torch.zeros((P, n + -n % 8), dtype=t.dtype, device="cuda")
    monkeypatch.setenv("GAR_TUNE_FUSED_FORM", "3")

    def plan():
        p = gar.gar_plan_create(P, n, "bf16", "sum", S)
        gar.gar_plan_prepare(p, "fused")
        assert gar.gar_plan_get_info(p)["fused_form"] == gar.GAR_FORM_STREAM
        return p

    good = plan()
    monkeypatch.setenv("GAR_TUNE_ST_PHANTOM", "1")
    monkeypatch.setenv("GAR_TUNE_ST_WAIT_MS", "100")
    a, b, c = plan(), plan(), plan()
    for p in (a, b):
        gar.gar_allreduce(p, store, "fused")
    assert gar.gar_plan_status(c) == gar.GAR_OK
    for p in (a, b):
        assert gar.gar_plan_status(p) == -8
        assert gar.gar_plan_status(p) == gar.GAR_OK
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=side):
        gar.gar_allreduce(c, store, "fused", side)
        assert gar.gar_plan_status(c) == gar.GAR_OK
    for want in (-8, gar.GAR_OK):
        if want != gar.GAR_OK:
            graph.replay()
        torch.cuda.synchronize()
        assert gar.gar_plan_status(c) == want
    store[:, :n] = t.cuda()
    gar.gar_allreduce(good, store, "fused")
    assert gar.gar_plan_status(good) == gar.GAR_OK
    want = G.allreduce([r.float().numpy() for r in t], S, "sum", "bf16")
    got = store[:, :n].float().cpu().numpy()
    for x in range(P):
        assert np.array_equal(got[x].view(np.uint32), np.asarray(want[x], np.float32).view(np.uint32)), x
