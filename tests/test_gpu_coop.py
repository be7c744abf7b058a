"""The cooperative fused kernel on the GPU, bit for bit against the oracle: vectors shorter
than the rank count, ragged tiles, tiles at every width, both groups, every type, the plans on
both sides of the line that take the form, pinned host vectors, and back-to-back calls."""

import numpy as np
import pytest
import torch

import gar_inputs
from oracle import gar_oracle as G

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2004_09362_gb300 import gar


def _check(P, n, dtype, op, S, group="cyclic", form=None, calls=1, where="cuda"):
    dist = ("int", -1000, 1000) if dtype == "i32" else ("normal", 0.0, 1.0)
    t = gar_inputs.rank_inputs(P, n, dtype, dist, 3 * P + n + S, device="cpu")
    store = torch.zeros((P, n + -n % 8), dtype=t.dtype, device="cpu" if where == "pinned" else "cuda")
    store = store.pin_memory() if where == "pinned" else store
    store[:, :n].copy_(t)
    plan = gar.gar_plan_create_group(P, n, dtype, op, S, group)
    rows = gar.rank_pointer_array([store[x] for x in range(P)])
    host = [r.numpy() if dtype == "i32" else r.float().numpy() for r in t]
    for _ in range(calls):                    # in place: a call reduces the last one's results
        if where == "pinned":
            dev = torch.empty(store.shape, dtype=t.dtype, device="cuda")
            gar.gar_allreduce_host(plan, rows, rows, gar.rank_pointer_array([dev[x] for x in range(P)]), "fused")
        else:
            gar.gar_allreduce(plan, rows, "fused")
        kw = {"group": "xor"} if group == "xor" else {}
        host = [np.asarray(h) for h in G.allreduce(host, "ring" if S < 0 else S, op, dtype, **kw)]
    torch.cuda.synchronize()
    if form is not None:
        assert gar.gar_plan_get_info(plan)["fused_form"] == form
    got = store[:, :n].cpu()
    got = got.numpy() if dtype == "i32" else got.float().numpy()
    for x in range(P):
        assert np.array_equal(got[x].view(np.uint32), host[x].astype(got.dtype).view(np.uint32)), (P, n, dtype, S, x)
    assert not store[:, n:].any()


CASES = [(2, 1, "f32", "sum", 1, "cyclic"), (3, 7, "bf16", "sum", 3, "cyclic"), (5, 1000, "f32", "max", 4, "cyclic"),
         (100, 3, "f32", "sum", 9, "cyclic"), (24, 607, "i32", "sum", 7, "cyclic"), (24, 609, "bf16", "min", 8, "cyclic"),
         (24, 1217, "f32", "sum", 5, "cyclic"), (24, 10007, "bf16", "sum", 10, "cyclic"), (13, 999, "f32", "sum", -3, "cyclic"),
         (13, 2435, "bf16", "sum", 12, "cyclic"), (8, 77, "bf16", "sum", 4, "xor"), (64, 1300, "f32", "sum", 12, "xor"),
         (127, 999, "bf16", "sum", 7, "cyclic")]


@pytest.mark.parametrize("P,n,dtype,op,S,group", CASES)
def test_cooperative_form(P, n, dtype, op, S, group, monkeypatch):
    monkeypatch.setenv("GAR_TUNE_FUSED_FORM", "4")
    _check(P, n, dtype, op, S, group, gar.GAR_FORM_COOP)


@pytest.mark.parametrize("P,n,S,coop", [(16, 1, 4, False), (16, 1, 8, True), (15, 100, 8, False), (32, 9728, 10, True),
                                        (32, 9729, 10, False), (33, 4864, 12, True), (33, 4865, 12, False), (24, 100, -3, False),
                                        (127, 212, 14, True), (127, 4608, 10, True), (127, 1003, 8, True), (127, 4608, 8, False), (40, 100, 6, False)])
def test_plans_that_take_the_cooperative_form(P, n, S, coop):
    plan = gar.gar_plan_create(P, n, "f32", "sum", S)
    gar.gar_plan_prepare(plan, "fused")
    assert (gar.gar_plan_get_info(plan)["fused_form"] == gar.GAR_FORM_COOP) == coop
    _check(P, n, "f32", "sum", S)


def test_back_to_back_calls():
    _check(127, 212, "bf16", "max", 14, form=gar.GAR_FORM_COOP, calls=5)
    _check(24, 5000, "f32", "sum", 10, form=gar.GAR_FORM_COOP, calls=4)


@pytest.mark.parametrize("P,n,dtype,S", [(24, 4001, "f32", 10), (127, 300, "bf16", 9)])
def test_pinned_host_vectors(P, n, dtype, S):
    _check(P, n, dtype, "sum", S, form=gar.GAR_FORM_COOP, where="pinned")
