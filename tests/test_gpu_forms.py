"""The fused forms that short vectors do not take by themselves any more, and the new ones at
their edges, bit for bit: the single-thread form over ranks, step counts, types and groups;
vectors that block boundaries cut, at 2 and 4 positions per thread; special values and many
ranks in the cooperative form; rank pointers in any order in every form."""

import numpy as np
import pytest
import torch

import gar_inputs
from oracle import gar_oracle as G
from paper_2004_09362_gb300 import gar

FORM = "GAR_TUNE_FUSED_FORM"


def _steps(P):
    L = G.ceil_log2(P)
    return range(L, 2 * L + 1)


def _inputs(P, n, dtype, seed):
    dist = ("int", -1000, 1000) if dtype == "i32" else ("normal", 0.0, 1.0)
    t = gar_inputs.rank_inputs(P, n, dtype, dist, seed, device="cpu")
    return t, [r.numpy().copy() if dtype == "i32" else r.float().numpy().copy() for r in t]


def _run(plan, t, order=None):
    P, n = t.shape
    store = torch.zeros((P, n + -n % 8), dtype=t.dtype, device="cuda")
    place = list(range(P)) if order is None else order        # row of rank x
    store[place, :n] = t.cuda()
    gar.gar_allreduce(plan, gar.rank_pointer_array([store[r] for r in place]), "fused")
    torch.cuda.synchronize()
    assert not store[:, n:].any()
    return store[place, :n].cpu()


def _same(got, want, dtype, what):
    got = got.numpy() if dtype == "i32" else got.float().numpy()
    for x, w in enumerate(want):
        assert np.array_equal(got[x].view(np.uint32), np.asarray(w, got.dtype).view(np.uint32)), (*what, x)


@pytest.mark.gpu
@pytest.mark.parametrize("P", range(16, 41))
def test_single_thread_form_every_step_count(P, monkeypatch):
    """What every P up to 40 ran by itself at this size; now the forced form."""
    n = 4 * P + 3
    types = ("f32", "i32", "bf16") if P in (16, 17, 24, 31, 32, 33) else ("f32",)
    for dtype in types:
        t, host = _inputs(P, n, dtype, P)
        for S in _steps(P):
            monkeypatch.setenv(FORM, "0")
            plan = gar.gar_plan_create(P, n, dtype, "sum", S)
            _same(_run(plan, t), G.allreduce(host, S, "sum", dtype), dtype, (P, dtype, S))
            assert gar.gar_plan_get_info(plan)["fused_form"] == gar.GAR_FORM_SINGLE
            monkeypatch.delenv(FORM)
            if dtype == "f32" and P % 8 == 0:
                plan = gar.gar_plan_create(P, n, dtype, "sum", S)
                gar.gar_plan_prepare(plan, "fused")
                info = gar.gar_plan_get_info(plan)
                coop = info["K"] == 1 or (P >= 20 and info["K"] < P)
                assert info["fused_form"] == (gar.GAR_FORM_COOP if coop else gar.GAR_FORM_SINGLE)


@pytest.mark.gpu
@pytest.mark.parametrize("P", [16, 32, 64])
def test_single_thread_form_xor_group(P, monkeypatch):
    monkeypatch.setenv(FORM, "0")
    n = 5 * P + 3
    t, host = _inputs(P, n, "f32", P)
    for S in _steps(P):
        plan = gar.gar_plan_create_group(P, n, "f32", "sum", S, "xor")
        _same(_run(plan, t), G.allreduce(host, S, "sum", "f32", group="xor"), "f32", (P, S))
        assert gar.gar_plan_get_info(plan)["fused_form"] == gar.GAR_FORM_SINGLE


@pytest.mark.gpu
@pytest.mark.parametrize("P,S,dtype,op,group", [
    (3, 3, "f32", "sum", "cyclic"), (5, 4, "i32", "sum", "cyclic"), (7, 6, "f32", "max", "cyclic"), (12, 5, "f32", "sum", "cyclic"),
    (24, 10, "f32", "sum", "cyclic"), (24, 7, "i32", "min", "cyclic"), (48, 9, "f32", "sum", "cyclic"), (100, 14, "f32", "sum", "cyclic"),
    (13, 24, "f32", "sum", "cyclic"), (8, 5, "f32", "sum", "xor"), (16, 8, "i32", "sum", "xor"), (32, 7, "f32", "sum", "xor"),
    (24, 10, "bf16", "sum", "cyclic"), (16, 6, "bf16", "sum", "xor")])
@pytest.mark.parametrize("width", [2, 4])
def test_vectors_that_block_boundaries_cut(P, S, dtype, op, group, width, monkeypatch):
    monkeypatch.setenv("GAR_TUNE_FUSED_W", str(width))
    for n in (P // 2 + 1, 3 * P + 2, 33 * P + P // 2, 257 * P + 1):
        t, host = _inputs(P, n, dtype, P + n)
        plan = gar.gar_plan_create_group(P, n, dtype, op, S, group)
        kw = {"group": "xor"} if group == "xor" else {}
        _same(_run(plan, t), G.allreduce(host, S, op, dtype, **kw), dtype, (P, S, n))
        info = gar.gar_plan_get_info(plan)
        assert (info["fused_form"], info["fused_width"]) == (gar.GAR_FORM_SINGLE, width)


@pytest.mark.gpu
@pytest.mark.parametrize("P,n,S", [(24, 1003, 10), (24, 1003, 7), (127, 1500, 14)])
@pytest.mark.parametrize("dtype,op", [("f32", "sum"), ("f32", "max"), ("bf16", "sum"), ("bf16", "min")])
def test_special_values_in_the_cooperative_form(P, n, S, dtype, op, monkeypatch):
    """Infinities, NaN, signed zeros, subnormals and overflowing sums: the bits of the
    single-thread form (order of combines and roundings are the schedule's in both)."""
    g = torch.Generator().manual_seed(P + n + S)
    values = torch.tensor([0.0, -0.0, 1.0, -1.0, 1e-40, -1e-40, 9e-41, 3.0e38, -3.0e38, float("inf"), -float("inf"), float("nan")])
    weights = torch.tensor([8.0, 8, 8, 8, 8, 8, 8, 0.1, 0.1, 0.1, 0.1, 0.1])
    x = values[torch.multinomial(weights, P * n, replacement=True, generator=g)].view(P, n)
    x[:, ::3] = x[:, ::3].clamp(-2e-40, 2e-40).nan_to_num()       # subnormal sums
    x = x.to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    got = []
    for form in (gar.GAR_FORM_SINGLE, gar.GAR_FORM_COOP):
        monkeypatch.setenv(FORM, str(form))
        plan = gar.gar_plan_create(P, n, dtype, op, S)
        got.append(_run(plan, x).view(torch.int16 if dtype == "bf16" else torch.int32))
        assert gar.gar_plan_get_info(plan)["fused_form"] == form
    assert torch.equal(got[0], got[1])


@pytest.mark.gpu
@pytest.mark.parametrize("P,n,dtype,S", [(256, 300, "f32", 16), (256, 4864, "bf16", 16), (200, 199, "i32", 16), (500, 7, "f32", 18)])
def test_cooperative_form_with_many_ranks(P, n, dtype, S):
    t, host = _inputs(P, n, dtype, P + n)
    plan = gar.gar_plan_create(P, n, dtype, "sum", S)
    _same(_run(plan, t), G.allreduce(host, S, "sum", dtype), dtype, (P, n))
    assert gar.gar_plan_get_info(plan)["fused_form"] == gar.GAR_FORM_COOP


@pytest.mark.gpu
@pytest.mark.parametrize("form,P,n,S", [(0, 24, 500, 7), (0, 40, 999, 12), (1, 24, 500, 7), (3, 5, 5 * 600 + 3, 4), (4, 24, 500, 7),
                                        (4, 127, 212, 14)])
@pytest.mark.parametrize("order", ["descending", "mixed"])
def test_rank_pointers_in_any_order(form, P, n, S, order, monkeypatch):
    monkeypatch.setenv(FORM, str(form))
    t, host = _inputs(P, n, "f32", P + n)
    place = list(range(P))[::-1] if order == "descending" else np.random.default_rng(P).permutation(P).tolist()
    plan = gar.gar_plan_create(P, n, "f32", "sum", S)
    _same(_run(plan, t, place), G.allreduce(host, S, "sum", "f32"), "f32", (P, form))
    assert gar.gar_plan_get_info(plan)["fused_form"] == form


@pytest.mark.parametrize("pointers", [[5, 4, 3, 3, 1], [1, 2, 3, 4, 4], [1, 2, 3, 4, 1], [4, 1, 5, 2, 4]])
def test_ranks_that_share_a_buffer_are_refused(pointers):
    with pytest.raises(gar.GarError) as e:
        gar.gar_allreduce(gar.gar_plan_create(5, 10), [16 * p for p in pointers], "fused", stream=0)
    assert e.value.code == -1 and "share one buffer" in str(e.value)
