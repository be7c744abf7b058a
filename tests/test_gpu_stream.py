"""The streaming fused kernel on the GPU, bit for bit against the oracle: block boundaries
at every residue of a 16-byte unit and of a tile, ragged ends, one tile and several rounds of
the ring, every type, sums and max, in place; pinned host vectors; the plans that take the
form by themselves."""

import numpy as np
import pytest
import torch

import gar_inputs
from oracle import gar_oracle as G

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2004_09362_gb300 import gar


def _check(P, n, dtype, op, S, where="cuda", force=True, samples=3000):
    dist = ("int", -1000, 1000) if dtype == "i32" else ("normal", 0.0, 1.0)
    t = gar_inputs.rank_inputs(P, n, dtype, dist, 5 * P + n % 1000 + S, device="cuda" if P * n > 1 << 24 else "cpu")
    pad = -n % 8
    store = torch.zeros((P, n + pad), dtype=t.dtype, device="cpu" if where == "pinned" else "cuda")
    store = store.pin_memory() if where == "pinned" else store
    store[:, :n].copy_(t)
    plan = gar.gar_plan_create(P, n, dtype, op, S)
    rows = gar.rank_pointer_array([store[x] for x in range(P)])
    if where == "pinned":
        dev = torch.empty((P, n + pad), dtype=t.dtype, device="cuda")
        gar.gar_allreduce_host(plan, rows, rows, gar.rank_pointer_array([dev[x] for x in range(P)]), "fused")
    else:
        gar.gar_allreduce(plan, rows, "fused")
    torch.cuda.synchronize()
    assert gar.gar_plan_get_info(plan)["fused_form"] == gar.GAR_FORM_STREAM
    assert gar.gar_plan_status(plan) == gar.GAR_OK
    q, rem = divmod(n, P)
    starts = np.array([b * q + min(b, rem) for b in range(P)])
    rng = np.random.default_rng(n)
    near = (starts[:, None] + np.arange(-9, 10)).ravel()
    pos = np.unique(np.concatenate([near, np.arange(n - 20, n), rng.integers(0, n, samples), np.arange(300)]))
    pos = pos[(pos >= 0) & (pos < n)]
    idx = torch.from_numpy(pos).to(t.device)
    cols = [t[x][idx] for x in range(P)]
    host = np.zeros((P, n), np.int32 if dtype == "i32" else np.float32) if P * n < 1 << 22 else None
    if host is None:                     # the oracle on the sampled columns' own blocks
        want = _sampled(cols, pos, P, n, S, op, dtype)
    else:
        for x in range(P):
            host[x, pos] = cols[x].float().cpu().numpy() if dtype != "i32" else cols[x].cpu().numpy()
        want = G.allreduce(list(host), S, op, dtype, elements=pos)
    got = store[:, :n][:, torch.from_numpy(pos).to(store.device)].cpu()
    got = got.numpy() if dtype == "i32" else got.float().numpy()
    for x in range(P):
        w = np.asarray(want[x], got.dtype)
        assert np.array_equal(got[x].view(np.uint32), w.view(np.uint32)), (P, n, dtype, S, x)
    assert not store[:, n:].any()


def _sampled(cols, pos, P, n, S, op, dtype):
    full = []
    for c in cols:
        v = np.zeros(n, np.float32)
        v[pos] = c.float().cpu().numpy()
        full.append(v)
    return G.allreduce(full, S, op, dtype, elements=pos)


CASES = [(5, 5 * 512 + d, dt, op, S) for d, dt, op, S in
         [(0, "bf16", "sum", 3), (1, "bf16", "sum", 4), (2, "f32", "sum", 4), (3, "bf16", "max", 5), (4, "i32", "sum", 4)]]
CASES += [(2, 1024, "bf16", "sum", 1), (3, 3 * 515 + 2, "f32", "sum", 3), (13, 13 * 517 + 6, "bf16", "sum", 5),
          (24, 24 * 1000 + 7, "bf16", "sum", 6), (7, 7 * 60001 + 4, "f32", "sum", 4), (40, 40 * 3001 + 11, "bf16", "sum", 7),
          (127, 127 * 519 + 5, "bf16", "sum", 8), (200, 200 * 512 + 9, "bf16", "sum", 8)]


@pytest.mark.parametrize("P,n,dtype,op,S", CASES)
def test_stream_form(P, n, dtype, op, S, monkeypatch):
    monkeypatch.setenv("GAR_TUNE_FUSED_FORM", "3")
    _check(P, n, dtype, op, S)


@pytest.mark.parametrize("groups,ring", [(1, 1), (2, 2), (2, 3), (3, 4), (4, 7)])
def test_stream_rings(groups, ring, monkeypatch):
    """Several rounds of rings that groups share and that they do not."""
    monkeypatch.setenv("GAR_TUNE_FUSED_FORM", "3")
    monkeypatch.setenv("GAR_TUNE_ST_GROUPS", str(groups))
    monkeypatch.setenv("GAR_TUNE_ST_RING", str(ring))
    _check(5, 5 * 400003 + 3, "bf16", "sum", 4)


@pytest.mark.parametrize("P,n,dtype,S", [(5, 5 * 30001 + 2, "bf16", 4), (24, 24 * 5003 + 1, "f32", 6)])
def test_stream_form_on_host_vectors(P, n, dtype, S, monkeypatch):
    monkeypatch.setenv("GAR_TUNE_FUSED_FORM", "3")
    _check(P, n, dtype, "sum", S, where="pinned")


@pytest.mark.parametrize("P,n,dtype,S", [(127, (1 << 19) + 13, "bf16", 7), (110, (1 << 19) + 2, "bf16", 8),
                                         (120, (1 << 20) + 1, "f32", 7)])
def test_plans_that_take_the_stream_form(P, n, dtype, S):
    _check(P, n, dtype, "sum", S, samples=500)


@pytest.mark.parametrize("P,n,dtype,op,S", [(24, 24 * 1000 + 7, "bf16", "sum", 6), (24, 24 * 1000 + 7, "f32", "sum", 6),
                                            (24, 24 * 1000 + 7, "bf16", "max", 6), (127, 127 * 519 + 5, "bf16", "sum", 7)])
def test_special_values(P, n, dtype, op, S, monkeypatch):
    """Infinities, NaN, signed zeros, subnormals and overflowing sums: the bits of the
    single-thread form (order of combines and roundings are the schedule's in both)."""
    g = torch.Generator().manual_seed(P + n + S)
    big = 3.0e38
    values = torch.tensor([0.0, -0.0, 1.0, -1.0, 1e-40, -1e-40, 9e-41, big, -big, float("inf"), -float("inf"), float("nan")])
    # the large and non-finite values are rare: most positions stay finite
    weights = torch.tensor([8.0, 8, 8, 8, 8, 8, 8, 0.1, 0.1, 0.1, 0.1, 0.1])
    x = values[torch.multinomial(weights, P * n, replacement=True, generator=g)].view(P, n)
    x[:, ::3] = x[:, ::3].clamp(-2e-40, 2e-40).nan_to_num()       # subnormal sums
    pad = -n % 8
    got = []
    for form in (0, 3):
        monkeypatch.setenv("GAR_TUNE_FUSED_FORM", str(form))
        store = torch.zeros((P, n + pad), dtype=getattr(torch, {"bf16": "bfloat16", "f32": "float32"}[dtype]), device="cuda")
        store[:, :n] = x.cuda()
        plan = gar.gar_plan_create(P, n, dtype, op, S)
        gar.gar_allreduce(plan, gar.rank_pointer_array([store[r] for r in range(P)]), "fused")
        torch.cuda.synchronize()
        assert gar.gar_plan_get_info(plan)["fused_form"] == form
        got.append(store.view(torch.int16 if dtype == "bf16" else torch.int32).cpu())
    assert torch.equal(got[0], got[1])
