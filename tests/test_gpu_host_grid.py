"""Fused Allreduce of pinned host vectors on the capped grid: every thread takes several
vectors, with a ragged end, in the 32-thread single-copy form, the rotated and unrotated
many-copy forms and the breadth-first form; bit for bit against the oracle at both ends of
the vectors and on sampled positions between."""

import numpy as np
import pytest
import torch

import gar_inputs
from oracle import gar_oracle as G

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2004_09362_gb300 import gar


@pytest.mark.parametrize("P,S,dtype,form", [(40, 12, "bf16", None), (40, 9, "f32", None), (40, 6, "bf16", 0),
                                            (40, 6, "bf16", 1), (2, 1, "f32", None)])
def test_host_vectors_on_the_capped_grid(P, S, dtype, form, monkeypatch):
    if form is not None:
        monkeypatch.setenv("GAR_TUNE_FUSED_FORM", str(form))
    n = 900011 if P == 2 else 200011
    t = gar_inputs.rank_inputs(P, n, dtype, ("normal", 0.0, 1.0), 3 * P + S)
    rows = [torch.empty((P, n + 13), dtype=t.dtype, pin_memory=True) for _ in range(2)]
    rows[0][:, :n].copy_(t)
    rows[1].zero_()
    plan = gar.gar_plan_create(P, n, dtype, "sum", S)
    ptrs = [gar.rank_pointer_array([r[x, :n] for x in range(P)]) for r in rows]
    dev = torch.empty((P, n + 13), dtype=t.dtype, device="cuda")
    gar.gar_allreduce_host(plan, ptrs[0], ptrs[1], gar.rank_pointer_array([dev[x] for x in range(P)]), "fused")
    torch.cuda.synchronize()
    rng = np.random.default_rng(P)
    pos = np.unique(np.concatenate([np.arange(300), np.arange(n - 300, n), rng.integers(0, n, 2000)]))
    host = [t[x].float().numpy() for x in range(P)]
    want = G.allreduce(host, S, "sum", dtype, elements=pos)
    got = rows[1]
    for x in range(P):
        g = got[x, :n].float().numpy()[pos]
        assert np.array_equal(g.view(np.uint32), np.asarray(want[x], np.float32).view(np.uint32)), f"rank {x}"
    assert not got[:, n:].any()
