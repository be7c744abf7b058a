"""The Allreduce calls that this library is timed on, through its public entry points.

A case names an entry point and the sizes of one call; `prepare` makes the rank vectors on
the GPU (in pinned host memory for the host-buffer call), the plan, and the pointer array
or descriptor table that a program keeps from call to call; `run` makes the one call.
`gar_allreduce` works in place, as MPI_Allreduce does with MPI_IN_PLACE: a second pass over
one state reduces the results of the first.

The sizes are the ones the paper experiments with (P = 127 processes; 425 B, 9 KB and
growing messages), the gradient-bucket-sized workload of 24 x 64 MiB, and the smaller and
ragged ones between them.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_2004_09362_gb300 import gar

SIZE = {"f32": 4, "bf16": 2, "i32": 4}
TORCH = {"f32": torch.float32, "bf16": torch.bfloat16, "i32": torch.int32}
MIB = 1 << 20
LARGEST = 24 * 64 * MIB          # bytes of all rank vectors of the largest listed case


def _levels(P: int) -> int:
    return (P - 1).bit_length()


def listed():
    return [
        # The smallest call: 4 KiB per rank among 5 ranks, default (bandwidth-optimal)
        # schedule.  A scalar loss or a norm being reduced; latency and launches only.
        {"name": "fused_p5_4kib_f32", "call": "fused", "P": 5, "n": 1024, "dtype": "f32", "op": "sum", "S": 6},
        # The paper's average message, 425 B among 127 processes, with the default schedule
        # of a program that names no step count: blocks of one or two elements.
        {"name": "fused_p127_425b_bf16", "call": "fused", "P": 127, "n": 212, "dtype": "bf16", "op": "sum", "S": 14},
        # The paper's 9 KB message at a step count between the two ends.
        {"name": "fused_p127_9kib_bf16", "call": "fused", "P": 127, "n": 4608, "dtype": "bf16", "op": "sum", "S": 10},
        # A gradient bucket: 24 x 64 MiB fp32, bandwidth-optimal.  The largest case.
        {"name": "fused_p24_64mib_f32", "call": "fused", "P": 24, "n": 16777216, "dtype": "f32", "op": "sum", "S": 10},
        # 127 x 8 MiB bf16, latency-optimal: every rank its own result copy, the most
        # arithmetic per byte that the step range has.
        {"name": "fused_p127_8mib_bf16_lo", "call": "fused", "P": 127, "n": 4194304, "dtype": "bf16", "op": "sum", "S": 7},
        # The same vectors in the middle of the step range (16 result copies).
        {"name": "fused_p127_8mib_bf16_mid", "call": "fused", "P": 127, "n": 4194304, "dtype": "bf16", "op": "sum", "S": 10},
        # Every schedule step as its own launch, on large bf16 vectors (HBM-bound) ...
        {"name": "step_p127_8mib_bf16", "call": "step", "P": 127, "n": 4194304, "dtype": "bf16", "op": "sum", "S": 14},
        # ... and on small ones, 9 KB among 127 ranks, where step boundaries count.
        {"name": "step_p127_9kib_bf16", "call": "step", "P": 127, "n": 4608, "dtype": "bf16", "op": "sum", "S": 10},
        # The steps in one cooperative launch: ragged int32 vectors of about 4 MiB, max.
        {"name": "persistent_p24_4mib_i32_max", "call": "persistent", "P": 24, "n": 1048583, "dtype": "i32", "op": "max", "S": 10},
        # The call for programs that may not allocate: 1 MiB per rank, between the two ends
        # of the step range (its partial results fill most of the fixed scratch array).
        {"name": "noalloc_p20_1mib_f32", "call": "noalloc", "P": 20, "n": 262147, "dtype": "f32", "op": "sum", "S": 9},
        # Thousands of independent 425-byte Allreduces of 6 and 7 ranks in one launch.
        {"name": "batched_65536x425b_f32", "call": "batched", "P": 6, "P2": 7, "count": 65536, "n": 106, "dtype": "f32", "op": "sum", "S": 3},
        # Vectors in pinned host memory, results back in host memory.
        {"name": "host_p24_4mib_f32", "call": "host", "P": 24, "n": 1048576, "dtype": "f32", "op": "sum", "S": 10},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["fused", "fused", "fused", "fused", "step", "step", "persistent", "noalloc", "batched", "host"])
    dtype = rng.choice(["f32", "f32", "bf16", "bf16", "i32"])
    op = rng.choice(["sum", "sum", "sum", "max", "min"])
    if call == "batched":
        P, P2 = rng.sample(range(2, 17), 2)
        n = _log_uniform(rng, 16, 4096)
        most = 400 * MIB // (max(P, P2) * n * SIZE[dtype])
        return {"call": call, "P": P, "P2": P2, "count": _log_uniform(rng, 16, min(100000, most)), "n": n, "dtype": dtype, "op": op,
                "S": _levels(max(P, P2)) if _levels(P) == _levels(P2) else 0}
    P = _log_uniform(rng, 2, 64 if call == "noalloc" else 127)
    L = _levels(P)
    S = rng.choice([2 * L, 2 * L, 2 * L, L, rng.randint(L, 2 * L), -3])
    if 2 * (P - 1) > 2 * L and rng.random() < 0.1:
        S = 2 * rng.randint(L + 1, P - 1)               # a fold schedule
    group = "xor" if P & (P - 1) == 0 and call != "noalloc" and L <= S <= 2 * L and rng.random() < 0.5 else "cyclic"
    # bytes of all rank vectors: as the largest listed case at most; the schedules that keep
    # several result copies move many times their vectors' bytes when every step is run
    most = LARGEST // 2
    if call in ("step", "persistent") and L <= S < 2 * L:
        most = 96 * MIB
    if call == "persistent":
        most = min(most, 256 * MIB)
    if call == "noalloc":
        most = 64 * MIB // (3 * 4) * SIZE[dtype]          # what the scratch array holds
    if call == "host":
        most = 192 * MIB
    n = _log_uniform(rng, 100, most // (P * SIZE[dtype]) - 64)
    if rng.random() < 0.3:
        n = max(64, n // 64 * 64)
    return {"call": call, "P": P, "n": n, "dtype": dtype, "op": op, "S": S, "group": group}


def _ranks(case):
    """(ranks of each instance, how many instances have them), in memory order."""
    if case["call"] != "batched":
        return [(case["P"], 1)]
    half = case["count"] // 2
    return [(case["P"], half), (case["P2"], case["count"] - half)]


def _values(count, dtype, seed):
    """Gradient-like values: normal in the float types, small whole numbers in int32."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    if dtype == "i32":
        return torch.randint(-1000, 1001, (count,), generator=gen, device="cuda", dtype=torch.int32)
    x = torch.randn(count, generator=gen, device="cuda", dtype=torch.float32)
    return x.mul_(1e-3) if dtype == "f32" else x.to(torch.bfloat16)


def _inputs(case, seed):
    """The rank vectors [P, n], rows padded to 16 bytes; a batch's instances back to back."""
    if case["call"] == "batched":
        return _values(sum(P * count for P, count in _ranks(case)) * case["n"], case["dtype"], seed)
    P, n = case["P"], case["n"]
    pad = -n % (16 // SIZE[case["dtype"]])
    return _values(P * (n + pad), case["dtype"], seed).view(P, n + pad)[:, :n]


def _plan(case, P, S):
    if case.get("group", "cyclic") == "xor":
        return gar.gar_plan_create_group(P, case["n"], case["dtype"], case["op"], S, "xor")
    return gar.gar_plan_create(P, case["n"], case["dtype"], case["op"], S)


def prepare(case, seed):
    call = case["call"]
    x = _inputs(case, seed)
    if call == "batched":
        out = torch.empty_like(x)
        plans, index, ptrs, at = [], [], [], 0
        for k, (P, count) in enumerate(_ranks(case)):
            plans.append(_plan(case, P, case["S"] if case["S"] >= _levels(P) else gar.GAR_STEPS_LO))
            step = P * case["n"] * SIZE[case["dtype"]]
            index.append(np.full(count, k))
            ptrs.append(at + step * np.arange(count, dtype=np.uint64))
            at += step * count
        index, ptrs = np.concatenate(index), np.concatenate(ptrs).astype(np.uint64)
        desc = gar.make_batch_desc(index, ptrs + np.uint64(x.data_ptr()), ptrs + np.uint64(out.data_ptr()))
        state = {"call": call, "plans": plans, "desc": desc, "count": case["count"], "in": x, "out": out}
        gar.gar_allreduce_batched(plans, desc, case["count"])   # compiles the plans' kernel
        torch.cuda.synchronize()
        out.zero_()
        return state
    plan = _plan(case, case["P"], case["S"])
    if call == "host":
        pinned = []
        for src in (x, None):
            rows = torch.empty((x.shape[0], x.stride(0)), dtype=x.dtype, pin_memory=True)[:, : x.shape[1]]
            if src is not None:
                rows.copy_(src)
            pinned.append(rows)
        gar.gar_plan_prepare(plan, "fused")
        host = [gar.rank_pointer_array(rows) for rows in pinned]
        # device buffers: the call uses them where the GPU cannot address the host rows itself
        return {"call": call, "plan": plan, "in": pinned[0], "out": pinned[1], "dev": x,
                "ptrs": host + [gar.rank_pointer_array(x)]}
    if call in ("step", "persistent"):
        gar.ensure_workspace(plan)
    gar.gar_plan_prepare(plan, "step" if call == "noalloc" else call)
    return {"call": call, "plan": plan, "out": x, "ptrs": gar.rank_pointer_array(x)}


def run(state):
    call = state["call"]
    if call == "batched":
        gar.gar_allreduce_batched(state["plans"], state["desc"], state["count"])
    elif call == "host":
        gar.gar_allreduce_host(state["plan"], *state["ptrs"], "fused")
    elif call == "noalloc":
        gar.gar_allreduce_noalloc(state["plan"], state["ptrs"])
    else:
        gar.gar_allreduce(state["plan"], state["ptrs"], call)
    return state["out"]


def work(case):
    """Every input read once, every result written once, P - 1 combines per position."""
    values = sum(P * count for P, count in _ranks(case)) * case["n"]
    combines = sum((P - 1) * count for P, count in _ranks(case)) * case["n"]
    return {"bytes": 2 * values * SIZE[case["dtype"]], "flops": combines}


def _reduce(x, op, dim):
    if op == "sum":
        return x.sum(dim, keepdim=True)
    return x.amax(dim, keepdim=True) if op == "max" else x.amin(dim, keepdim=True)


def exact(case, seed):
    x = _inputs(case, seed)
    wide = torch.int64 if case["dtype"] == "i32" else torch.float64
    if case["call"] == "batched":
        parts, at = [], 0
        for P, count in _ranks(case):
            size = P * count * case["n"]
            part = x[at: at + size].view(count, P, case["n"]).to(wide)
            parts.append(_reduce(part, case["op"], 1).expand_as(part).reshape(-1))
            at += size
        got = torch.cat(parts)
    else:
        total = None
        for row in x:
            row = row.to(wide)
            if total is None:
                total = row
            elif case["op"] == "sum":
                total = total + row
            else:
                total = torch.maximum(total, row) if case["op"] == "max" else torch.minimum(total, row)
        got = total.expand(x.shape)
    return got.to(torch.int32) if case["dtype"] == "i32" else got
