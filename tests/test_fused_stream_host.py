"""Host-side checks of the streaming fused kernel (GAR_FORM_STREAM, no GPU).

The generated evaluation function, run by a small interpreter in numpy float32, gives the
oracle's bits for every rank; so does the program table that evaluates the units the stream
leaves out; stream and table together cover every element position exactly once, for all
block layouts; every contribution is read after the wait for its part of the tile; NVRTC
compiles the kernels for sm_103a.
"""

import re

import numpy as np
import pytest

from oracle import gar_oracle as O
from paper_2004_09362_gb300 import gar as G


@pytest.fixture(autouse=True)
def _force(monkeypatch):
    monkeypatch.setenv("GAR_TUNE_FUSED_FORM", "3")


def _source(P, n, dtype, S, op="sum"):
    pl = G.gar_plan_create(P, n, dtype, op, S)
    info = G.gar_plan_get_info(pl)
    return G.gar_plan_fused_source(pl), info


def _block(n, P):
    q, rem = divmod(n, P)
    start = [b * q + min(b, rem) for b in range(P + 1)]
    return start, np.repeat(np.arange(P), np.diff(start))


def _combine(dtype, op):
    if dtype == "i32":
        return {"sum": lambda a, b: (a.astype(np.int64) + b).astype(np.int32), "max": np.maximum, "min": np.minimum}[op]
    return {"sum": lambda a, b: a + b, "max": np.maximum, "min": np.minimum}[op]


def _finish(v, dtype):
    return O.round_to_bf16(v) if dtype == "bf16" else v


def _run_stream(src, P, leaves, dtype, op):
    """Results by placement of one position (or an array of them) from contributions by
    index, through the text of gar_eval_st."""
    comb = _combine(dtype, op)
    body = re.search(r"bool gar_eval_st\(.*?\{\n(.*?)\n  return true;\n\}\n", src, re.S).group(1)
    part_rows = int(re.search(r"#define GAR_PART_ROWS (\d+)", src).group(1))
    here, out = set(), {}
    env = {"gar_open": lambda x: x, "gar_comb2": comb, "gar_combl": comb}

    def leaf(j):
        assert j // part_rows in here, f"contribution {j} read before its part has arrived"
        return leaves[j]

    env["L"] = leaf
    for line in body.split("\n"):
        line = line.strip()
        m = re.fullmatch(r"if \(!gar_wait\(handed, bar \+ (\d+), turn\)\) return false;", line)
        if m:
            here.add(int(m.group(1)) // 8)
            continue
        m = re.fullmatch(r"const gar_v (v\d+) = (.*);", line)
        if m:
            env[m.group(1)] = eval(re.sub(r"gar_leaf\(sl \+ (\d+) \* GAR_ROW\)", r"L(\1)", m.group(2)), env)
            continue
        m = re.fullmatch(r"gar_put\(gar_row\(rows \+ (\d+)\) \+ e, (v\d+)\);", line)
        assert m, line
        assert int(m.group(1)) // 8 not in out
        out[int(m.group(1)) // 8] = env[m.group(2)]
    assert sorted(out) == list(range(P))
    return [_finish(out[p], dtype) for p in range(P)]


def _run_table(src, P, leaves, dtype, op):
    comb = _combine(dtype, op)
    table = {k: [int(x) for x in re.search(k + r"\[\d+\] = \{([\d,]*)\}", src).group(1).split(",") if x]
             for k in ("gar_ops", "gar_ends", "gar_outs")}
    v = {j: leaves[j] for j in range(P)}
    k = 0
    for end in table["gar_ends"]:
        new = {}
        for t in range(k, end):
            o, a, b = table["gar_ops"][3 * t: 3 * t + 3]
            new[o] = comb(v[a], v[b])          # operands from earlier levels only
        v.update(new)
        k = end
    assert 3 * k == len(table["gar_ops"])
    return [_finish(v[x], dtype) for x in table["gar_outs"]]


def _inputs(P, n, dtype, seed):
    rng = np.random.default_rng(seed)
    if dtype == "i32":
        return [rng.integers(-2 ** 31, 2 ** 31, n).astype(np.int32) for _ in range(P)]
    xs = [(rng.standard_normal(n) * np.exp2(rng.integers(-12, 13, n))).astype(np.float32) for _ in range(P)]
    return [O.round_to_bf16(x) for x in xs] if dtype == "bf16" else xs


CASES = [(P, dt, op, S) for P in (2, 3, 5, 6, 7, 8, 12, 13, 24) for dt, op in (("bf16", "sum"), ("f32", "sum"))
         for S in range((P - 1).bit_length(), 2 * (P - 1).bit_length())]
CASES += [(7, "i32", "sum", 4), (13, "bf16", "max", 5), (12, "f32", "min", 4), (40, "bf16", "sum", 6), (40, "f32", "sum", 8),
          (100, "bf16", "sum", 8), (127, "bf16", "sum", 7), (127, "f32", "sum", 7), (127, "bf16", "sum", 9), (128, "bf16", "sum", 8)]


@pytest.mark.parametrize("P,dtype,op,S", CASES)
def test_stream_and_table_reproduce_the_oracle(P, dtype, op, S):
    """At sampled positions of every block, bit for bit, at ranks of every rotation."""
    n = P * 521 + P // 2
    src, info = _source(P, n, dtype, S, op)
    assert info["fused_form"] == G.GAR_FORM_STREAM and info["K"] > 1
    start, block = _block(n, P)
    blocks = range(P) if P <= 13 else sorted({0, 1, P // 2, P - 1})
    pos = np.array(sorted({start[b] + d for b in blocks for d in (0, 7, start[b + 1] - start[b] - 1)}))
    xs = [np.zeros(n, np.int32 if dtype == "i32" else np.float32) for _ in range(P)]
    for x, v in zip(xs, _inputs(P, len(pos), dtype, 31 * P + S)):
        x[pos] = v
    want = O.allreduce(xs, S, op, dtype, elements=pos)
    for i, e in enumerate(pos):
        b = int(block[e]) if info["K"] != P else 0
        leaves = [xs[(b + j) % P][e: e + 1] for j in range(P)]
        for got in (_run_stream(src, P, leaves, dtype, op), _run_table(src, P, leaves, dtype, op)):
            for p in range(P):
                w = np.asarray(want[(b + p) % P][i: i + 1], got[p].dtype)
                assert np.array_equal(got[p].view(np.uint32), w.view(np.uint32)), (P, S, dtype, int(e), p)


@pytest.mark.parametrize("P,dtype,S", [(5, "bf16", 3), (5, "bf16", 4), (7, "f32", 5), (3, "i32", 3), (24, "bf16", 7)])
def test_every_position_is_covered_once(P, dtype, S):
    """The positions that lanes of tiles evaluate and those that the table serves, by the
    kernel's own arithmetic, for block lengths of every residue: a partition of [0, n), and
    no 16-byte unit that is copied reaches past the last full one."""
    unit = 8 if dtype == "bf16" else 4
    width = 2 if dtype == "bf16" else 1
    tile = 512 // (2 if dtype == "bf16" else 4)
    for n in range(P * 512, P * 512 + 2 * unit * P + 1, max(1, P // 3)):
        src, info = _source(P, n, dtype, S)
        rotate = info["K"] != P
        start, block = _block(n, P)
        hi = n // unit * unit
        seen = np.zeros(n, np.int64)

        def whole(e):
            u = e // unit * unit
            b = block[u] if rotate else 0
            return not rotate or u + unit <= start[b + 1]

        for t in range((hi + tile - 1) // tile):
            for lane in range(128):
                e = t * tile + lane * width
                if e < hi and whole(e):
                    seen[e: e + width] += 1
        if n > hi:
            seen[hi:] += 1
        if rotate:
            for k in range(1, P):
                u = start[k] // unit * unit
                if u != start[k] and u < hi:
                    seen[u: u + unit] += 1
        assert (seen == 1).all(), (n, np.nonzero(seen != 1)[0][:5])


def test_interpreter_catches_planted_mistakes():
    """A result stored one placement off, and a wait moved behind its first read."""
    P, n, S = 7, 7 * 521 + 3, 4
    src, _ = _source(P, n, "f32", S)
    xs = [np.float32([np.exp2(7 * x - 20) * 1.37]) for x in range(P)]
    puts = re.findall(r"gar_put\(gar_row\(rows \+ (\d+)\) \+ e, (v\d+)\);", src)
    (_, v0), (row, v1) = puts[0], puts[-1]
    assert v0 != v1
    bad = src.replace(f"gar_put(gar_row(rows + {row}) + e, {v1});", f"gar_put(gar_row(rows + {row}) + e, {v0});")
    good, got = _run_stream(src, P, xs, "f32", "sum"), _run_stream(bad, P, xs, "f32", "sum")
    assert not np.array_equal(good[int(row) // 8], got[int(row) // 8])
    wait = re.search(r"  if \(!gar_wait\(handed, bar \+ 0, turn\)\) return false;\n", src).group(0)
    with pytest.raises(AssertionError, match="before its part"):
        _run_stream(src.replace(wait, "", 1), P, xs, "f32", "sum")


def test_selection_before_and_after_force(monkeypatch):
    """Forced plans only take the form where it applies; an unprepared plan reports the
    form of its first compile."""
    form = lambda *a: G.gar_plan_get_info(G.gar_plan_create(*a))["fused_form"]
    assert form(24, 24 * 512, "f32", "sum", 7) == G.GAR_FORM_STREAM
    assert form(24, 24 * 512 - 1, "f32", "sum", 7) == G.GAR_FORM_BREADTH      # blocks of 511 elements
    assert form(24, 24 * 512, "f32", "sum", 10) == G.GAR_FORM_SINGLE          # one result copy
    xor = G.gar_plan_create_group(8, 8 * 600, "f32", "sum", 4, "xor")
    assert G.gar_plan_get_info(xor)["fused_form"] == G.GAR_FORM_BREADTH
    monkeypatch.delenv("GAR_TUNE_FUSED_FORM")
    assert form(127, 4194304, "bf16", "sum", 7) == G.GAR_FORM_BREADTH


@pytest.mark.parametrize("P,S", [(2, 1), (3, 3), (5, 3), (8, 4), (13, 5), (33, 7), (127, 7), (200, 9)])
def test_stream_kernels_compile(P, S):
    for dtype, op in (("f32", "sum"), ("bf16", "sum"), ("i32", "max")) if P < 100 else (("bf16", "sum"),):
        G.gar_plan_compile(G.gar_plan_create(P, 513 * P + 1, dtype, op, S), "fused")
