"""Calls whose plan packs the heads of a group into query tiles or cuts key ranges over CTAs, against the
oracle: one row per matrix, row counts that are not a multiple of 4, rows of several heads in one tile, two to
64 parts, windows and bitmaps of both block sizes cut into parts, rows without a visible key in a part or at all,
software exponents.  Each case states what its plan shows.  Repeated calls are bit-identical (the parts are combined
in a fixed order, whichever ends last), also after a call that was interrupted and beside other runs of the handle."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2607_09385_b200 import binding as B
from paper_2607_09385_b200 import inputs

import helpers as H

pytestmark = pytest.mark.gpu
CAUSAL, WINDOW, BITMAP = inputs.MASK_CAUSAL, inputs.MASK_WINDOW, inputs.MASK_BITMAP

CASES = [  # batch, heads_q, heads_kv, seq_q, seq_kv, head_dim, flags, window, emulation
    (2, 32, 8, 1, 6001, 128, CAUSAL, 0, 0), (3, 16, 16, 1, 3000, 64, CAUSAL, 0, 0), (1, 1, 1, 1, 32768, 128, 0, 0, 0),
    (1, 8, 1, 3, 1000, 64, CAUSAL, 0, 0), (2, 10, 2, 7, 5000, 128, CAUSAL, 0, 2), (1, 4, 1, 40, 5000, 64, WINDOW, 600, 0),
    (1, 8, 2, 500, 6500, 128, CAUSAL, 0, 0), (1, 6, 2, 200, 900, 128, CAUSAL | WINDOW, 150, 0),
    (1, 1, 1, 3000, 3000, 128, CAUSAL, 0, 0), (1, 3, 1, 129, 2500, 64, 0, 0, 1), (1, 4, 2, 60, 20, 128, CAUSAL, 0, 0),
    (1, 2, 1, 400, 4096, 64, BITMAP, 0, 0),
]
# what the plan of each shows: packed heads, fewest and most parts of a cut query tile (0, 0: none is cut)
SHOWN = [(1, 18, 18), (0, 6, 6), (0, 64, 64), (1, 0, 0), (1, 12, 12), (1, 0, 0), (0, 8, 8), (1, 0, 0), (0, 0, 0),
         (1, 0, 0), (1, 0, 0), (0, 0, 0)]

CUT = [  # the same with the block size of the mask, what its bitmap holds, and what the plan shows
    (1, 32, 16, 700, 4000, 128, CAUSAL, 0, 0, 128, None, (1, 2, 2)),
    (8, 16, 16, 1, 2000, 64, CAUSAL, 0, 0, 128, None, (0, 2, 2)),
    (1, 4, 2, 300, 9000, 64, CAUSAL | WINDOW, 5000, 0, 128, None, (1, 6, 7)),
    (1, 4, 4, 128, 9000, 128, WINDOW, 6000, 0, 128, None, (0, 8, 8)),
    (1, 2, 2, 128, 8192, 128, BITMAP, 0, 0, 128, "random", (0, 4, 4)),
    (1, 2, 2, 128, 8192, 128, BITMAP, 0, 0, 64, "ends", (0, 4, 8)),
    (1, 2, 2, 128, 8192, 64, BITMAP, 0, 3, 64, "ends", (0, 4, 8)),
    (1, 4, 2, 300, 6000, 64, BITMAP | CAUSAL, 0, 0, 64, "random", (0, 6, 7)),
]


def block_bitmap(case):
    """"random": half of the blocks.  "ends", two rows of blocks: the first keeps only early keys, the second only late
    ones, so that parts hold rows without a visible key; the last head keeps nothing in its second row."""
    _, hq, _, sq, skv, _, _, _, _, block, kind, _ = case
    tq, tkv = -(-sq // block), -(-skv // block)
    bits = np.random.default_rng(2).random((hq, tq, -(-tkv // 32) * 32)) < 0.5
    if kind == "ends":
        bits[:] = False
        bits[:, 0, :48] = True
        bits[:, 1, tkv - 48:tkv] = True
        bits[-1, 1] = False
    weight = np.uint64(1) << np.arange(32, dtype=np.uint64)
    return (bits.reshape(hq, tq, -1, 32).astype(np.uint64) * weight).sum(3).astype(np.uint32)


def make(case, seed=5, block=128, bitmap=None):
    b, hq, hkv, sq, skv, d, flags, window, emu = case
    rng = np.random.default_rng(seed)
    q, k, v = (torch.from_numpy(rng.standard_normal(s, np.float32)).to(torch.bfloat16)
               for s in ((b, hq, sq, d), (b, hkv, skv, d), (b, hkv, skv, d)))
    if flags & BITMAP and bitmap is None:
        bitmap = rng.integers(0, 1 << 32, (hq, -(-sq // 128), -(-skv // 4096)), dtype=np.uint32)
    args = (b, hq, hkv, sq, skv, d, 1.0 / math.sqrt(d), flags)
    attn = B.SteelAttention(*args, block=block, window=window, bitmap=bitmap, exp_emulation=emu)
    p = oracle.OracleProblem(*args, block, block, window, bitmap)
    return attn, p, q, k, v


def compare_with_oracle(attn, p, q, k, v):
    dev = [x.cuda() for x in (q, k, v)]
    o = torch.full_like(dev[0], float("nan"))
    lse = torch.full(q.shape[:3], float("nan"), device="cuda")
    attn.run(*dev, o, lse)
    assert attn.last_status() == B.STEEL_OK
    rows = oracle.steel_oracle.all_rows(p)
    if len(rows) > 400:
        rows = rows[np.sort(np.random.default_rng(1).choice(len(rows), 400, replace=False))]
    bits = [x.view(torch.int16).numpy().view(np.uint16) for x in (q, k, v)]
    o_ref, lse_ref = oracle.rows(p, *bits, rows)
    at = tuple(torch.from_numpy(rows[:, c].astype(np.int64)) for c in range(3))
    o_gpu, lse_gpu = o.float().cpu()[at].numpy(), lse.cpu()[at].numpy()
    err = np.abs(o_gpu - o_ref)
    assert err.max() <= H.TOL_O_MAX and err.mean() <= H.TOL_O_MEAN
    seen = np.isfinite(lse_ref)
    assert np.array_equal(np.isfinite(lse_gpu), seen) and np.abs(lse_gpu[seen] - lse_ref[seen]).max(initial=0) <= H.TOL_LSE
    for _ in range(3):
        o2, lse2 = attn.run(*dev)
        assert torch.equal(o2, o) and torch.equal(lse2, lse)
    attn.close()


def assert_shown(lines, shown):
    counts = [int(x.split()[2]) for x in lines if x.startswith("split")] or [0]
    assert (int(lines[0].split()[2]), min(counts), max(counts)) == shown


@pytest.mark.parametrize("case,shown", list(zip(CASES, SHOWN)))
def test_against_oracle(case, shown, plan_dump):
    attn, p, q, k, v = make(case)
    b, hq, hkv, sq, skv, _, flags, window, _ = case
    words = p.bitmap.ravel() if flags & BITMAP else ()
    assert_shown(plan_dump(148, b, hq, hkv, sq, skv, flags, window, 128, words), shown)
    compare_with_oracle(attn, p, q, k, v)


@pytest.mark.parametrize("case", CUT)
def test_cut_masks_against_oracle(case, plan_dump):
    b, hq, hkv, sq, skv, _, flags, window, _, block, kind, shown = case
    bitmap = block_bitmap(case) if kind else None
    assert_shown(plan_dump(148, b, hq, hkv, sq, skv, flags, window, block, bitmap.ravel() if kind else ()), shown)
    compare_with_oracle(*make(case[:9], block=block, bitmap=bitmap))


def test_interrupted_call_leaves_nothing_behind():
    attn, _, q, k, v = make(CASES[6])
    dev = [x.cuda() for x in (q, k, v)]
    o, lse = attn.run(*dev)
    assert attn.last_status() == B.STEEL_OK
    B.steel_attn_debug_stall(attn.handle, 3, 200_000_000)  # 0.1 s
    attn.run(*dev)
    assert attn.last_status() == B.STEEL_ERR_TIMEOUT
    B.steel_attn_debug_stall(attn.handle, -1)
    for _ in range(2):
        o2, lse2 = attn.run(*dev)
        assert attn.last_status() == B.STEEL_OK
        assert torch.equal(o2, o) and torch.equal(lse2, lse)
    attn.close()


@pytest.mark.parametrize("case", [CASES[0], CASES[1], CASES[6]])  # 18, 6 and 8 parts per tile: batches of 4 and a rest
@pytest.mark.parametrize("what", ["v", "q", "k"])
def test_infinite_and_nan_operands_as_in_an_uncut_plan(case, what):
    """One infinite value of V, one row of NaN in Q or in K: infinities and NaN of O and LSE do not depend on
    the plan (policy 1 never packs or cuts)."""
    attn, _, q, k, v = make(case)
    b, hq, hkv, sq, skv, d, flags, window, emu = case
    if what == "v":
        v[0, 0, skv - sq, 3] = math.inf  # every query sees this key
    elif what == "q":
        q[0, 0, sq // 2] = math.nan
    else:
        k[0, 0, skv // 2] = math.nan
    dev = [x.cuda() for x in (q, k, v)]
    uncut = B.SteelAttention(b, hq, hkv, sq, skv, d, 1.0 / math.sqrt(d), flags, policy=1)
    (o, lse), (o_ref, lse_ref) = attn.run(*dev), uncut.run(*dev)
    assert attn.last_status() == B.STEEL_OK and uncut.last_status() == B.STEEL_OK
    for x, y in ((o, o_ref), (lse, lse_ref)):
        assert torch.equal(x.isnan(), y.isnan()) and torch.equal(x.isposinf(), y.isposinf())
        assert torch.equal(x.isneginf(), y.isneginf())
    assert o.isposinf().any() if what == "v" else o.isnan().any()
    attn.close()
    uncut.close()


@pytest.mark.parametrize("case", [CASES[0], CASES[6]])
def test_calls_after_an_interrupted_one_need_no_repair(case):
    """A call whose waits expire, others queued behind it before anyone asks for the status: those are right."""
    attn, _, q, k, v = make(case)
    dev = [x.cuda() for x in (q, k, v)]
    o, lse = attn.run(*dev)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        for cta in (3, 0):
            B.steel_attn_debug_stall(attn.handle, cta, 200_000_000)  # 0.1 s
            attn.run(*dev)
            B.steel_attn_debug_stall(attn.handle, -1)
            later = [attn.run(*dev) for _ in range(3)]
            assert attn.last_status() == B.STEEL_ERR_TIMEOUT
            later += [attn.run(*dev) for _ in range(2)]
            assert attn.last_status() == B.STEEL_OK
            for o2, lse2 in later:
                assert torch.equal(o2, o) and torch.equal(lse2, lse)
    attn.close()


def several_inputs(case, n):
    """A handle, n sets of operands on the GPU, and each one's results from runs that nothing overlaps."""
    attn, _, q, k, v = make(case)
    sets = [[x.roll(m, -2).contiguous().cuda() for x in (q, k, v)] for m in range(n)]
    ref = []
    for dev in sets:
        ref.append(attn.run(*dev))
        torch.cuda.synchronize()
    assert attn.last_status() == B.STEEL_OK
    return attn, sets, ref


def outputs_like(ref, n):
    return [tuple(torch.full_like(x, float("nan")) for x in ref[m % len(ref)]) for m in range(n)]


@pytest.mark.parametrize("case", [CASES[0], CASES[6]])
def test_one_handle_on_several_streams(case):
    """Runs of a cut plan queued on four streams at once, beside work that holds part of the GPU."""
    attn, sets, ref = several_inputs(case, 5)
    streams = [torch.cuda.current_stream()] + [torch.cuda.Stream() for _ in range(3)]
    out = outputs_like(ref, 120)
    other = torch.randn((4096, 4096), device="cuda", dtype=torch.bfloat16)
    torch.cuda.synchronize()
    busy = torch.cuda.Stream()
    with torch.cuda.stream(busy):
        for _ in range(60):
            other @ other
    for n, (o, lse) in enumerate(out):
        with torch.cuda.stream(streams[n * 7 % 4]):
            if n < 4:
                torch.cuda._sleep(1_000_000)
            attn.run(*sets[n % 5], o, lse)
    torch.cuda.synchronize()
    assert attn.last_status() == B.STEEL_OK
    for n, (o, lse) in enumerate(out):
        assert torch.equal(o, ref[n % 5][0]) and torch.equal(lse, ref[n % 5][1]), n
    attn.close()


def test_cut_plan_in_graphs_that_overlap():
    """Two captured graphs, the first with two branches and a join, replayed beside each other and eager runs."""
    attn, sets, ref = several_inputs(CASES[0], 5)
    out = outputs_like(ref, 5)
    side, graphs = torch.cuda.Stream(), [torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()]
    torch.cuda.synchronize()
    with torch.cuda.graph(graphs[0]):
        here = torch.cuda.current_stream()
        side.wait_stream(here)
        with torch.cuda.stream(side):
            attn.run(*sets[0], *out[0])
        attn.run(*sets[1], *out[1])
        here.wait_stream(side)
        attn.run(*sets[2], *out[2])
    with torch.cuda.graph(graphs[1]):
        attn.run(*sets[3], *out[3])
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(20):
        for o, lse in out:
            o.fill_(float("nan"))
            lse.fill_(float("nan"))
        for g, stream in zip(graphs, streams):
            stream.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(stream):
                g.replay()
                g.replay()
        for _ in range(4):
            attn.run(*sets[4], *out[4])
        torch.cuda.synchronize()
        for (o, lse), (o_ref, lse_ref) in zip(out, ref):
            assert torch.equal(o, o_ref) and torch.equal(lse, lse_ref)
    assert attn.last_status() == B.STEEL_OK
    del graphs
    attn.close()


def test_more_captures_than_part_buffers():
    """Captures beyond the handle's bound run the plan without cuts: the same result within rounding."""
    attn, sets, ref = several_inputs(CASES[0], 3)
    out, graphs = outputs_like(ref, 36), []
    torch.cuda.synchronize()
    for n in range(36):
        graphs.append(torch.cuda.CUDAGraph())
        with torch.cuda.graph(graphs[-1]):
            attn.run(*sets[n % 3], *out[n])
    for g in graphs:
        g.replay()
    torch.cuda.synchronize()
    assert attn.last_status() == B.STEEL_OK
    exact = [torch.equal(o, ref[n % 3][0]) for n, (o, _) in enumerate(out)]
    assert all(exact[:30])
    for n, (o, lse) in enumerate(out):
        err = (o.float() - ref[n % 3][0].float()).abs()
        assert float(err.max()) <= H.TOL_O_MAX and float(err.mean()) <= H.TOL_O_MEAN
        assert float((lse - ref[n % 3][1]).abs().max()) <= H.TOL_LSE
    del graphs
    attn.close()
