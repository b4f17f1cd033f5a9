"""The allocation-free entry point, called through the C ABI, against the handle-based one.

steel_attn_run_noalloc serves callers that may not allocate device memory (a locked framework
memory pool, a latency path that cannot take cudaMalloc's implicit synchronisation, a fixed memory
budget): its work lists live in a fixed array inside the library.  That array is shared by every
call and keeps the previous call's contents, so the test makes two calls in a row with different
problems and checks each against steel_attn_run on the same inputs.  This file is collected last
on purpose: a run that stops at the first failure has then already run every other test.
"""
import subprocess
import sys

import numpy as np
import pytest
import torch

from paper_2607_09385_b200 import binding as B
from paper_2607_09385_b200 import inputs

import helpers as H
from test_noalloc_plan import DEVICE_LISTS

pytestmark = pytest.mark.gpu
CAUSAL, WINDOW, BITMAP = inputs.MASK_CAUSAL, inputs.MASK_WINDOW, inputs.MASK_BITMAP


def run_both(w, seed):
    data = inputs.make_inputs(w, seed)
    q, k, v = (H.to_device(data[x]) for x in "qkv")
    # handle-based path
    attn = H.make_attention(w, data["bitmap"])
    o_ref, lse_ref = attn.run(q, k, v)
    assert attn.last_status() == B.STEEL_OK
    attn.close()
    # allocation-free path: no handle, outputs pre-filled so that unwritten rows would show
    params, keep = B.make_params(w.batch, w.heads_q, w.heads_kv, w.seq, w.seq, w.head_dim, w.scale, w.flags,
                                 w.block, w.block, w.window, data["bitmap"])
    o = torch.full_like(q, float("nan"))
    lse = torch.full((w.batch, w.heads_q, w.seq), float("nan"), dtype=torch.float32, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    args = (params, q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), lse.data_ptr(), stream)
    # The first call on a device loads the kernels and resolves the array's address, so it is made
    # before measuring.  torch's own counters cannot see an allocation made inside the library (its
    # CUDA runtime is linked statically and bypasses torch's caching allocator): the device's free
    # memory is compared instead, around a second call with no torch allocation in between.
    st = B.steel_attn_run_noalloc(*args)
    assert st == B.STEEL_OK, B.steel_status_string(st)
    torch.cuda.synchronize()
    free_before, _ = torch.cuda.mem_get_info()
    st = B.steel_attn_run_noalloc(*args)
    free_after, _ = torch.cuda.mem_get_info()
    assert st == B.STEEL_OK, B.steel_status_string(st)
    assert free_after == free_before, (free_before, free_after)
    # the same kernel; the plans may differ (this one never cuts key ranges), so the two paths agree within the
    # tolerances the parity tests use
    err_o = (o.float() - o_ref.float()).abs()
    assert not torch.isnan(o.float()).any() and not torch.isnan(lse).any()
    assert float(err_o.max()) <= H.TOL_O_MAX and float(err_o.mean()) <= H.TOL_O_MEAN
    fin = torch.isfinite(lse_ref)
    assert torch.equal(torch.isfinite(lse), fin)
    assert float((lse[fin] - lse_ref[fin]).abs().max()) <= H.TOL_LSE
    return data, o, lse


def test_noalloc_matches_handle_path_on_two_calls_in_a_row():
    # first call: bitmap mask (explicit step lists in the shared array), GQA
    w1 = inputs.Workload("noalloc_bitmap", 1, 4, 2, 2048, 128, 128, CAUSAL | BITMAP, keep_prob=0.35)
    d1, o1, lse1 = run_both(w1, seed=41)
    H.assert_parity(w1, d1, o1, lse1, H.sampled_rows(w1, range(4), 2, 32))
    # second call: a smaller causal-window problem with head_dim 64; stale lists of the first call
    # are still in the array when it starts
    w2 = inputs.Workload("noalloc_window", 2, 2, 1, 640, 64, 64, CAUSAL | WINDOW, window=200)
    d2, o2, lse2 = run_both(w2, seed=42)
    H.assert_parity(w2, d2, o2, lse2, H.all_rows(w2))
    # and the first problem again, after the second overwrote the lists
    run_both(w1, seed=41)


@pytest.mark.parametrize("shape", [(1, 8, 1, 3, 1000, 64), (1, 6, 2, 200, 900, 128), (2, 32, 8, 1, 6001, 128)])
def test_noalloc_with_packed_heads(shape):
    # rows of several heads in a query tile; the last one is also cut into key ranges by a handle, but not here
    b, hq, hkv, sq, skv, d = shape
    rng = np.random.default_rng(43)
    q, k, v = (torch.from_numpy(rng.standard_normal(s, np.float32)).to(torch.bfloat16).cuda()
               for s in ((b, hq, sq, d), (b, hkv, skv, d), (b, hkv, skv, d)))
    params, _ = B.make_params(b, hq, hkv, sq, skv, d, d ** -0.5, CAUSAL)
    o = torch.full_like(q, float("nan"))
    lse = torch.full(q.shape[:3], float("nan"), device="cuda")
    for _ in range(2):
        st = B.steel_attn_run_noalloc(params, q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), lse.data_ptr(),
                                      torch.cuda.current_stream().cuda_stream)
        assert st == B.STEEL_OK, B.steel_status_string(st)
    attn = B.SteelAttention(b, hq, hkv, sq, skv, d, d ** -0.5, CAUSAL)
    o_ref, lse_ref = attn.run(q, k, v)
    assert attn.last_status() == B.STEEL_OK
    err = (o.float() - o_ref.float()).abs()
    assert float(err.max()) <= H.TOL_O_MAX and float(err.mean()) <= H.TOL_O_MEAN
    assert float((lse - lse_ref).abs().max()) <= H.TOL_LSE
    if skv < 6001:  # the same plan
        assert torch.equal(o, o_ref) and torch.equal(lse, lse_ref)
    attn.close()


@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("shape,flags,window", [((2, 4, 2, 700, 1333, 64), CAUSAL | BITMAP, 0), ((1, 3, 3, 1000, 300, 128), BITMAP, 0),
                                                ((1, 6, 1, 129, 2001, 64), CAUSAL | WINDOW | BITMAP, 900)])
def test_noalloc_lists_written_on_the_device(shape, flags, window, block):
    # single query tiles under a bitmap: ragged and unequal lengths, tiles and rows without any visible key (the last two
    # shapes have so few entries that the host writes them; DEVICE_LISTS below has longer ones)
    b, hq, hkv, sq, skv, d = shape
    rng = np.random.default_rng(44)
    q, k, v = (torch.from_numpy(rng.standard_normal(s, np.float32)).to(torch.bfloat16).cuda()
               for s in ((b, hq, sq, d), (b, hkv, skv, d), (b, hkv, skv, d)))
    words = -(-(-(-skv // block)) // 32)
    bits = rng.integers(0, 2 ** 32, (hq, -(-sq // block), words), np.uint32) & rng.integers(0, 2 ** 32, (words,), np.uint32)
    bits[0, 0] = 0
    params, keep = B.make_params(b, hq, hkv, sq, skv, d, d ** -0.5, flags, block, block, window, bits)
    o = torch.full_like(q, float("nan"))
    lse = torch.full(q.shape[:3], float("nan"), device="cuda")
    st = B.steel_attn_run_noalloc(params, q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), lse.data_ptr(),
                                  torch.cuda.current_stream().cuda_stream)
    assert st == B.STEEL_OK, B.steel_status_string(st)
    attn = B.SteelAttention(b, hq, hkv, sq, skv, d, d ** -0.5, flags, block=block, window=window, bitmap=bits)
    o_ref, lse_ref = attn.run(q, k, v)
    assert attn.last_status() == B.STEEL_OK
    err = (o.float() - o_ref.float()).abs()
    assert not torch.isnan(o).any() and float(err.max()) <= H.TOL_O_MAX and float(err.mean()) <= H.TOL_O_MEAN
    fin = torch.isfinite(lse_ref)
    assert torch.equal(torch.isfinite(lse), fin) and float((lse[fin] - lse_ref[fin]).abs().max()) <= H.TOL_LSE
    attn.close()


@pytest.mark.parametrize("shape", DEVICE_LISTS)
def test_noalloc_longer_lists_written_on_the_device(shape):
    b, hq, hkv, sq, skv, flags, window, block = shape
    g = torch.Generator(device="cuda").manual_seed(sq)
    q, k, v = (torch.randn(s, generator=g, device="cuda").to(torch.bfloat16) for s in ((b, hq, sq, 64), (b, hkv, skv, 64), (b, hkv, skv, 64)))
    rng = np.random.default_rng(skv)
    bits = rng.integers(0, 2 ** 32, (hq, -(-sq // block), -(-(-(-skv // block)) // 32)), np.uint32)
    bits[0, 0] = 0
    params, keep = B.make_params(b, hq, hkv, sq, skv, 64, 0.125, flags, block, block, window, bits)
    o, lse = torch.full_like(q, float("nan")), torch.full(q.shape[:3], float("nan"), device="cuda")
    st = B.steel_attn_run_noalloc(params, q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), lse.data_ptr(),
                                  torch.cuda.current_stream().cuda_stream)
    assert st == B.STEEL_OK, B.steel_status_string(st)
    attn = B.SteelAttention(b, hq, hkv, sq, skv, 64, 0.125, flags, block=block, window=window, bitmap=bits)
    o_ref, lse_ref = attn.run(q, k, v)
    assert attn.last_status() == B.STEEL_OK
    err = (o.float() - o_ref.float()).abs()
    assert not torch.isnan(o).any() and float(err.max()) <= H.TOL_O_MAX and float(err.mean()) <= H.TOL_O_MEAN
    fin = torch.isfinite(lse_ref)
    assert torch.equal(torch.isfinite(lse), fin) and float((lse[fin] - lse_ref[fin]).abs().max()) <= H.TOL_LSE
    attn.close()


FIRST_CALLS = """
import numpy as np, torch
from paper_2607_09385_b200 import binding as B
q, k, v = (torch.randn((1, 8, 1024, 64), device="cuda").to(torch.bfloat16) for _ in "qkv")
o = torch.empty_like(q)
free = []
for flags, bits in ((B.STEEL_MASK_CAUSAL, None), (B.STEEL_MASK_CAUSAL | B.STEEL_MASK_BITMAP, np.full((8, 16, 1), 0xFFFFFFFF, np.uint32))):
    params, keep = B.make_params(1, 8, 8, 1024, 1024, 64, 0.125, flags, 64, 64, 0, bits)
    st = B.steel_attn_run_noalloc(params, q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), None,
                                  torch.cuda.current_stream().cuda_stream)
    assert st == B.STEEL_OK, st
    free.append(torch.cuda.mem_get_info()[0])
assert free[0] == free[1], free
"""


def test_noalloc_sets_up_in_the_first_call_only(repo_root):
    # the first call of a process has no bitmap; the first one with lists written on the device takes no memory either
    out = subprocess.run([sys.executable, "-c", FIRST_CALLS], cwd=repo_root, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr


def test_noalloc_rejects_plans_beyond_the_fixed_array():
    # 32 heads x 2048 query tiles = 32768 work items > 16384: refused, nothing launched
    params, _ = B.make_params(1, 32, 32, 262144, 262144, 128, 0.1, CAUSAL)
    t = torch.zeros(16, dtype=torch.bfloat16, device="cuda")
    st = B.steel_attn_run_noalloc(params, t.data_ptr(), t.data_ptr(), t.data_ptr(), t.data_ptr(), None, 0)
    assert st == B.STEEL_ERR_UNSUPPORTED
    assert B.steel_attn_run_noalloc(params, None, t.data_ptr(), t.data_ptr(), t.data_ptr(), None, 0) == B.STEEL_ERR_INVALID_ARG
