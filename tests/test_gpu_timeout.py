"""Bounded device-side waits: when a role never gets what it waits for, the kernel gives up after
the configured number of cycles, returns normally and reports STEEL_ERR_TIMEOUT; the context and
the handle stay usable.  The stall is made with the library's test hook (one CTA's producer
withholds its commands); nothing faults, traps or spins without a limit."""
import time

import pytest
import torch

from paper_2607_09385_b200 import binding, inputs

import helpers as H

pytestmark = pytest.mark.gpu


def test_wait_expiry_sets_status_and_context_stays_usable():
    w = inputs.Workload("stall", 1, 4, 2, 1024, 128, 128, inputs.MASK_CAUSAL)
    data = inputs.make_inputs(w, seed=91)
    attn, o, lse = H.run_gpu(w, data)                      # normal run first
    q, k, v = (H.to_device(data[x]) for x in "qkv")
    binding.steel_attn_debug_stall(attn.handle, 0, 200_000_000)   # about 0.1 s of SM clock
    t0 = time.time()
    attn.run(q, k, v)
    status = attn.last_status()                            # synchronises the stream
    elapsed = time.time() - t0
    assert status == binding.STEEL_ERR_TIMEOUT
    assert elapsed < 30.0
    assert attn.last_status() == binding.STEEL_OK          # the status word was cleared by the read
    binding.steel_attn_debug_stall(attn.handle, -1, 0)     # hook off, default bound restored
    o2, lse2 = attn.run(q, k, v)
    assert attn.last_status() == binding.STEEL_OK
    assert torch.equal(o.view(torch.int16), o2.view(torch.int16)) and torch.equal(lse, lse2)
    H.assert_parity(w, data, o2, lse2, H.sampled_rows(w, range(4), 1, 32))
    with pytest.raises(binding.SteelError):
        binding.steel_attn_debug_stall(attn.handle, 10_000, 0)     # no such CTA
    attn.close()


def test_status_is_read_and_cleared_on_its_own_stream():
    """last_status on a side stream neither waits for nor is ordered with work on the default stream."""
    w = inputs.Workload("stall_side", 1, 4, 2, 1024, 128, 128, inputs.MASK_CAUSAL)
    data = inputs.make_inputs(w, seed=92)
    attn = H.make_attention(w)
    q, k, v = (H.to_device(data[x]) for x in "qkv")
    o = torch.empty_like(q)
    torch.cuda.synchronize()
    side, busy = torch.cuda.Stream(), torch.cuda.Event()
    for stalled in (True, False, True):
        binding.steel_attn_debug_stall(attn.handle, 0 if stalled else -1, 50_000_000)
        torch.cuda._sleep(2_000_000_000)                   # about a second of the default stream
        busy.record()
        with torch.cuda.stream(side):
            attn.run(q, k, v, o, want_lse=False)
            status = attn.last_status()
        assert not busy.query()
        assert status == (binding.STEEL_ERR_TIMEOUT if stalled else binding.STEEL_OK)
        torch.cuda.synchronize()
    binding.steel_attn_debug_stall(attn.handle, -1)
    attn.close()


@pytest.mark.parametrize("limit", [30_000_000, 300_000_000])
def test_the_bound_holds_where_only_softmax_warps_wait(limit):
    """Two key tiles per query tile: the stalled CTA's producer finds room for all of them in its ring and leaves, and so do
    the issuers, so that nothing but the softmax warps' own bound ends the launch."""
    q, k, v = (torch.randn((1, 1, 256, 128), device="cuda").to(torch.bfloat16) for _ in "qkv")
    attn = binding.SteelAttention(1, 1, 1, 256, 256, 128, 0.1, 0)
    o_ref, lse_ref = attn.run(q, k, v)
    torch.cuda.synchronize()
    binding.steel_attn_debug_stall(attn.handle, 0, limit)
    t0 = time.time()
    attn.run(q, k, v)
    assert attn.last_status() == binding.STEEL_ERR_TIMEOUT
    elapsed = time.time() - t0
    # below the highest clock (1.965 GHz) and above a low one; a wait is looked at after its first 64 polls
    assert limit / 2.0e9 * 0.99 < elapsed < limit / 0.3e9 + 2.0
    binding.steel_attn_debug_stall(attn.handle, -1, 0)
    o, lse = attn.run(q, k, v)
    assert attn.last_status() == binding.STEEL_OK
    assert torch.equal(o, o_ref) and torch.equal(lse, lse_ref)
    attn.close()
