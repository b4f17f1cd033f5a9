"""Structural GPU probes with closed-form answers derived from the mask alone.  Random-input
parity cannot see one missing or doubled tile in a long row (it moves O and LSE by about
128 / n); these probes can: every executed tile leaves its own mark on every row."""
import numpy as np
import pytest
import torch

from paper_2607_09385_b200 import binding, inputs

import helpers as H

pytestmark = pytest.mark.gpu
CAUSAL, WINDOW, BITMAP = inputs.MASK_CAUSAL, inputs.MASK_WINDOW, inputs.MASK_BITMAP


def expected_mass(w, bitmap, h, rows):
    """For Q = 0 and V[j, c] = [(j // block) % d == c]: O[i, c] = visible keys of row i in key blocks
    congruent to c, divided by the number n_i of visible keys; LSE_i = ln n_i.  Built from the
    predicate (causal / window intervals, bitmap bits) with torch ops, independent of the planner."""
    dev = rows.device
    T, bm, d = w.seq // w.block, w.block, w.head_dim
    i = rows[:, None].to(torch.int64)
    blk_lo = (torch.arange(T, device=dev, dtype=torch.int64) * bm)[None, :]
    hi = torch.full_like(i, w.seq - 1)
    lo = torch.zeros_like(i)
    if w.flags & CAUSAL:
        hi = torch.minimum(hi, i)
    if w.flags & WINDOW:
        lo = torch.maximum(lo, i - w.window + 1)
    vis = (torch.minimum(hi, blk_lo + bm - 1) - torch.maximum(lo, blk_lo) + 1).clamp_(min=0).float()
    if w.flags & BITMAP:
        words = torch.from_numpy(bitmap[h].astype(np.int64)).to(dev)            # [T, words]
        J = torch.arange(T, device=dev)
        bits = ((words[:, J >> 5] >> (J & 31)[None, :]) & 1).float()            # [T_q, T_kv]
        vis = vis * bits[(rows // bm).long()]
    n = vis.sum(dim=1)
    pad = (-T) % d
    if pad:
        vis = torch.nn.functional.pad(vis, (0, pad))
    mass = vis.view(vis.shape[0], -1, d).sum(dim=1)
    return mass / n[:, None], torch.log(n)


@pytest.mark.parametrize("name", ["c1", "c2", "c3", "c4", "c5"])
def test_mass_per_block_probe_all_rows(name):
    w = inputs.workload(name)
    bitmap = inputs.block_bitmap(w.heads_q, w.tiles, w.tiles, w.keep_prob) if w.flags & BITMAP else None
    attn = H.make_attention(w, bitmap)
    q = torch.zeros((w.batch, w.heads_q, w.seq, w.head_dim), dtype=torch.bfloat16, device="cuda")
    k = torch.randn((w.batch, w.heads_kv, w.seq, w.head_dim), device="cuda").to(torch.bfloat16)
    j = torch.arange(w.seq, device="cuda")
    v1 = torch.nn.functional.one_hot((j // w.block) % w.head_dim, w.head_dim).to(torch.bfloat16)
    v = v1[None, None].expand(w.batch, w.heads_kv, -1, -1).contiguous()
    o = torch.full_like(q, float("nan"))
    lse = torch.full((w.batch, w.heads_q, w.seq), float("nan"), device="cuda")
    attn.run(q, k, v, o, lse)
    assert attn.last_status() == binding.STEEL_OK
    chunk = 8192
    for h in range(w.heads_q):
        for r0 in range(0, w.seq, chunk):
            rows = torch.arange(r0, min(r0 + chunk, w.seq), device="cuda")
            exp_o, exp_lse = expected_mass(w, bitmap, h, rows)
            got = o[0, h, rows].float()
            assert torch.allclose(got, exp_o, rtol=6e-3, atol=1e-6), (name, h, r0, (got - exp_o).abs().max().item())
            assert torch.allclose(lse[0, h, rows], exp_lse, rtol=0, atol=2e-5 * max(1.0, float(exp_lse.max())))
    attn.close()


@pytest.mark.parametrize("flags,window,block", [(CAUSAL, 0, 128), (CAUSAL | WINDOW, 384, 128),
                                                (CAUSAL | WINDOW, 200, 128), (CAUSAL | BITMAP, 0, 64)])
def test_dominant_key_probe(flags, window, block):
    """One key scores far above all others for every query: rows that see it return its V row
    (bf16-exact), rows that do not return the plain average of what they see.  Checks mask edges
    (diagonal, window edge i - j = W - 1 vs W, bitmap bit order) at token resolution."""
    S, D, H_ = 1024, 128, 2
    w = inputs.Workload("dom", 1, H_, H_, S, D, block, flags, window=window, keep_prob=0.5)
    bitmap = inputs.block_bitmap(H_, S // block, S // block, 0.5, seed=3) if flags & BITMAP else None
    rng = np.random.default_rng(1)
    for jstar in (0, 127, 128, 300, 511, 640, 1023):
        q = np.zeros((1, H_, S, D), np.float32)
        k = np.zeros((1, H_, S, D), np.float32)
        q[..., 5] = 16.0
        k[0, :, jstar, 5] = 16.0                      # score 256 * scale on key j*, 0 elsewhere
        v = rng.standard_normal((1, H_, S, D)).astype(np.float32)
        data = {"q": inputs.f32_to_bf16_bits(q), "k": inputs.f32_to_bf16_bits(k),
                "v": inputs.f32_to_bf16_bits(v), "bitmap": bitmap}
        attn, o, lse = H.run_gpu(w, data, scale=1.0)
        vb = inputs.bf16_bits_to_f64(data["v"])
        og = o.float().cpu().numpy()
        for h in range(H_):
            i = np.arange(S)
            sees = i >= jstar if flags & CAUSAL else np.ones(S, bool)
            if flags & WINDOW:
                sees &= (i - jstar) < window
            if flags & BITMAP:
                sees &= np.array([inputs.bitmap_bit(bitmap, h, r // block, jstar // block) for r in i])
            assert np.array_equal(og[0, h, sees], np.broadcast_to(vb[0, h, jstar], (int(sees.sum()), D)).astype(np.float32))
            # rows that do not see j* : uniform average over their visible keys (oracle checks values)
        rows = np.array([(0, h, r) for h in range(H_) for r in (0, 1, 127, 128, 129, 255, 256, 400, 639, 640, 641, 1023)])
        H.assert_parity(w, data, o, lse, rows, scale=1.0)
        attn.close()


@pytest.mark.parametrize("direction", ["increasing", "decreasing", "spikes"])
def test_rescale_stress(direction):
    """Scores ramp with the key index so the running maximum grows at every tile (every step
    rescales O), shrinks at every tile (never rescales), or jumps by far more than the lazy
    threshold at scattered keys."""
    S, D = 2048, 128
    w = inputs.Workload("ramp", 1, 2, 1, S, D, 128, 0 if direction == "spikes" else CAUSAL)
    rng = np.random.default_rng(2)
    q = rng.standard_normal((1, 2, S, D)).astype(np.float32) * 0.1
    k = rng.standard_normal((1, 1, S, D)).astype(np.float32) * 0.1
    v = rng.standard_normal((1, 1, S, D)).astype(np.float32)
    q[..., 0] = 8.0
    ramp = np.arange(S, dtype=np.float32) / S * 12.0          # score ramp of about 96 * scale ... large
    if direction == "increasing":
        k[0, 0, :, 0] = ramp
    elif direction == "decreasing":
        k[0, 0, :, 0] = ramp[::-1]
    else:
        k[0, 0, rng.choice(S, 24, replace=False), 0] = rng.uniform(4.0, 16.0, 24).astype(np.float32)
    data = {"q": inputs.f32_to_bf16_bits(q), "k": inputs.f32_to_bf16_bits(k), "v": inputs.f32_to_bf16_bits(v),
            "bitmap": None}
    attn, o, lse = H.run_gpu(w, data, scale=1.0)
    H.assert_parity(w, data, o, lse, H.all_rows(w), scale=1.0)
    attn.close()


def test_rows_masked_in_their_first_tile():
    """Window mask whose far-left partial tile hides every key from the last rows of a query tile
    while their running maximum is still -inf: no NaN, parity holds (W a multiple of the tile)."""
    w = inputs.Workload("farleft", 1, 2, 2, 1024, 128, 128, CAUSAL | WINDOW, window=256)
    data = inputs.make_inputs(w, seed=77)
    attn, o, lse = H.run_gpu(w, data)
    assert not torch.isnan(o.float()).any() and not torch.isnan(lse).any()
    H.assert_parity(w, data, o, lse, H.all_rows(w))
    attn.close()


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("seq", [1, 129, 300])
def test_output_at_any_16_byte_boundary(head_dim, seq):
    """O may start at any multiple of 16 bytes; where it is no multiple of 32 the stores are narrower, the bytes the same."""
    g = torch.Generator(device="cuda").manual_seed(head_dim + seq)
    q, k, v = (torch.randn((2, 3, seq, head_dim), generator=g, device="cuda").to(torch.bfloat16) for _ in "qkv")
    attn = binding.SteelAttention(2, 3, 3, seq, seq, head_dim, 0.125, CAUSAL)
    outs = []
    for offset in (0, 8):  # elements of 2 bytes
        room = torch.full((q.numel() + 16,), float("nan"), dtype=torch.bfloat16, device="cuda")
        o = room[offset:offset + q.numel()].view(q.shape)
        assert o.data_ptr() % 32 == 2 * offset
        attn.run(q, k, v, o)
        assert attn.last_status() == binding.STEEL_OK
        assert room[:offset].isnan().all() and room[offset + q.numel():].isnan().all()  # nothing beside it
        outs.append(o)
    assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_a_score_that_is_no_number_reaches_its_rows_from_every_column(head_dim, value):
    """At head_dim 64 some columns of a tile take another exponential than the others.  A key that is NaN or infinite must
    show in every row that sees it, whatever its column, and in no other row."""
    g = torch.Generator(device="cuda").manual_seed(head_dim)
    q, k, v = (torch.rand((1, 1, 128, head_dim), generator=g, device="cuda").to(torch.bfloat16) for _ in "qkv")  # q > 0
    attn = binding.SteelAttention(1, 1, 1, 128, 128, head_dim, 0.125, CAUSAL)
    o_ref, lse_ref = attn.run(q, k, v)
    for j in range(128):
        bad = k.clone()
        bad[0, 0, j] = value
        o, lse = attn.run(q, bad, v)
        assert o[0, 0, j:].isnan().all(), j
        assert torch.equal(o[0, 0, :j], o_ref[0, 0, :j]) and torch.equal(lse[0, 0, :j], lse_ref[0, 0, :j]), j


def test_far_apart_scores_at_head_dim_64():
    """Scores from one to far below the smallest number's logarithm beneath the maximum, in every column: weights that
    vanish are exactly 0, the others right to bf16's rounding (V is one-hot in the key's column, so O is the weight)."""
    n, d = 64, 64
    q = torch.zeros((1, 1, 128, d), device="cuda")
    q[0, 0, :, 0] = torch.arange(128, device="cuda") * 2.0   # steepness per row
    k = torch.zeros((1, 1, n, d), device="cuda")
    k[0, 0, :, 0] = -torch.arange(n, device="cuda")          # score of key j: -2 * row * j (exact in bf16)
    v = torch.eye(n, device="cuda")[None, None]
    attn = binding.SteelAttention(1, 1, 1, 128, n, d, 0.5, 0)
    o, lse = attn.run(q.to(torch.bfloat16), k.to(torch.bfloat16), v.to(torch.bfloat16))
    y = -(torch.arange(128, dtype=torch.float64)[:, None] * torch.arange(n, dtype=torch.float64)[None])
    p = torch.softmax(y, 1)
    got = o[0, 0].double().cpu()
    # P and O are rounded to bf16: 8 significant bits, so at most half of 2^-7 each, relative, and (1 + 2^-8)^2 together;
    # the exponentials and the fp32 row sum add less than 2^-20
    assert (got - p).abs().le(p * (2.0 ** -7 + 2.0 ** -16 + 2.0 ** -20) + 1e-37).all()
    assert (got[p < 1e-45] == 0).all()
    assert torch.allclose(lse[0, 0].double().cpu(), torch.logsumexp(y, 1), rtol=0, atol=2e-6)  # fp32 values up to 4.2


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("size", [2.0 ** 33, 2.0 ** 37, 2.0 ** 44])
def test_weights_beyond_the_largest_number_are_infinite_in_every_column(head_dim, size):
    """Scaled scores so large that rounding the running maximum leaves exponents of 128 and more: 2 to their power is
    infinite, and the row must show it (no row of such scores is right), whatever the column of the key."""
    d, scale = head_dim, 1.1
    a = 1.0 + torch.arange(128, device="cuda") / 128.0                    # exact in bf16
    q, k, v = (torch.zeros((1, 1, 128, d), device="cuda") for _ in "qkv")
    q[0, 0, :, 0] = a
    v[0, 0, :, 1] = 1.0
    # the exponent that is left of the largest score: its product with scale * log2(e) less that product rounded
    scale_log2 = float(np.float32(scale) * np.float32(1.4426950408889634))
    product = (a.double().cpu() * size * scale_log2).numpy()              # 8 and 24 bits: exact
    left = torch.from_numpy(product - product.astype(np.float32).astype(np.float64))
    rows = left >= 128.5
    assert rows.sum() > 20
    attn = binding.SteelAttention(1, 1, 1, 128, 128, d, scale, 0)
    for j in range(128):
        k.zero_()
        k[0, 0, j, 0] = size
        o, lse = attn.run(q.to(torch.bfloat16), k.to(torch.bfloat16), v.to(torch.bfloat16))
        assert not o[0, 0].cpu()[rows][:, 1].isfinite().any(), j
        assert (lse[0, 0].cpu()[rows] == float("inf")).all(), j
