"""The attention calls that the performance of this library is measured on.

Every case goes through the public classes and functions of `paper_2607_09385_b200.binding`: a plan built
once for the problem (what a program that serves one shape keeps), then calls on tensors it has at hand.
Shapes come from this repository's workload table (`inputs.WORKLOADS`, `inputs.paper_workloads()`), its
parity tests (few queries against many keys, ragged lengths, odd query groups, batches) and its benchmark
(host-memory calls); `draw` spreads over the ranges between them.

A case:
    entry   "run"      `SteelAttention.run` on device tensors, outputs allocated by the call
            "host"     `SteelAttentionHost.run` on page-locked host tensors, copies included
            "noalloc"  `steel_attn_run_noalloc`: plan, run and wait in one call, a mask that is new each time
    batch, heads_q, heads_kv, seq_q, seq_kv, head_dim
    mask    "dense", "causal", "window" (causal, `window` keys), "bitmap" (causal, `keep` of the blocks below
            the diagonal, blocks of `block` tokens)
"""
import math

import numpy as np
import torch

from paper_2607_09385_b200 import binding

FLAGS = {"dense": 0, "causal": binding.STEEL_MASK_CAUSAL,
         "window": binding.STEEL_MASK_CAUSAL | binding.STEEL_MASK_WINDOW,
         "bitmap": binding.STEEL_MASK_CAUSAL | binding.STEEL_MASK_BITMAP}


def _case(entry, batch, heads_q, heads_kv, seq_q, seq_kv, head_dim, mask, window=0, block=128, keep=0.0, name=None):
    c = dict(entry=entry, batch=batch, heads_q=heads_q, heads_kv=heads_kv, seq_q=seq_q, seq_kv=seq_kv,
             head_dim=head_dim, mask=mask, window=window, block=block, keep=keep)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call of the workload table: latency of one launch, one head
        _case("run", 1, 1, 1, 256, 256, 64, "causal", block=64, name="one_head_s256"),
        # an encoder layer on one short sequence: 48 query tiles, no mask
        _case("run", 1, 12, 12, 512, 512, 64, "dense", name="encoder_h12_d64_s512"),
        # decoder prefill at head_dim 64, a prompt of ordinary length
        _case("run", 1, 32, 32, 8192, 8192, 64, "causal", name="prefill_h32_d64_s8k"),
        # decoder prefill at head_dim 128, multi-head
        _case("run", 1, 32, 32, 4096, 4096, 128, "causal", name="prefill_h32_d128_s4k"),
        # a batch of prompts of odd length, query groups of three
        _case("run", 4, 24, 8, 1777, 1777, 128, "causal", name="batch4_gqa24x8_s1777"),
        # sliding-window layer of a long prompt, grouped queries
        _case("run", 1, 32, 8, 16384, 16384, 128, "window", window=4096, name="window4k_gqa32x8_s16k"),
        # block-sparse prefill of a long prompt, a pattern of its own for each head
        _case("run", 1, 16, 16, 32768, 32768, 128, "bitmap", keep=0.25, name="bitmap25_h16_s32k"),
        # the largest: a 128K-token prompt
        _case("run", 1, 32, 8, 131072, 131072, 128, "causal", name="prefill_gqa32x8_s128k"),
        # the next chunk of a prompt against the keys that are there already
        _case("run", 1, 32, 8, 500, 12500, 128, "causal", name="chunk500_gqa32x8_kv12k"),
        # one decode step of a small batch, cache length not a multiple of anything
        _case("run", 8, 32, 8, 1, 6001, 128, "causal", name="decode_b8_gqa32x8_kv6k"),
        # operands and results in host memory
        _case("host", 1, 32, 32, 4096, 4096, 128, "causal", name="host_h32_d128_s4k"),
        # a block mask that is new at every call (planning counts), 64-token blocks
        _case("noalloc", 1, 8, 8, 4096, 4096, 64, "bitmap", block=64, keep=0.25, name="new_bitmap64_h8_s4k"),
    ]


def _log(rng, lo, hi):
    """An integer from lo to hi, spread over its logarithm."""
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(("prefill", "prefill", "prefill", "bitmap", "chunk", "decode", "host", "noalloc"))
    head_dim = rng.choice((64, 128))
    heads_kv = rng.choice((1, 2, 4, 8, 12, 16))
    group = rng.choice((1, 2, 3, 4, 8))
    heads_q = heads_kv * group
    if kind == "prefill":
        seq = _log(rng, 128, 32768)
        batch = rng.choice((1, 2, 4, 8)) if seq <= 4096 else 1
        mask = rng.choice(("dense", "causal", "causal", "window"))
        window = _log(rng, 64, max(64, seq // 2)) if mask == "window" else 0
        return _case("run", batch, heads_q, heads_kv, seq, seq, head_dim, mask, window)
    if kind == "bitmap":
        return _case("run", 1, heads_q, heads_kv, *[_log(rng, 1024, 16384)] * 2, head_dim, "bitmap",
                     block=rng.choice((64, 128)), keep=round(rng.uniform(0.1, 0.6), 3))
    if kind in ("chunk", "decode"):
        seq_q = _log(rng, 16, 2048) if kind == "chunk" else rng.randint(1, 8)
        seq_kv = seq_q + _log(rng, 256, 32768)
        batch = rng.choice((1, 2, 4)) if kind == "chunk" else _log(rng, 1, 16)
        return _case("run", batch, heads_q, heads_kv, seq_q, seq_kv, head_dim, "causal")
    if kind == "host":
        seq = _log(rng, 256, 8192)
        return _case("host", rng.choice((1, 2, 4)), min(heads_q, 32), min(heads_kv, min(heads_q, 32)) if
                     min(heads_q, 32) % heads_kv == 0 else 1, seq, seq, head_dim, rng.choice(("dense", "causal")))
    return _case("noalloc", 1, min(heads_q, 16), 1 if min(heads_q, 16) % heads_kv else heads_kv,
                 *[_log(rng, 512, 4096)] * 2, head_dim, "bitmap", block=rng.choice((64, 128)),
                 keep=round(rng.uniform(0.1, 0.6), 3))


def _bitmap(case, generator):
    """Words [heads_q][T_q][ceil(T_kv / 32)]: the diagonal and key block 0 kept, of the others `keep`."""
    t = -(-case["seq_q"] // case["block"])
    words = -(-t // 32)
    bits = torch.rand((case["heads_q"], t, words * 32), generator=generator, device="cuda") < case["keep"]
    i, j = torch.arange(t, device="cuda")[:, None], torch.arange(words * 32, device="cuda")[None, :]
    bits = (bits & (j < i)) | (j == i) | ((j == 0) & (j <= i))
    packed = (bits.view(case["heads_q"], t, words, 32).to(torch.int64) << torch.arange(32, device="cuda")).sum(3)
    return packed.cpu().numpy().astype(np.uint32)


def _inputs(case, seed):
    """q, k, v on the GPU and the bitmap's words (None for the other masks), from the seed alone."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    b, hq, hkv, sq, skv, d = (case[x] for x in ("batch", "heads_q", "heads_kv", "seq_q", "seq_kv", "head_dim"))

    def normal(heads, seq):
        out = torch.empty((b, heads, seq, d), dtype=torch.bfloat16, device="cuda")
        for n in range(b):
            for h in range(heads):
                out[n, h] = torch.randn((seq, d), generator=g, device="cuda")
        return out

    q, k, v = normal(hq, sq), normal(hkv, skv), normal(hkv, skv)
    # heads differ in how peaked their scores are
    q *= (0.5 + torch.rand((hq, 1, 1), generator=g, device="cuda")).to(torch.bfloat16)
    return q, k, v, _bitmap(case, g) if case["mask"] == "bitmap" else None


def prepare(case, seed):
    q, k, v, bitmap = _inputs(case, seed)
    b, hq, hkv, sq, skv, d = (case[x] for x in ("batch", "heads_q", "heads_kv", "seq_q", "seq_kv", "head_dim"))
    args = (b, hq, hkv, sq, skv, d, 1.0 / math.sqrt(d), FLAGS[case["mask"]])
    state = {"entry": case["entry"], "q": q, "k": k, "v": v}
    if case["entry"] == "run":
        state["attn"] = binding.SteelAttention(*args, block=case["block"], window=case["window"], bitmap=bitmap)
    elif case["entry"] == "host":
        for x in "qkv":
            state[x] = torch.empty(state[x].shape, dtype=torch.bfloat16, pin_memory=True).copy_(state[x])
        state["o"] = torch.empty(q.shape, dtype=torch.bfloat16, pin_memory=True)
        state["lse"] = torch.empty(q.shape[:3], dtype=torch.float32, pin_memory=True)
        state["attn"] = binding.SteelAttentionHost(*args, block=case["block"], window=case["window"], bitmap=bitmap,
                                                   max_chunks=8)
    else:
        state["params"], state["bitmap"] = binding.make_params(*args, case["block"], case["block"], case["window"],
                                                               bitmap)
    return state


def run(state):
    q, k, v = state["q"], state["k"], state["v"]
    if state["entry"] == "run":
        return state["attn"].run(q, k, v)
    if state["entry"] == "host":
        state["attn"].run(q, k, v, state["o"], state["lse"])
        # the result is read on the host: the program waits for it
        torch.cuda.current_stream().synchronize()
        return state["o"], state["lse"]
    o, lse = torch.empty_like(q), torch.empty(q.shape[:3], dtype=torch.float32, device=q.device)
    status = binding.steel_attn_run_noalloc(state["params"], q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(),
                                            lse.data_ptr(), torch.cuda.current_stream().cuda_stream)
    if status != binding.STEEL_OK:
        raise binding.SteelError(status, "steel_attn_run_noalloc")
    return o, lse


def _visible_pairs(case):
    """Visible (query, key) pairs of one query head (for a bitmap: their expected number)."""
    sq, skv, off = case["seq_q"], case["seq_kv"], case["seq_kv"] - case["seq_q"]
    if case["mask"] == "dense":
        return float(sq) * skv
    seen = np.arange(sq, dtype=np.int64) + off + 1
    if case["mask"] == "causal":
        return float(seen.sum())
    if case["mask"] == "window":
        return float(np.minimum(seen, case["window"]).sum())
    n, t = case["block"], -(-sq // case["block"])
    below = sum(1 + (i - 1) * case["keep"] for i in range(1, t))  # blocks left of the diagonal
    return below * n * n + t * n * (n + 1) / 2


def work(case):
    d, b, hq, hkv = case["head_dim"], case["batch"], case["heads_q"], case["heads_kv"]
    keys = case["seq_kv"] if case["mask"] != "window" else min(case["seq_kv"], case["seq_q"] - 1 + case["window"])
    return {"bytes": 2.0 * d * b * (2 * hq * case["seq_q"] + 2 * hkv * keys) + 4.0 * b * hq * case["seq_q"],
            "flops": 4.0 * d * b * hq * _visible_pairs(case)}


def tolerance(case):
    # bf16 operands, P and O rounded to bf16.  Against attention in float64 on the same operands, O of the
    # listed and of drawn cases is off by 2.0e-3 to 2.4e-3 (2-norm) and by at most 0.035 of the larger of the
    # value and the root mean square; LSE by 2e-6.  Four times that.
    return {"rel": 1e-2, "max": 0.14}


def exact(case, seed):
    """O and LSE in float64 from the same operands: explicit scores, mask and softmax over blocks of query rows."""
    b, hq, hkv, sq, skv, d = (case[x] for x in ("batch", "heads_q", "heads_kv", "seq_q", "seq_kv", "head_dim"))
    if 1.0 * b * hq * sq * skv * d > 2e13:  # over about 20 s
        return None
    q, k, v, bitmap = _inputs(case, seed)
    o = torch.empty((b, hq, sq, d), dtype=torch.float64, device="cuda")
    lse = torch.empty((b, hq, sq), dtype=torch.float64, device="cuda")
    keys = torch.arange(skv, device="cuda")
    rows = max(1, min(sq, (1 << 28) // skv))
    for i0 in range(0, sq, rows):
        i1 = min(i0 + rows, sq)
        # a key block's end bounds what these rows see under a causal mask; the first key, under a window
        pos = torch.arange(i0, i1, device="cuda") + (skv - sq)
        end = skv if case["mask"] == "dense" else min(skv, i1 + skv - sq)
        begin = max(0, i0 + skv - sq - case["window"] + 1) if case["mask"] == "window" else 0
        seen = torch.ones((i1 - i0, end - begin), dtype=torch.bool, device="cuda")
        if case["mask"] != "dense":
            seen &= keys[None, begin:end] <= pos[:, None]
        if case["mask"] == "window":
            seen &= pos[:, None] - keys[None, begin:end] < case["window"]
        for n in range(b):
            for h in range(hq):
                kept = seen
                if bitmap is not None:
                    words = torch.from_numpy(bitmap[h].astype(np.int64)).cuda()
                    n_j = -(-end // case["block"])
                    j = torch.arange(n_j, device="cuda")
                    i_blocks = torch.arange(i0, i1, device="cuda") // case["block"]
                    bits = ((words[i_blocks][:, j >> 5] >> (j & 31)) & 1).bool()
                    kept = seen & bits.repeat_interleave(case["block"], 1)[:, :end]
                g = h // (hq // hkv)
                s = q[n, h, i0:i1].double() @ k[n, g, begin:end].double().T
                s *= 1.0 / math.sqrt(d)
                s.masked_fill_(~kept, -math.inf)
                lse[n, h, i0:i1] = torch.logsumexp(s, 1)
                o[n, h, i0:i1] = s.sub_(lse[n, h, i0:i1, None]).exp_() @ v[n, g, begin:end].double()
    return o, lse
