"""Short launches overlap their set-up with the end of the launch before them on the stream.  In a chain of calls each
of which reads what the one before it wrote, queued without synchronisation, nothing may be read or overwritten early:
the chain has to give, bit for bit, what it gives with a synchronisation after every call."""
import math

import numpy as np
import pytest
import torch

from paper_2607_09385_b200 import binding as B
from paper_2607_09385_b200 import inputs

pytestmark = pytest.mark.gpu
CAUSAL = inputs.MASK_CAUSAL

# batch, heads_q, heads_kv, seq_q, seq_kv, head_dim: one tile; packed heads; packed and cut; cut; four tiles in a row
SHAPES = [(1, 1, 1, 128, 128, 64), (1, 8, 1, 3, 1000, 64), (2, 32, 8, 1, 6001, 128), (3, 16, 16, 1, 3000, 64),
          (1, 4, 4, 512, 512, 128)]
STEPS = 24


def operands(shape, seed):
    b, hq, hkv, sq, skv, d = shape
    rng = np.random.default_rng(seed)
    return [torch.from_numpy(rng.standard_normal(s, np.float32)).to(torch.bfloat16).cuda()
            for s in ((b, hq, sq, d), (b, hkv, skv, d), (b, hkv, skv, d))]


def chain(handles, shape, sync):
    """O of one call is Q of the next; torch kernels write K and V before each call, the handles take turns."""
    q, k0, v0 = operands(shape, 3)
    k, v = torch.empty_like(k0), torch.empty_like(v0)
    o, lse = [q], []
    for _ in range(STEPS):
        o.append(torch.full_like(q, float("nan")))
        lse.append(torch.full(q.shape[:3], float("nan"), device="cuda"))
    torch.cuda.synchronize()
    for n in range(STEPS):
        torch.mul(k0, 1.0 + n / 64, out=k)
        torch.add(v0, n, out=v) if n % 3 else v.copy_(v0)
        handles[n % len(handles)].run(o[n], k, v, o[n + 1], lse[n])
        if sync:
            torch.cuda.synchronize()
    torch.cuda.synchronize()
    return o[1:], lse


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("n_handles", [1, 2])
def test_chain_of_dependent_short_calls(shape, n_handles):
    args = (*shape, 1.0 / math.sqrt(shape[-1]), CAUSAL)
    handles = [B.SteelAttention(*args), B.SteelAttention(*args, policy=1)][:n_handles]
    assert handles[0].stats()["max_cta_steps"] <= 32  # launches that overlap
    ref = chain(handles, shape, sync=True)
    for _ in range(5):
        got = chain(handles, shape, sync=False)
        for x, y in zip(ref, got):
            for n in range(STEPS):
                assert torch.equal(x[n], y[n]), n
    for h in handles:
        assert h.last_status() == B.STEEL_OK
        h.close()


@pytest.mark.parametrize("shape", SHAPES)
def test_chain_without_other_kernels_in_between(shape):
    """Launch after launch of the same kernel, eagerly and as one captured graph."""
    attn = B.SteelAttention(*shape, 1.0 / math.sqrt(shape[-1]), CAUSAL)
    q, k, v = operands(shape, 4)
    ref = [q]
    for _ in range(STEPS):
        ref.append(attn.run(ref[-1], k, v)[0])
        torch.cuda.synchronize()
    out = [q] + [torch.full_like(q, float("nan")) for _ in range(STEPS)]
    lse = torch.empty(q.shape[:3], device="cuda")

    def queue():
        for n in range(STEPS):
            attn.run(out[n], k, v, out[n + 1], lse)

    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        queue()
    for once in (queue, graph.replay, queue, graph.replay):
        for x in out[1:]:
            x.fill_(float("nan"))
        once()
        torch.cuda.synchronize()
        for n in range(1, STEPS + 1):
            assert torch.equal(out[n], ref[n]), n
    assert attn.last_status() == B.STEEL_OK
    del graph
    attn.close()
