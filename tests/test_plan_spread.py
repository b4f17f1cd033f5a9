"""Plans that pack the heads of a group into query tiles and cut key ranges over CTAs: every key tile that a
query tile sees is executed exactly once, with the right mask flag, and the parts of a cut tile are numbered
completely.  The visible tiles come from the mask's definition, row by row.  CPU only."""
import numpy as np
import pytest

CAUSAL, WINDOW, BITMAP = 1, 2, 4

# ctas, batch, heads_q, heads_kv, seq_q, seq_kv, flags, window, kept share of a bitmap's blocks, and what the plan is
# to show: packed heads, fewest and most parts of a cut query tile (0, 0: none is cut)
CASES = [
    (148, 8, 32, 8, 1, 6001, CAUSAL, 0, 0, (1, 4, 4)), (148, 1, 8, 1, 3, 1000, CAUSAL, 0, 0, (1, 0, 0)),
    (148, 2, 12, 4, 8, 40, 0, 0, 0, (1, 0, 0)), (148, 1, 32, 8, 500, 12500, CAUSAL, 0, 0, (0, 3, 3)),
    (148, 1, 3, 1, 129, 129, CAUSAL, 0, 0, (1, 0, 0)), (148, 1, 6, 2, 200, 900, CAUSAL | WINDOW, 150, 0, (1, 0, 0)),
    (148, 1, 4, 1, 40, 5000, WINDOW, 600, 0, (1, 0, 0)), (148, 1, 12, 12, 512, 512, 0, 0, 0, (0, 0, 0)),
    (148, 1, 1, 1, 256, 256, CAUSAL, 0, 0, (0, 0, 0)), (148, 1, 1, 1, 1, 32768, 0, 0, 0, (0, 64, 64)),
    (148, 1, 2, 1, 300, 100, CAUSAL, 0, 0, (0, 0, 0)), (4, 1, 5, 5, 1000, 1000, CAUSAL, 0, 0, (0, 0, 0)),
    (3, 2, 4, 2, 700, 2000, CAUSAL, 0, 0, (1, 0, 0)), (148, 1, 2, 1, 2048, 2048, CAUSAL | BITMAP, 0, 0.4, (0, 0, 0)),
    (148, 1, 2, 2, 128, 8192, BITMAP, 0, 0.6, (0, 6, 6)), (148, 16, 128, 16, 8, 4096, CAUSAL, 0, 0, (1, 0, 0)),
    (7, 1, 7, 1, 130, 3000, 0, 0, 0, (1, 0, 0)), (148, 1, 1, 1, 16384, 16384, CAUSAL, 0, 0, (0, 2, 5)),
    (148, 1, 16, 4, 2048, 2048, CAUSAL, 0, 0, (0, 0, 0)), (148, 16, 16, 16, 1, 3000, CAUSAL, 0, 0, (0, 2, 4)),
    (148, 1, 2, 2, 8192, 8192, BITMAP | CAUSAL, 0, 0.3, (0, 0, 0)),
    (148, 1, 4, 2, 300, 9000, CAUSAL | WINDOW, 5000, 0, (1, 6, 7)), (148, 1, 4, 4, 128, 9000, WINDOW, 6000, 0, (0, 8, 8)),
    (148, 1, 32, 16, 700, 4000, CAUSAL, 0, 0, (1, 2, 2)),
]


@pytest.mark.parametrize("case", CASES)
def test_every_visible_key_tile_exactly_once(plan_dump, case):
    ctas, batch, hq, hkv, sq, skv, flags, window, keep, shown = case
    tq, tkv = -(-sq // 128), -(-skv // 128)
    bits, words = np.ones((hq, tq, tkv), bool), []
    if flags & BITMAP:
        bits = np.random.default_rng(2).random((hq, tq, tkv)) < keep
        packed_bits = np.zeros((hq, tq, -(-tkv // 32)), np.uint32)
        for h, i, j in zip(*np.nonzero(bits)):
            packed_bits[h, i, j >> 5] |= np.uint32(1 << (j & 31))
        words = packed_bits.ravel()
    out = plan_dump(ctas, batch, hq, hkv, sq, skv, flags, window, 128, words)
    grid, packed, n_parts, n_items = (int(x) for x in out[0].split()[1:])
    assert grid <= ctas and n_items == sum(l.startswith("item") for l in out)
    splits = [tuple(int(x) for x in l.split()[1:]) for l in out if l.startswith("split")]
    assert sum(n for _, n in splits) == n_parts and all(2 <= n <= 64 for _, n in splits)
    assert [f for f, _ in splits] == list(np.cumsum([0] + [n for _, n in splits])[:-1])
    counts = [n for _, n in splits] or [0]
    assert (packed, min(counts), max(counts)) == shown
    seen, parts, tiles = {}, {}, set()
    for l in out[1:]:
        if l.startswith("item"):
            _, n_steps, _, lo0, hi0, lo1, hi1 = (int(x) for x in l.split()[1:])
            if hi0 >= lo0 and hi1 >= lo1:
                assert lo0 <= lo1
            assert max(hi0, hi1 if hi1 >= lo1 else -1) == n_steps - 1
        if l.startswith("slot"):
            f = l.split()
            s, b, head, tile, split = (int(x) for x in f[1:6])
            tiles.add((b, head, tile))
            if split >= 0:
                parts.setdefault(split >> 6, []).append((split & 63, b, head, tile))
            for e in f[6:]:
                j, partial = (int(x) for x in e.split(":"))
                assert (b, head, tile, j) not in seen
                seen[b, head, tile, j] = partial
    assert len(parts) == len(splits)
    for n, (_, count) in enumerate(splits):
        assert sorted(x[0] for x in parts[n]) == list(range(count)) and len({x[1:] for x in parts[n]}) == 1
    # the same from the definition: row r of a matrix is query r % sq of its head
    heads, rows = (hkv, hq // hkv * sq) if packed else (hq, sq)
    keys = np.arange(skv)
    for tile in range(-(-rows // 128)):
        pos = (np.arange(tile * 128, min(tile * 128 + 128, rows)) % sq)[:, None] + skv - sq
        vis = np.ones((len(pos), skv), bool)
        if flags & CAUSAL:
            vis &= keys[None] <= pos
        if flags & WINDOW:
            vis &= pos - keys[None] < window
        for j in range(tkv):
            block = vis[:, j * 128:j * 128 + 128]
            partial = int(not block.all() or block.shape[1] < 128)
            for b in range(batch):
                for h in range(heads):
                    kept = block.any() and (not flags & BITMAP or bits[h, tile, j])
                    assert (b, h, tile) in tiles
                    assert seen.get((b, h, tile, j)) == (partial if kept else None), (b, h, tile, j)
