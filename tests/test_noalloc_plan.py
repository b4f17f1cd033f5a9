"""How steel_attn_run_noalloc lays out a call, from the planner.  CPU only."""
import os
import random
import subprocess

import pytest

CAUSAL, WINDOW, BITMAP = 1, 2, 4
# batch, heads, KV heads, queries, keys, flags, window, block: calls whose lists the device writes where about half of the
# bitmap's bits are set (tests/test_zz_no_alloc.py runs them)
DEVICE_LISTS = [(2, 4, 2, 700, 1333, CAUSAL | BITMAP, 0, 64), (1, 9, 9, 1000, 900, BITMAP, 0, 128),
                (1, 12, 2, 515, 4001, CAUSAL | WINDOW | BITMAP, 900, 64), (1, 5, 1, 130, 16500, BITMAP, 0, 64)]


@pytest.fixture(scope="module")
def noalloc_plan(tmp_path_factory, repo_root):
    exe = str(tmp_path_factory.mktemp("noalloc") / "noalloc_plan")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-o", exe, os.path.join(repo_root, "tests", "noalloc_plan.cpp"),
                           os.path.join(repo_root, "paper_2607_09385_b200", "csrc", "steel_planner.cpp")])

    def plan(*args):
        out = subprocess.check_output([exe, *map(str, args)], text=True).split()
        return out if out == ["refused"] else [int(x) for x in out]

    return plan


@pytest.mark.parametrize("shape,items,entries,device", [
    ((1, 1, 1, 256, 256, CAUSAL | BITMAP, 0, 64, "ffffffff"), 2, 3, 0),
    ((1, 1, 1, 512, 512, CAUSAL | BITMAP, 0, 64, "ffffffff"), 4, 10, 0),
    ((1, 4, 4, 512, 512, CAUSAL | BITMAP, 0, 128, "ffffffff"), 16, 40, 0),
    ((1, 1, 1, 1536, 1536, BITMAP, 0, 128, "ffffffff"), 12, 144, 0),   # 216
    ((1, 1, 1, 1664, 1664, BITMAP, 0, 128, "ffffffff"), 13, 169, 1),   # 247
    ((1, 8, 8, 1024, 1024, CAUSAL | BITMAP, 0, 64, "ffffffff"), 64, 288, 1),
    ((1, 3, 1, 128, 128 * 73, BITMAP, 0, 64, "ffffffff"), 3, 219, 0),  # 237: the last below the line
    ((1, 3, 1, 128, 128 * 74, BITMAP, 0, 64, "ffffffff"), 3, 222, 1),  # 240: the first on it
])
def test_short_lists_are_written_by_the_host(noalloc_plan, shape, items, entries, device):
    # a launch of its own costs a call of few entries more than writing them here
    assert noalloc_plan(*shape) == [items, entries, device]


@pytest.mark.parametrize("shape", DEVICE_LISTS)
def test_lists_that_the_device_writes(noalloc_plan, shape):
    assert noalloc_plan(*shape, "33cc33cc")[2] == 1


@pytest.mark.parametrize("words,entries,device", [("1", 131072, 0), ("0", 0, 0)])
def test_bitmaps_too_large_to_go_beside_their_lists(noalloc_plan, words, entries, device):
    # 1 MiB of bitmap and 1 MiB of lists: written by the host.  No visible tile: no list at all
    assert noalloc_plan(1, 128, 1, 128, 64 * 32 * 1024, BITMAP, 0, 64, words)[1:] == [entries, device]


@pytest.mark.parametrize("keys,device", [(64 * 32 * 960, 1), (64 * 32 * 1021, 1), (64 * 32 * 1022, 0)])
def test_the_largest_bitmaps_that_fit(noalloc_plan, keys, device):
    n = keys // (64 * 32)
    assert noalloc_plan(1, 128, 1, 128, keys, BITMAP, 0, 64, "1") == [128, 128 * n, device]


def test_more_lists_than_fit_are_refused(noalloc_plan):
    assert noalloc_plan(1, 128, 1, 128, 64 * 32 * 1025 * 2, BITMAP, 0, 64, "1") == ["refused"]
    assert noalloc_plan(1, 32, 32, 262144, 262144, CAUSAL, 0, 128, "0") == ["refused"]


@pytest.mark.parametrize("seed", range(40))
def test_layout_of_random_calls(noalloc_plan, seed):
    g = random.Random(seed)
    kv = g.choice((1, 2, 3, 8))
    flags = g.choice((0, CAUSAL, CAUSAL | WINDOW, BITMAP, CAUSAL | BITMAP, CAUSAL | WINDOW | BITMAP))
    out = noalloc_plan(g.choice((1, 2, 5)), kv * g.choice((1, 2, 4)), kv, g.randint(1, 5000), g.randint(1, 6000), flags,
                       g.randint(1, 2000), g.choice((64, 128)), "%x" % g.getrandbits(32))
    assert len(out) == 3 and (flags & BITMAP or out[1] == 0)


def test_a_list_of_another_length_than_planned_is_noticed(tmp_path, repo_root):
    # and nothing is written beside it, and every planned place holds an entry that the attention kernel can walk
    exe = str(tmp_path / "list_writer")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-o", exe, os.path.join(repo_root, "tests", "list_writer.cpp"),
                           os.path.join(repo_root, "paper_2607_09385_b200", "csrc", "steel_planner.cpp")])
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
