"""How steel_attn_run_noalloc lays out a call, from the planner.  CPU only."""
import os
import subprocess

import pytest

CAUSAL, WINDOW, BITMAP = 1, 2, 4


@pytest.fixture(scope="module")
def noalloc_plan(tmp_path_factory, repo_root):
    exe = str(tmp_path_factory.mktemp("noalloc") / "noalloc_plan")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-o", exe, os.path.join(repo_root, "tests", "noalloc_plan.cpp"),
                           os.path.join(repo_root, "paper_2607_09385_b200", "csrc", "steel_planner.cpp")])
    return lambda *args: [int(x) for x in subprocess.check_output([exe, *map(str, args)], text=True).split()]


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


def test_a_list_of_another_length_than_planned_is_noticed(tmp_path, repo_root):
    # and nothing is written beside it, and every planned place holds an entry that the attention kernel can walk
    exe = str(tmp_path / "list_writer")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-o", exe, os.path.join(repo_root, "tests", "list_writer.cpp"),
                           os.path.join(repo_root, "paper_2607_09385_b200", "csrc", "steel_planner.cpp")])
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
