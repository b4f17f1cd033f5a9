"""The step lists that steel_attn_run_noalloc writes on the device, against the planner's: the same items in the same places
and the same entries, for random bitmaps, both block sizes, every mask combination, ragged and unequal lengths.  CPU only."""
import os
import subprocess

import pytest


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_device_lists_equal_the_planners(tmp_path, repo_root, seed):
    exe = str(tmp_path / "list_entries")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-o", exe, os.path.join(repo_root, "tests", "list_entries.cpp"),
                           os.path.join(repo_root, "paper_2607_09385_b200", "csrc", "steel_planner.cpp")])
    out = subprocess.run([exe, "1500", str(seed)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    assert int(out.stdout) > 500  # plans of single tiles, which the device's lists are for
