"""The wait that the 32 lanes of a softmax warp make together, and the question whether a role has given up, on host
threads: all lanes get the same answer whatever moment each one reads the abort flag at, a wait ends within the bound that
the kernel was given however long a poll takes, and it passes as soon as the phase is complete.  CPU only."""
import os
import subprocess

import pytest


@pytest.fixture(scope="module")
def warp_wait(tmp_path_factory, repo_root):
    exe = str(tmp_path_factory.mktemp("wait") / "warp_wait")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-pthread", "-Wno-unknown-pragmas", "-o", exe,
                           os.path.join(repo_root, "tests", "warp_wait.cpp")])
    return exe


@pytest.mark.parametrize("what", ["abort", "bound", "full", "leave"])
def test_lanes_wait_together(warp_wait, what):
    out = subprocess.run([warp_wait, what], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout
