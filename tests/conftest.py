import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (B200)")


@pytest.fixture(scope="session")
def repo_root():
    return ROOT


@pytest.fixture(scope="session")
def plan_dump(tmp_path_factory):
    """Runs tests/plan_dump.cpp: the lines of the plan that steel_attn_create builds for a problem."""
    exe = str(tmp_path_factory.mktemp("plan") / "plan_dump")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-o", exe, os.path.join(ROOT, "tests", "plan_dump.cpp"),
                           os.path.join(ROOT, "paper_2607_09385_b200", "csrc", "steel_planner.cpp")])

    def dump(ctas, batch, heads_q, heads_kv, seq_q, seq_kv, flags, window, block=128, words=()):
        args = (ctas, batch, heads_q, heads_kv, seq_q, seq_kv, flags, window, block)
        return subprocess.check_output([exe] + [str(x) for x in args] + ["%x" % x for x in words], text=True).split("\n")

    return dump
