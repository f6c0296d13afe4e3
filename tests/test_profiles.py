"""Captures under profiles/ name the sources they were taken of: those that the
bench's traffic figures rest on are the same, and commands run committed files.
"""
import os
import re
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
sys.argv = sys.argv[:1]
import bench  # noqa: E402


def text(name):
    return open(os.path.join(ROOT, "profiles", name), encoding="utf-8").read()


@pytest.mark.parametrize("kernel,name", [("k_tiles", "k_tiles_medium_tile32.md"), ("k_query1", "k_query1_medium.md")])
def test_the_bench_rests_on_the_capture(kernel, name):
    digests = dict(re.findall(r"(ahpp_\w+\.cuh?) ([0-9a-f]{16})", text(name)))
    assert digests == bench.NCU_TRAFFIC[kernel]["sources"]


def test_commands_run_committed_files():
    for name in os.listdir(os.path.join(ROOT, "profiles")):
        for script in re.findall(r"python3? ([\w/.]+\.py)", text(name)):
            assert os.path.exists(os.path.join(ROOT, script)), (name, script)
