"""The rule for how many tiles run at once (csrc/ahpp_groups.h), compiled for
the host: no group without a tile, a configured number kept by batches, and no
more tiles at once in a serving step than the rule allows.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MB = 1 << 20


@pytest.fixture(scope="module")
def groups_of(tmp_path_factory):
    cc = shutil.which("g++")
    if cc is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("groups")
    src = d / "main.cpp"
    src.write_text('#include "ahpp_groups.h"\n#include <cstdio>\n#include <cstdlib>\n'
                   "int main(int, char** v) {\n"
                   "  std::printf(\"%u\", ahpp::groups_of(std::atoi(v[1]), std::atoi(v[2]), std::atoi(v[3]),"
                   " std::strtoull(v[4], nullptr, 10), std::atoi(v[5]) != 0));\n}\n")
    exe = str(d / "groups")
    subprocess.run([cc, "-std=c++17", "-I", os.path.join(ROOT, "paper_2512_11606_gb300", "csrc"), str(src), "-o", exe],
                   check=True)

    def call(configured, n_tiles, table, serving=False, most=64):
        out = subprocess.run([exe, *(str(int(x)) for x in (configured, n_tiles, most, table, serving))],
                             capture_output=True, text=True, check=True)
        return int(out.stdout)

    return call


@pytest.mark.parametrize("serving", [False, True])
@pytest.mark.parametrize("configured", [0, 1, 2, 4, 8])
def test_no_group_without_a_tile(groups_of, configured, serving):
    for n_tiles in (1, 2, 3, 7, 9, 200):
        for table in (MB, 20 * MB, 260 * MB):
            n = groups_of(configured, n_tiles, table, serving)
            assert 1 <= n <= n_tiles
            assert n <= 64 and (not configured or n <= configured)


def test_one_tile_has_all_blocks(groups_of):
    assert groups_of(8, 1, 260 * MB) == 1
    assert groups_of(8, 1, 260 * MB, serving=True) == 1


def test_batches_keep_the_configured_number(groups_of):
    assert groups_of(8, 40, 260 * MB) == 8
    assert groups_of(2, 40, MB) == 2


def test_serving_follows_the_rule_under_the_configured_limit(groups_of):
    # tables beyond L2: one tile after another, whatever is configured
    assert groups_of(8, 8, 260 * MB, serving=True) == 1
    assert groups_of(0, 8, 260 * MB, serving=True) == 1
    # small tables: as many as there are, up to the limit
    assert groups_of(0, 8, MB, serving=True) == 8
    assert groups_of(2, 8, MB, serving=True) == 2
    assert groups_of(1, 8, MB, serving=True) == 1


def test_waves_are_even(groups_of):
    # 20 MB a table: six fit, so 32 tiles go in six waves of at most six
    assert groups_of(0, 32, 20 * MB) == 6
    assert groups_of(0, 7, 20 * MB) == 4
