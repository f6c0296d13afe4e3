"""Host threads of the library (csrc/ahpp_threads.h), compiled for the host: an
exception in one of them ends in the caller, after all have ended, and threads
that cannot be started leave their work to the caller.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "ahpp_threads.h"
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <sys/resource.h>
int main(int, char** v) {
  const unsigned n = std::atoi(v[1]), bad = std::atoi(v[2]);
  if (std::strcmp(v[3], "small") == 0) {      // no room for the stacks of many threads
    const rlimit r{64u << 20, 64u << 20};
    if (setrlimit(RLIMIT_AS, &r)) return 3;
  }
  std::atomic<unsigned> done{0};
  int caught = 0;
  try {
    ahpp::run_threads(n, [&](unsigned t) {
      if (t == bad) throw std::bad_alloc();
      ++done;
    });
  } catch (const std::bad_alloc&) {
    caught = 1;
  }
  std::printf("%u %d", done.load(), caught);
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    cc = shutil.which("g++")
    if cc is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("threads")
    (d / "main.cpp").write_text(SRC)
    exe = str(d / "threads")
    subprocess.run([cc, "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "paper_2512_11606_gb300", "csrc"),
                    str(d / "main.cpp"), "-o", exe], check=True)

    def call(n, bad, room="all"):
        r = subprocess.run([exe, str(n), str(bad), room], capture_output=True, text=True)
        assert r.returncode == 0, r
        done, caught = r.stdout.split()
        return int(done), bool(int(caught))

    return call


@pytest.mark.parametrize("n", [1, 2, 32])
def test_every_part_runs(run, n):
    assert run(n, n) == (n, False)


@pytest.mark.parametrize("n,bad", [(1, 0), (2, 0), (2, 1), (32, 7), (32, 31)])
def test_an_exception_reaches_the_caller(run, n, bad):
    assert run(n, bad) == (n - 1, True)


def test_threads_that_cannot_start(run):
    assert run(200, 200, "small") == (200, False)
    assert run(200, 150, "small") == (199, True)


def test_the_library_starts_its_threads_there():
    csrc = os.path.join(ROOT, "paper_2512_11606_gb300", "csrc")
    for f in ("ahpp_graph.cu", "ahpp_q1layout.cu", "ahpp_tilelayout.cu", "ahpp_cluster.cu"):
        src = open(os.path.join(csrc, f), encoding="utf-8").read()
        assert "std::thread " not in src and "std::vector<std::thread>" not in src, f
