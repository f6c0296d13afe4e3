"""Host data is on the device before a launch can read it.

The library launches on non-blocking streams, which do not wait for the default
stream; a cudaMemcpy from pageable memory may return before its copy has
arrived, and cudaMemset always may.  So the sources (beside the self-test, whose
kernels run on the default stream itself) move data to the device by upload(),
which waits on a stream of its own, or in order on the stream of the launch.
"""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2512_11606_gb300", "csrc")


def calls(name):
    """(file, arguments) of every call of `name` in the library's sources."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*"))):
        src = re.sub(r"//[^\n]*", "", open(path, encoding="utf-8").read())
        for m in re.finditer(r"\b%s\(" % name, src):
            depth, i = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(src[i], 0)
                i += 1
            yield os.path.basename(path), src[m.end():i - 1]


def test_no_unordered_upload():
    up = [c for c in calls("cudaMemcpy") if "HostToDevice" in c[1]]
    assert not up, up
    sets = [c for c in calls("cudaMemset") if c[0] != "ahpp_selftest.cu"]
    assert not sets, sets


def test_asynchronous_copies_name_a_stream():
    for name, n_args in (("cudaMemcpyAsync", 5), ("cudaMemsetAsync", 4), ("cudaMemset2DAsync", 6)):
        found = list(calls(name))
        assert found, name
        for path, args in found:
            top, depth = 1, 0
            for ch in args:
                depth += {"(": 1, ")": -1, "[": 1, "]": -1}.get(ch, 0)
                top += ch == "," and depth == 0
            assert top == n_args, (path, args)
