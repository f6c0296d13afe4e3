"""No kernel block ends while its asynchronous copies are in flight: every ring
that issues cp.async waits for all of them where its scope ends, which is every
way out of the kernels, also when a bounded wait gives up.
"""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2512_11606_gb300", "csrc")


def test_rings_wait_where_they_end():
    found = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        src = open(path, encoding="utf-8").read()
        if "cp.async.cg" not in src:
            continue
        for m in re.finditer(r"struct (\w*Ring) \{(.*?)\n\};", src, re.S):
            body = m.group(2)
            assert "cp.async.cg" in body, m.group(1)
            assert re.search(r"~%s\(\) \{[^}]*cp\.async\.wait_all" % m.group(1), body), m.group(1)
            src = src.replace(m.group(0), "")
            found += 1
        assert "cp.async.cg" not in src, path        # no copies outside a ring
    assert found == 2
