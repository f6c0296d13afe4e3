"""The two sides of the grid barrier are accesses of one width.

PTX orders what comes before a release behind an acquire that reads it only
where both are accesses of the same size to the same place; a vector load is as
many loads of its element's size.
"""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
INTERNAL = os.path.join(ROOT, "paper_2512_11606_gb300", "csrc", "ahpp_internal.cuh")


def test_release_and_acquire_have_the_same_width():
    src = open(INTERNAL, encoding="utf-8").read()
    released = re.findall(r"red\.release\.gpu\.global\.add\.[ub](\d+)", src)
    acquired = re.findall(r"ld\.acquire\.gpu\.global(?:\.v\d)?\.[ub](\d+)", src)
    assert released and acquired
    assert set(released) == set(acquired) == {"32"}
    # the words that are loaded together are the arrivals and, next to them, the error flag
    words = re.search(r"struct alignas\(16\) GridBarrier \{(.*?)\};", src, re.S).group(1)
    assert re.findall(r"unsigned int (\w+)", words)[:2] == ["count", "err"]
