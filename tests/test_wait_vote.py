"""The bounded waits' outcome is per thread; what a block does next must not be.

A copy that lands between the limits of two threads lets one wait run out and the other complete.
If each thread then chose its own way past a barrier, the block's barriers would pair up wrongly or
one part would retire mbarriers that the other still waits on: a hang. That case is not run on a GPU;
the sources are read for it here, and acs_wait_selftest runs the vote itself with half of a block's waits
running out (test_gpu_failure.py).
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2306_13002_gb300", "csrc")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


@pytest.mark.parametrize("name", ["star_fixed.cuh", "rhs_fixed.cuh"])
def test_segments_end_with_the_blocks_verdict(name):
    """The march's loop over segments branches on `ok`: every call of segment() must be followed at once by
    the vote that makes it the same in all threads."""
    code = _code(name)
    calls = [m.end() for m in re.finditer(r"\.segment\([^;]*;", code)]
    assert calls
    for at in calls:
        assert re.match(r"\s*ok\s*=\s*block_ok\(ok\);", code[at:]), code[at:at + 80]
    # before a segment `ok` is decided by what all threads share
    starts = re.findall(r"bool ok = ([^;]*);", code)
    assert starts and all("tid" not in s and "threadIdx" not in s and "wait" not in s for s in starts)


@pytest.mark.parametrize("name", ["star_fixed.cuh", "rhs_fixed.cuh"])
def test_a_failed_wait_ends_a_segment_through_the_blocks_vote(name):
    """Inside a segment the outcome reaches the block through shared memory or the vote on `bad`; no loop or
    return of it depends on `ok` itself."""
    code = _code(name)
    body = code[code.index(" segment("):code.index(".segment(")]
    body = body[:body.index("_fixed_march(")]
    assert "if (!ok) bad = -1;" in body and re.search(r"if \(!ok\) note\[0\] = 0x7f+u?;", body)
    for line in body.splitlines():
        if re.search(r"\bok\b", line):
            assert not re.search(r"\b(for|while|break)\b", line), line
            assert "return" not in line or "landed" in line or line.strip() == "if (!TMA || !ok) return;", line
