"""A relaxed wait orders nothing after it: only copies into the released buffer may follow.

`warp_wait_relaxed` polls with relaxed semantics in lane 0 alone.  A role that writes the
released buffer with ordinary shared-memory stores needs the acquire that `warp_wait` gives
every lane, else nothing orders its stores after the reads that the release announced.  Read
from the sources: no ordinary shared store between a relaxed wait and the next wait.  (The
reconstructions' A operand lies in tensor memory, whose accesses have fences of their own.)"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2506_01260_gb300", "csrc")
FILES = sorted(f for f in glob.glob(os.path.join(CSRC, "*.cu"))
               if "warp_wait_relaxed(" in open(f).read())


def after_relaxed_waits(text):
    """The code that follows each relaxed wait, up to the next wait or the end of its kernel."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"\bwarp_wait_relaxed\(", text):
        rest = text[m.end():]
        end = re.search(r"\b(?:warp_wait|warp_wait_relaxed|mbar_wait|__syncthreads)\(", rest)
        yield rest[:end.start()] if end else rest


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_only_copies_follow_a_relaxed_wait(path):
    for code in after_relaxed_waits(open(path).read()):
        assert not re.search(r"\b(?:sts128|repack_half)\(", code), code


def test_the_reading_finds_an_ordinary_store():
    code = "if (!warp_wait_relaxed(b, 0, f, e)) break; %s fence_async_smem(); warp_wait(c, 0, f, e);"
    assert list(after_relaxed_waits(code % "sts128(dst, v);"))[0].count("sts128") == 1
    assert "repack_half" not in list(after_relaxed_waits(code % ""))[0]
