"""Kernels that start before the previous kernel on the stream has finished (programmatic dependent launch) read its output
after griddepcontrol.wait.  A const __restrict__ pointer or __ldg would tell the compiler that this memory does not change
while the kernel runs, which would let it move the load ahead of the wait: the sources use the volatile loads of
kmq_common.cuh instead.  No run of the result can show that reliably, so the sources are checked."""
import glob
import os
import re

import pytest

from paper_2602_15563_b200 import build as kb

# parameters that hold what an earlier kernel may have written: activations, partial sums, the source of a copy
WRITTEN = r"(?:x|xrow|scratch|src)"
SOURCES = [p for p in sorted(glob.glob(os.path.join(kb.CSRC, "*.cu*"))) if "griddepcontrol.wait" in open(p).read()]


def test_there_are_such_kernels():
    assert len(SOURCES) >= 7


@pytest.mark.parametrize("path", SOURCES, ids=[os.path.basename(p) for p in SOURCES])
def test_no_read_only_promise_about_written_memory(path):
    text = re.sub(r"//[^\n]*", "", open(path).read())
    assert not re.findall(rf"const\s+\w+\s*\*\s*__restrict__\s+{WRITTEN}\b", text)
    assert not re.findall(rf"__ldg\((?:[^();]|\([^()]*\))*(?<!\.)\b(?:x|xrow|px_src|src|scratch)\b", text)
