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


def functions(text):
    """(name, parameters, body) of the functions at the outermost level of a source without comments."""
    for m in re.finditer(r"\b(\w+)\(((?:[^()]|\([^()]*\))*)\)\s*\{", text):
        if m.group(1) in ("if", "for", "while", "switch"):
            continue
        depth, at = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[at], 0)
            at += 1
        yield m.group(1), m.group(2), text[m.end():at]


# The fit of the block format's codebook starts beside the kernel that draws its sample; its rows come as W, w.  The block
# assignment starts beside the kernels that write its scales and codebook.
@pytest.mark.parametrize("source,function,names", [
    ("kmq_fit.cu", "fit_rows_kernel", ("W", "w")), ("kmq_fit.cu", "fit_by_buckets", ("w",)),
    ("kmq_fit.cu", "fit_by_sorting", ("w",)), ("kmq_quantize.cu", "block_assign_kernel", ("scales", "codebook"))])
def test_inputs_of_a_dependent_kernel_are_read_behind_its_wait(source, function, names):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(kb.CSRC, source)).read())
    (_, parameters, body), = [f for f in functions(text) if f[0] == function]
    for name in names:
        assert not re.search(rf"__restrict__\s+{name}\b", parameters + body)
        assert not re.search(rf"\b{name}\s*\[", body)                 # no plain load ...
        assert not re.search(rf"__ldg\((?:[^();]|\([^()]*\))*\b{name}\b", body)
