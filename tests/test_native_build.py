"""The extension module against torch headers without the DLPack exchange table, or none at all: it builds, and takes
addresses and streams through the Python attributes (every call here is refused before anything is launched)."""
import os
import shutil
import subprocess
import sys

import pytest

from paper_2602_15563_b200 import build as kb

CALLS = r"""
import sys
from paper_2602_15563_b200 import kmq
kmq._NATIVE_PATH = sys.argv[1]


class Tensor:                      # named like torch's
    def data_ptr(self):
        return 0x1000


class Stream:
    cuda_stream = 0


t, s = Tensor(), Stream()
assert kmq.kmq_pack(t, 4, 32, 3, t, stream=s, check=False) == kmq.KMQ_ERR_BITS
assert kmq.kmq_pack(None, 4, 32, 1, t, stream=s, check=False) == kmq.KMQ_ERR_NULL
assert kmq.kmq_linear(t, t, t, t, 4, 32, 1, 1, layout=9, stream=0, check=False) == kmq.KMQ_ERR_LAYOUT
"""


@pytest.mark.parametrize("headers", ("none", "dlpack_1_0"))
def test_builds_without_the_exchange_table(headers, tmp_path):
    kb.build()
    include = []
    if headers == "dlpack_1_0":
        (tmp_path / "ATen").mkdir()
        (tmp_path / "ATen" / "dlpack.h").write_text("#define DLPACK_MAJOR_VERSION 1\n#define DLPACK_MINOR_VERSION 0\n")
        include = ["-I", str(tmp_path)]
    out = tmp_path / os.path.basename(kb.NATIVE_PATH)
    res = subprocess.run(kb.native_command(str(out), include), capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    shutil.copy(kb.LIB_PATH, tmp_path)
    res = subprocess.run([sys.executable, "-c", CALLS, str(out)], cwd=kb.ROOT, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
