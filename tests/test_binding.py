"""The extension module's argument handling: positional and keyword arguments, defaults, errors (every call here is
refused by the library's own validation before anything is launched)."""
import pytest

from paper_2602_15563_b200 import build as kb
from paper_2602_15563_b200 import kmq

A = 0x1000   # non-NULL, 16-byte aligned, never dereferenced


class FakeTensor:
    def __init__(self, address, numel=0):
        self.address, self.n = address, numel

    def data_ptr(self):
        return self.address

    def numel(self):
        return self.n

    def element_size(self):
        return 1


class FakeStream:
    cuda_stream = 0


@pytest.fixture(scope="module", autouse=True)
def built():
    kb.build()


@pytest.mark.parametrize("first", [A, FakeTensor(A), None])
def test_addresses_objects_and_none(first):
    want = kmq.KMQ_ERR_BITS if first is not None else kmq.KMQ_ERR_NULL
    assert kmq.kmq_pack(first, 4, 32, 3, A, stream=FakeStream(), check=False) == want


def test_keywords_reach_their_place():
    kw = dict(packed=A, codebooks=A, x=A, y=A, N=4, K=32, bits=1, M=1, layout=9, stream=0, check=False)
    assert kmq.kmq_linear(**kw) == kmq.KMQ_ERR_LAYOUT
    assert kmq.kmq_linear(A, A, A, A, 4, 32, 1, 1, None, None, 9, 0, False) == kmq.KMQ_ERR_LAYOUT
    assert kmq.kmq_linear(**{**kw, "layout": 0, "y": A + 4}) == kmq.KMQ_ERR_ALIGN
    assert kmq.kmq_block_linear(A, A, A, A, A, 4, 64, 1, 1, scale_order=2, stream=0, check=False) == kmq.KMQ_ERR_LAYOUT


@pytest.mark.parametrize("args,kw", [
    ((A, 4, 32, 1), {}),                                   # packed is missing
    ((A, 4, 32, 1, A), {"packed": A}),                     # given twice
    ((A, 4, 32, 1, A), {"no_such": 1}),
    ((A, 4, 32, 1, A, 0, 0, False, 1), {}),                # one too many
    ((A, 4.0, 32, 1, A), {"stream": 0}),                   # not an integer
    (("text", 4, 32, 1, A), {"stream": 0}),                # no data_ptr()
])
def test_bad_arguments_raise(args, kw):
    with pytest.raises((TypeError, AttributeError)):
        kmq.kmq_pack(*args, **kw)


def test_failed_status_raises_unless_told_otherwise():
    with pytest.raises(kmq.KmqError) as e:
        kmq.kmq_dequant_to_bf16(A, A, A, 4, 12, 4, stream=0)
    assert e.value.status == kmq.KMQ_ERR_SHAPE and "kmq_dequant_to_bf16" in str(e.value)
    with pytest.raises(AttributeError):
        kmq.kmq_no_such_call
