"""The words with which a pass clears its result are looked at before a kernel writes through them: their length, their
device and their layout.  Tensors are stand-ins, so that no device is needed: what is accepted reaches the library's check
for one."""
from types import SimpleNamespace

import pytest
import torch

import paper_2607_07632_b200 as sjq
from test_marshal import ALIGN, CUDA, FakeColumn, call

B = sjq.sjq
BUFFER_SMALL = 5
no_device = pytest.mark.skipif(torch.cuda.is_available(), reason="the addresses are made up: only without a device")


class Words(FakeColumn):
    def __init__(self, n=8, width=8, device=0, **kw):
        super().__init__(n, **kw)
        self.width, self.at, self.device = width, device, torch.device("cpu" if device < 0 else "cuda:%d" % device)

    @property
    def nbytes(self):
        return self.n * self.width

    def get_device(self):
        return self.at


def result(**kw):
    out = FakeColumn(1, torch.int64)
    return SimpleNamespace(mode="SCALAR", sums=out, counts=out, keys=None, n_groups=None, status_dev=FakeColumn(1),
                           workspace=None, info=B.RunInfo(), **kw)


@no_device
@pytest.mark.parametrize("words", [Words(8), Words(9), Words(16, 4), Words(64, 1), None])
def test_words_of_the_right_length_are_taken(words):
    assert call(result=result(sync=words)) == CUDA
    assert B._sync_pointer(result(sync=words), torch.device("cuda:0")) == (words.address if words else None)


@pytest.mark.parametrize("words", [Words(7), Words(15, 4), Words(63, 1), Words(1), Words(0)])
def test_short_words_are_refused(words):
    assert call(result=result(sync=words)) == BUFFER_SMALL
    with pytest.raises(B.SjqError) as e:
        B._sync_pointer(result(sync=words), torch.device("cuda:0"))
    assert e.value.status == BUFFER_SMALL


@pytest.mark.parametrize("words", [Words(device=-1), Words(device=1), Words(contiguous=False)])
def test_words_elsewhere_are_refused(words):
    with pytest.raises(ValueError, match="sync words"):
        call(result=result(sync=words))
    with pytest.raises(ValueError, match="sync words"):
        B._sync_pointer(result(sync=words), torch.device("cuda:0"))


def test_misaligned_words_are_refused_by_the_library():
    assert call(result=result(sync=Words(address=0x10004))) == ALIGN


@no_device
def test_a_result_without_the_attribute_brings_none():
    assert call(result=result()) == CUDA
    assert B._sync_pointer(result(), torch.device("cuda:0")) is None
