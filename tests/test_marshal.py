"""The extension module that fills the argument structures of sjq_run: what it accepts, what it rejects and with which
exception.  Columns are stand-ins with a tensor's interface, so that no device is needed: a well-formed call passes all
checks of the library that come before the device."""
import os
import sysconfig
from collections import OrderedDict, UserDict
from types import MappingProxyType

import pytest
import torch

import paper_2607_07632_b200 as sjq
from datagen.workloads import AggExpr, KeyExpr, Pred, Term

B = sjq.sjq
INVALID_ARG, ALIGN, CUDA = 1, 3, 4


class FakeColumn:
    def __init__(self, n=8, dtype=torch.int32, address=0x10000, cuda=True, contiguous=True, dim=1):
        self.n, self.dtype, self.address, self.is_cuda, self.flat, self.ndim = n, dtype, address, cuda, contiguous, dim

    def data_ptr(self):
        return self.address

    def numel(self):
        return self.n

    def is_contiguous(self):
        return self.flat

    def dim(self):
        return self.ndim


def call(fact=None, preds=(), joins=(), key=None, agg=None, mode="SCALAR", num_groups=1, capacity=0, opts=None,
         result=None):
    fact = {"a": FakeColumn(), "b": FakeColumn(dtype=torch.int64)} if fact is None else fact
    agg = agg or AggExpr("COL", Term("FACT", "a"))
    out = FakeColumn(1, torch.int64)
    res = result or B.Result(mode, out, out, out if mode == "HASHED" else None, out if mode == "HASHED" else None,
                             FakeColumn(1), out if mode == "HASHED" else None)
    return B.marshal().run(fact, preds, joins, key, agg, B.MODES[mode], num_groups, capacity, opts, res, 0, lambda: None)


@pytest.mark.skipif(torch.cuda.is_available(), reason="the addresses are made up: only without a device")
def test_well_formed_calls_reach_the_device_check():
    assert call() == CUDA
    assert call(preds=(Pred("a", "IN", values=(1, 2, 3)), Pred("b", "BETWEEN", -2**63, 2**63 - 1))) == CUDA
    assert call(key=KeyExpr((Term("FACT", "b", 0, -3),), offset=5, modulo=7), mode="DENSE", num_groups=7,
                agg=AggExpr("SUB", Term("FACT", "a"), Term("FACT", "b"), want_count=False)) == CUDA
    assert call(opts=B.RunOpts(order=[0], pass_ppm=[5], specialise=True), preds=[Pred("a", "LT", 3)]) == CUDA
    big = {("c%d" % i): FakeColumn() for i in range(64)}
    assert call(big, preds=[Pred("c63", "EQ", 1)], agg=AggExpr("COL", Term("FACT", "c0"))) == CUDA


def test_the_librarys_own_checks_see_what_was_passed():
    assert call({"a": FakeColumn(8), "b": FakeColumn(9)}) == INVALID_ARG  # lengths differ
    assert call({"a": FakeColumn(8, address=0x10004)}) == ALIGN
    assert call(opts=B.RunOpts(order=[0])) == INVALID_ARG  # an order for more filters than there are
    assert call(opts=B.RunOpts(rows_per_lane=8)) == INVALID_ARG  # only with specialise
    assert call(opts=B.RunOpts(dense_slots=3)) == INVALID_ARG
    assert call(opts=B.RunOpts(hot_keys=3)) == INVALID_ARG
    assert call(preds=[Pred("a", "EQ", 1)] * 17) == INVALID_ARG
    assert call(agg=AggExpr("COL", Term("PAYLOAD", 0, 0))) == INVALID_ARG  # no join 0
    assert call(mode="DENSE", num_groups=0, key=KeyExpr((Term("FACT", "a"),))) == INVALID_ARG
    assert call(key=KeyExpr((Term("FACT", "a"),))) == INVALID_ARG  # a key for a scalar


@pytest.mark.parametrize("bad", [FakeColumn(dtype=torch.float32), FakeColumn(cuda=False), FakeColumn(contiguous=False),
                                 FakeColumn(dim=2), torch.zeros(8, dtype=torch.int32)])
def test_columns_of_another_kind_are_value_errors(bad):
    with pytest.raises(ValueError, match="contiguous 1-D int32/int64 CUDA"):
        call({"a": bad})


def test_names_and_counts_that_do_not_fit_raise():
    with pytest.raises(ValueError, match="not a column"):
        call(preds=[Pred("zz", "EQ", 1)])
    with pytest.raises(ValueError, match="not a column"):
        call(agg=AggExpr("COL", Term("FACT", "zz")))
    with pytest.raises(KeyError):
        call(preds=[Pred("a", "LIKE", 1)])
    with pytest.raises(KeyError):
        call(agg=AggExpr("MAX", Term("FACT", "a")))
    with pytest.raises(ValueError, match="key terms"):
        call(key=KeyExpr((Term("FACT", "a"),) * 5), mode="DENSE")
    with pytest.raises(IndexError):
        call(opts=B.RunOpts(pass_ppm=[1] * 25))
    with pytest.raises(TypeError):
        call(preds=[Pred("a", "EQ", "x")])
    with pytest.raises(ValueError):
        sjq.run({"a": torch.zeros(8, dtype=torch.int32)}, agg=AggExpr("COL", Term("FACT", "a")))


def test_measured_fractions_may_be_floats():
    """As through ctypes: int() is applied to them, and to nothing else."""
    few = [Pred("a", "LT", 3)]
    assert call(preds=few, opts=B.RunOpts(pass_ppm=(2.5e5, True), rows_per_lane=8)) == INVALID_ARG  # read, then refused
    assert call(preds=few, opts=B.RunOpts(pass_ppm=torch.tensor([250_000.7]), rows_per_lane=8)) == INVALID_ARG
    for bad in (B.RunOpts(order=(0.0,)), B.RunOpts(block_threads=128.0), B.RunOpts(pass_ppm=(None,))):
        with pytest.raises(TypeError):
            call(preds=few, opts=bad)


@pytest.mark.parametrize("kind", [OrderedDict, UserDict, MappingProxyType])
def test_columns_come_in_any_mapping(kind):
    refused = B.RunOpts(rows_per_lane=8)  # by the library, after everything has been read
    assert call(kind({"a": FakeColumn()}), preds=[Pred("a", "EQ", 1)], opts=refused) == INVALID_ARG
    with pytest.raises(ValueError, match="contiguous 1-D"):
        call(kind({"a": FakeColumn(dim=2)}))
    with pytest.raises((TypeError, AttributeError)):
        call([FakeColumn()])


def test_the_module_is_the_one_built_for_this_interpreter():
    from paper_2607_07632_b200 import build

    assert build.MARSHAL.endswith(sysconfig.get_config_var("EXT_SUFFIX")) and "cpython" in os.path.basename(build.MARSHAL)
    assert os.path.samefile(B.marshal().__file__, build.MARSHAL)
    assert not os.path.exists(os.path.join(os.path.dirname(build.MARSHAL), "_marshal.so"))
