"""What the binding refuses and accepts: the per-batch calls convert their arguments in native code, with the outcomes of the
ctypes conversions.  No GPU needed: an argument that does not fit raises before the call looks for one."""
import ctypes as C

import numpy as np
import pytest
import torch

import paper_2002_00655_b200 as ps
from paper_2002_00655_b200 import binding

N = 4
IDX, VAL, F64 = torch.zeros(N, dtype=torch.int32), torch.zeros(N), torch.zeros(1, dtype=torch.float64)
GOOD = dict(h=None, i=IDX, j=IDX, v=VAL, base=7, lr=0.1, lam=0.0, loss=None, h_loss=F64)


class TensorLike:
    """Any object with a tensor's attributes was taken by the conversions in Python."""
    is_cuda, dtype = False, torch.int32

    def is_contiguous(self):
        return True

    def data_ptr(self):
        return IDX.data_ptr()

    def numel(self):
        return N


def call(**changed):
    binding._load_native()
    ps.ps_step_mf_host(*{**GOOD, **changed}.values())


@pytest.mark.parametrize("what,value,error", [
    ("i", IDX.long(), AssertionError), ("i", VAL, AssertionError), ("j", torch.zeros(2 * N, dtype=torch.int32)[::2], AssertionError),
    ("v", VAL.double(), AssertionError), ("loss", F64, AssertionError), ("h_loss", VAL, AssertionError),
    ("i", None, AttributeError), ("i", [1, 2], AttributeError), ("j", np.zeros(N, np.int32), AttributeError),
    ("base", 7.0, TypeError), ("base", None, TypeError), ("base", "7", TypeError), ("base", C.c_float(7), TypeError),
    ("lr", "0.1", TypeError), ("lr", None, TypeError), ("lr", C.c_uint64(1), TypeError),
    ("h", np.int64(3), TypeError), ("h", 1.5, TypeError), ("h", C.c_uint64(3), TypeError), ("h", torch.tensor(3), TypeError)])
def test_refused(what, value, error):
    with pytest.raises(error):
        call(**{what: value})


@pytest.mark.parametrize("what,value", [
    ("i", torch.zeros(N, dtype=torch.uint32)), ("i", IDX.reshape(2, 2)), ("j", None), ("i", TensorLike()),
    ("base", np.int64(7)), ("base", torch.tensor(7)), ("base", C.c_uint64(7)), ("base", True), ("base", -1),
    ("lr", 1), ("lr", np.float32(0.1)), ("lr", torch.tensor(0.1)), ("lr", C.c_float(0.1)), ("lr", -1.0), ("lr", float("nan")),
    ("h", 0), ("h", C.c_void_p()), ("h", C.POINTER(C.c_int)())])
def test_accepted(what, value):
    """The call gets past its arguments: to the library, which refuses the null handle, or, without a GPU, to the stream."""
    with pytest.raises(Exception) as e:
        call(**{what: value})
    assert not isinstance(e.value, (TypeError, AssertionError, AttributeError)), e.value
    if isinstance(e.value, ps.PSError):
        assert e.value.code == ps.PS_ERR_INVALID_ARG


@pytest.mark.gpu
def test_device_arguments_and_results():
    g = ps.Store(100, 8, max_batch_keys=64)
    keys, rows = torch.arange(10, device="cuda"), torch.ones((10, 8), device="cuda")
    for bad in (keys.cpu(), keys.int(), keys.repeat(2)[::2], keys.float()):
        for f in (g.pull, lambda k: g.push(k, rows), lambda k: g.localize(0, k), lambda k: g.set_rows(k, rows)):
            with pytest.raises(AssertionError):
                f(bad)
    for bad in (rows.cpu(), rows.double(), rows.half()):
        with pytest.raises(AssertionError):
            g.push(keys, bad)
    out = g.pull(keys.reshape(2, 5))
    assert out.shape == (10, 8) and out.dtype == torch.float32 and out.is_cuda
    g.h, h = None, g.h
    with pytest.raises(ps.PSError) as e:
        g.pull(keys)
    assert e.value.code == ps.PS_ERR_INVALID_ARG
    g.h = h
    g.push(keys, rows)
    assert g.sync() == ps.PS_OK and (g.pull(keys) == 1).all()
    m = ps.KeyMap(50, 64)
    dense = m.insert(keys * 11)
    assert dense.dtype == torch.int64 and (dense == torch.arange(10, device="cuda")).all() and (m.lookup(keys * 11) == dense).all()
    with pytest.raises(AssertionError):
        m.insert(keys.int())


def test_the_native_part_is_built_again_for_another_torch():
    from paper_2002_00655_b200 import build
    assert build._built_for(build.NATIVE, torch.__version__) and not build._built_for(build.NATIVE, torch.__version__ + ".post1")
