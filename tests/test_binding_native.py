"""The native call marshalling against the plain ctypes call: same status for the same arguments, and Python errors for
arguments that are not what the call takes.  Only calls that the library refuses before it looks for a device."""
import ctypes
import importlib.machinery
import os
import sysconfig

import pytest
import torch

from paper_2309_03824_b200 import binding as b
from paper_2309_03824_b200 import build

T = torch.zeros(64, dtype=torch.bfloat16)
ODD = torch.zeros(65, dtype=torch.uint8)[1:]           # not aligned to a bf16 element
WS = torch.zeros(1 << 16, dtype=torch.uint8)


def _ctypes_fwd(d, X, V, U, bias, Y, Z, freeze, ws):
    p = lambda t: None if t is None else ctypes.c_void_p(t.data_ptr())
    return b._lib.lrd_linear_fwd(ctypes.byref(d), p(X), p(V), p(U), p(bias), p(Y), p(Z), freeze, p(ws), 0 if ws is None else ws.numel(), None)


@pytest.mark.parametrize("args", [(T, T, T, None, T, T, 7, WS), (None, T, T, None, T, T, 0, WS), (T, T, T, T, T, None, 0, WS), (T, ODD, T, T, T, T, 0, WS),
                                  (T, T, T, T, T, T, 0, None), (T, T, T, T, T, T, 0, WS[:16])])
def test_refused_calls_return_the_library_status(args):
    d = b.linear_desc(256, 64, 64, 16, b.LRD_BF16)
    st = b.lrd_linear_fwd(d, *args, stream=0, check=False)
    assert st == _ctypes_fwd(d, *args) and st != b.LRD_OK
    with pytest.raises(b.LrdError):
        b.lrd_linear_fwd(d, *args, stream=0)


def test_arguments_of_the_wrong_kind_raise():
    d, t = b.linear_desc(256, 64, 64, 16, b.LRD_BF16), b.tucker2_desc(1, 4, 4, 8, 8, 4, 4, b.LRD_BF16)
    with pytest.raises(TypeError):
        b.lrd_linear_fwd(t, T, T, T, None, T, T, 0, WS, stream=0)
    for not_a_descriptor in (bytes(d), memoryview(bytes(d)), bytearray(bytes(d))):       # the right size is not enough
        with pytest.raises(TypeError):
            b.lrd_linear_fwd(not_a_descriptor, T, T, T, None, T, T, 0, WS, stream=0)
        with pytest.raises(TypeError):
            b.lrd_linear_group_fwd([not_a_descriptor], [T], [T], [T], None, [T], [T], 0, [WS], stream=0)
    with pytest.raises(AttributeError):
        b.lrd_linear_fwd(d, 5, T, T, None, T, T, 0, WS, stream=0)
    with pytest.raises(ValueError):
        b.lrd_linear_group_fwd([d, d], [T], [T, T], [T, T], None, [T, T], [T, T], 0, [WS, WS], stream=0)


def test_groups_take_lists_and_none():
    d = b.linear_desc(256, 64, 64, 16, b.LRD_BF16)
    assert b.lrd_linear_group_fwd([], [], [], [], None, [], None, 0, [], stream=0, check=False) == b.LRD_OK
    assert b.lrd_linear_group_bwd([d], [T], None, [T], [T], None, [T], None, [T], None, 1, [WS], stream=0, check=False) == b.LRD_ERR_INVALID_ARG
    n = 9                                              # one more than a group may have
    assert b.lrd_linear_group_fwd([d] * n, [T] * n, [T] * n, [T] * n, None, [T] * n, None, 1, [WS] * n, stream=0, check=False) == b.LRD_ERR_INVALID_ARG


def test_extension_is_named_for_its_interpreter():
    """Only the interpreter that it was built for imports it: the plain ".so" that every CPython takes is not its name."""
    suffix = sysconfig.get_config_var("EXT_SUFFIX")
    assert suffix in importlib.machinery.EXTENSION_SUFFIXES and suffix != ".so"
    assert os.path.basename(build.NATIVE) == "_native" + suffix
    assert os.path.samefile(b._native.__file__, build.NATIVE)
