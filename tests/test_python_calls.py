"""The native functions of the hot calls take their arguments as the ctypes signatures do (no GPU: invalid handles)."""
import ctypes

import pytest

from paper_2203_05705_b200 import ard


class Device:
    def __init__(self, p):
        self.p = p

    def data_ptr(self):
        return self.p


def test_every_function_has_the_signature_of_its_export():
    native, lib = ard._calls(), ard.lib()
    names = [n for n in dir(native) if n.startswith("ard_")]
    assert len(names) > 30 and set(names) <= set(ard.EXPORTS)
    for name in names:
        sig = getattr(lib, name).argtypes
        args = [0.5 if t in (ctypes.c_float, ctypes.c_double) else (None if t is ctypes.c_void_p else 0) for t in sig]
        assert getattr(native, name)(*args) == getattr(lib, name)(*args) != ard.ARD_OK, name   # no context
        with pytest.raises(TypeError):
            getattr(native, name)(*args[:-1])
        with pytest.raises(TypeError):
            getattr(native, name)(*args, 0)


def test_arguments():
    f = ard._calls().ard_fwd
    ok = [None, None, 0, 4, 4, 4, 1.0, Device(256), 4, 512, 4, ctypes.c_void_p(768), 4, 1, 0]
    assert f(*ok) == ard.ARD_ERR_INVALID_ARG
    assert f(*[2 ** 32 if i == 3 else a for i, a in enumerate(ok)]) == ard.ARD_ERR_INVALID_ARG   # cut off, as ctypes does
    for i, bad in ((2, "0"), (3, 1.5), (6, "1"), (7, object()), (0, 1.0)):
        with pytest.raises((TypeError, AttributeError)):
            f(*[bad if j == i else a for j, a in enumerate(ok)])
