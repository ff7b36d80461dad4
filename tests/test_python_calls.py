"""The native functions of the hot calls take their arguments as the ctypes signatures do (no GPU: invalid handles)."""
import ctypes
import os
import subprocess
import sys

import pytest

from paper_2203_05705_b200 import ard

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


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


class Handle(ctypes.c_void_p):
    pass


def test_arguments():
    f = ard._calls().ard_fwd
    ok = [None, None, 0, 4, 4, 4, 1.0, Device(256), 4, 512, 4, Device(768), 4, 1, 0]
    assert f(*ok) == ard.ARD_ERR_INVALID_ARG
    assert f(*[2 ** 32 if i == 3 else a for i, a in enumerate(ok)]) == ard.ARD_ERR_INVALID_ARG   # cut off, as ctypes does
    for i, bad in ((2, "0"), (3, 1.5), (6, "1"), (7, object()), (0, 1.0)):
        with pytest.raises((TypeError, AttributeError, ctypes.ArgumentError)):
            f(*[bad if j == i else a for j, a in enumerate(ok)])


# Of both ways of a call: what the native functions do not take themselves goes through ctypes.
@pytest.mark.parametrize("f", [lambda *a: ard._calls().ard_fwd(*a), lambda *a: ard._through_ctypes("ard_fwd", *a)])
def test_handles_and_memory(f):
    ok = [None, None, 0, 4, 4, 4, 1.0, Device(256), 4, 512, 4, Device(768), 4, 1, 0]
    put = lambda i, x: [x if j == i else a for j, a in enumerate(ok)]  # noqa: E731
    for handle in (Handle(), ctypes.c_void_p(), ctypes.POINTER(ctypes.c_int)(), None, 0):
        for i in (0, 1, 14):
            assert f(*put(i, handle)) == ard.ARD_ERR_INVALID_ARG   # taken, and no context
    assert f(*put(14, ctypes.c_void_p(64))) == f(*put(14, Handle(64))) == ard.ARD_ERR_INVALID_ARG
    for memory in (ctypes.c_void_p(768), Handle(768), ctypes.POINTER(ctypes.c_int)(), 1.5, "x"):
        for i in (7, 9, 11):
            with pytest.raises(AttributeError):   # no tensor: a handle in its place is a slip
                f(*put(i, memory))
    for i, bad in ((2, "0"), (3, 1.5), (6, "1"), (0, 1.0), (0, object()), (14, Device(64))):
        with pytest.raises(ctypes.ArgumentError):
            f(*put(i, bad))


def test_feeding_patterns_are_handles():
    for name in sorted(ard._FED):
        sig = getattr(ard.lib(), name).argtypes
        args = [0.5 if t in (ctypes.c_float, ctypes.c_double) else (None if t is ctypes.c_void_p else 0) for t in sig]
        args[2] = ctypes.c_void_p()
        assert getattr(ard._calls(), name)(*args) == ard._through_ctypes(name, *args) == ard.ARD_ERR_INVALID_ARG
        args[2] = Device(64)
        for f in (getattr(ard._calls(), name), lambda *a: ard._through_ctypes(name, *a)):
            with pytest.raises(ctypes.ArgumentError):
                f(*args)


def test_without_the_native_functions():
    """A library built for another interpreter: the calls go through ctypes, and how to build the functions is said once."""
    code = ("import sys, warnings; sys.modules['paper_2203_05705_b200._calls'] = None\n"
            "from paper_2203_05705_b200 import ard\n"
            "class T:\n    data_ptr = lambda self: 256\n"
            "with warnings.catch_warnings(record=True) as w:\n"
            "    warnings.simplefilter('always')\n"
            "    for _ in range(2):\n"
            "        try: ard.ard_fwd(None, None, 0, 4, 4, 4, 1.0, T(), 4, T(), 4, 768, 4, 1, stream=0)\n"
            "        except ard.ArdError as e: assert e.status == ard.ARD_ERR_INVALID_ARG\n"
            "        else: assert False\n"
            "    assert len(w) == 1 and 'python -m paper_2203_05705_b200.build' in str(w[0].message)\n")
    subprocess.run([sys.executable, "-c", code], cwd=ROOT, check=True)
