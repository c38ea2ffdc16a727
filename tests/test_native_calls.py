"""Native marshalling of the binding's calls: it takes an argument exactly as it stands or leaves the call to the checks in
binding.py (None).  On the CPU the tensors stop it at `is_cuda` or the library at its argument checks."""

import os
import subprocess
import sys
import sysconfig

import numpy as np
import pytest
import torch

from paper_2512_23353_b200 import binding as b
from paper_2512_23353_b200 import build

OFF = np.array([0, 2, 5], dtype=np.int64)


@pytest.fixture(autouse=True)
def null_stream():
    """A stream that needs no device."""
    b._bind_calls(b._calls, lambda: 0, lambda device: 0)
    yield
    b._bind_calls(b._calls, b._current_device, b._raw_stream)


def weight_grad(**kw):
    a = dict(X=torch.zeros(5, 8), dY=torch.zeros(5, 6), c=torch.zeros(2), off=OFF, dW=torch.zeros(6, 8),
             ws=torch.zeros(0, dtype=torch.uint8), info=torch.zeros(1, dtype=torch.int32), path=b.PATH_GRAM, beta=0.0)
    a.update(kw)
    return b._calls.weight_grad(*a.values())


def test_call_reaches_the_library():
    assert weight_grad(beta=0.5) == b.ERR_INVALID_ARG  # only 0 and 1
    with pytest.raises(b.IsopoError):
        b.isopo_weight_grad(torch.zeros(5, 8), torch.zeros(5, 6), torch.zeros(2), OFF, torch.zeros(6, 8),
                            torch.zeros(0, dtype=torch.uint8), torch.zeros(1, dtype=torch.int32), b.PATH_GRAM, 0.5)


@pytest.mark.parametrize("kw", [dict(off=[0, 2, 5]), dict(off=OFF.astype(np.int32)), dict(off=np.arange(6)[::2]),
                                dict(off=OFF.reshape(1, 3)), dict(off=OFF[:1]), dict(off=OFF.astype(np.float64)), dict(off=None),
                                dict(X=torch.zeros(5, 8).half()), dict(X=torch.zeros(5)), dict(c=torch.zeros(3)),
                                dict(c=torch.zeros(2).double()), dict(dW=torch.zeros(8, 6)), dict(dW=torch.zeros(8, 6).T),
                                dict(dW=torch.zeros(6, 8).bfloat16()), dict(ws=None), dict(info=3), dict(path="auto"),
                                dict(path=-1), dict(beta="x")])
def test_unusual_arguments_are_left_to_python(kw):
    assert weight_grad(**kw) is None


def test_wrong_number_of_arguments_and_other_calls():
    K, A, i = torch.zeros(4), torch.zeros(2), torch.zeros(1, dtype=torch.int32)
    assert b._calls.weight_grad() is None and b._calls.layer_gram(K) is None
    assert b._calls.layer_gram(torch.zeros(5, 8), torch.zeros(5, 6), OFF, K, torch.zeros(0, dtype=torch.uint8), i, 1) is None
    assert b._calls.transform(torch.zeros(5), A, b.VAR_NORMALISED, 0.0, A, i) is None
    assert b._calls.transform(K, A, b.VAR_NORMALISED, 0.0, torch.zeros(3), i) is None
    assert b._calls.transform(K, A, b.VAR_NORMALISED, -1.0, A, i) == b.ERR_INVALID_ARG
    assert b._calls.transform_rel(K, A, b.VAR_NORMALISED, 0.0, torch.zeros(3), A, i) is None
    assert b._calls.reg_ema(K, 0.9, torch.zeros(4)) is None
    assert b._calls.sampled(torch.zeros(5, 8), torch.zeros(5, 6), OFF, [0, 1], A, 0.0, A, A, i, None) is None


def test_trailing_dimensions_of_one_are_taken(monkeypatch):
    """[T, d, 1] holds the same rows as [T, d]: python reads the first two sizes only, and the library sees the call."""
    monkeypatch.setattr(b, "_stream", lambda: 0)
    a = [torch.zeros(5, 8, 1), torch.zeros(5, 6, 1), torch.zeros(2), OFF, torch.zeros(6, 8), torch.zeros(0, dtype=torch.uint8),
         torch.zeros(1, dtype=torch.int32), b.PATH_GRAM, 0.5]
    assert b._calls.weight_grad(*a) is None
    with pytest.raises(b.IsopoError, match="ISOPO_ERR_INVALID_ARG"):  # the beta, not the shapes
        b.isopo_weight_grad(*a)


def test_without_the_native_module_calls_go_through_ctypes():
    """A machine without Python's headers, or another interpreter than the one the module was built for."""
    code = """if True:
        import sys
        sys.modules["paper_2512_23353_b200._calls"] = None  # as if there were no such file
        import numpy as np, torch
        from paper_2512_23353_b200 import binding as b
        assert b._calls is b._NoCalls
        b._stream = lambda: 0
        K, A, i, off = torch.zeros(4), torch.zeros(2), torch.zeros(1, dtype=torch.int32), np.array([0, 2, 5])
        ws = torch.zeros(0, dtype=torch.uint8)
        for call in (lambda: b.isopo_weight_grad(torch.zeros(5, 8), torch.zeros(5, 6), A, off, torch.zeros(6, 8), ws, i, 1, 0.5),
                     lambda: b.isopo_transform_advantages(K, A, b.VAR_NORMALISED, -1.0, A, i),
                     lambda: b.isopo_transform_advantages_rel(K, A, b.VAR_NORMALISED, -1.0, torch.zeros(4), A, i)):
            try:
                call()
            except b.IsopoError as e:
                assert e.status == b.ERR_INVALID_ARG
            else:
                raise SystemExit("the library was not reached")
        print("through ctypes")
    """
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True)
    assert r.returncode == 0 and "through ctypes" in r.stdout, r.stderr


def test_module_is_named_for_its_interpreter_and_rebuilt_by_itself():
    assert build.CALLS_PATH.endswith("_calls" + sysconfig.get_config_var("EXT_SUFFIX")) and os.path.exists(build.CALLS_PATH)
    assert b._calls.__file__ == build.CALLS_PATH
    assert not any(p.endswith("py_calls.c") for p in build._deps())  # an edit there leaves the CUDA objects alone
