"""The natively marshalled calls hand the library the same arguments as their wrappers, and leave to them what they do not take."""
import ctypes as C
import inspect

import numpy as np
import pytest
import torch

import paper_2503_02508_b200 as q
from paper_2503_02508_b200 import _marshal, binding

X, Y, Z = torch.zeros(8), torch.zeros(16), torch.zeros(4, dtype=torch.int8)
QP = q.qparams(0.25, 3, -100, 90)
EPI = q.epilogue(w_scale=X, bias=Y, gate=Z, ld_gate=1 << 40, tokens_per_sample=7, out_qp=QP)
BIG = (1 << 62) + 5
CALLS = {
    "qdit_quantize_act": [(77, X, 1, BIG, 16, -3, 2, None, Y, Z, 24), (None, X, 0, 1, 2, 3, 0, QP, None, 1 << 63, 4)],
    "qdit_w8a8_linear": [(77, X, Y, BIG, 2, 3, QP, None, 0xFFFFFFFF, EPI, Z, -1), (77, X, Y, 1, 2, 3, QP, X, 1, None, None, 5)],
    "qdit_w4a8_linear": [(77, X, Y, 1, 2, 3, QP, None, 7, EPI, Z, 9, X), (77, X, Y, 1, 2, 3, QP, X, 1, None, Z, 5), (77, X, Y, 1, 2, 3, QP, X, 1, None, Z, 5, None)],
    "qdit_attention": [(77, 1, 2, 3, 4, 5, 6, 7, -8, 0.125, X, 2), (77, X, Y, Z, BIG, 5, 6, 7, 8, 0.1, X, 2, QP), (77, X, Y, Z, 4, 5, 6, 7, 8, 1e300, X, 2, None, Y)],
    "qdit_adaln_modulate": [(77, X, BIG, 2, 3, 1e-6, X, Y, 5, Z, 2), (77, X, 1, 2, 3, 0.5, X, Y, 5, Z, 2, QP, X)],
}


@pytest.fixture
def recorded(monkeypatch):
    """What reaches the library, through both routes, from functions of its signatures."""
    log, keep = [], []

    class Fake:
        qdit_last_error, qdit_status_string = binding.lib.qdit_last_error, binding.lib.qdit_status_string

    def flat(v):
        if isinstance(v, C.Structure):
            return tuple(flat(getattr(v, f)) for f, _ in v._fields_)
        if isinstance(v, C._Pointer):
            return flat(v.contents) if v else None
        return v

    status = {"now": 0}
    for name in CALLS:
        fn = getattr(binding.lib, name)
        proto = C.CFUNCTYPE(fn.restype, *fn.argtypes)

        def body(*args, name=name):
            log.append((name, tuple(flat(a) for a in args)))
            return status["now"]

        setattr(Fake, name, proto(body))
        keep.append(getattr(Fake, name))
    real = binding.lib
    monkeypatch.setattr(binding, "lib", Fake)
    _marshal.bind(tuple(C.cast(getattr(Fake, n), C.c_void_p).value for n in binding._NATIVE), binding._WRAPPERS, binding.check,
                  binding.qdit_qparams, binding.qdit_epilogue)
    yield log, status
    _marshal.bind(tuple(C.cast(getattr(real, n), C.c_void_p).value for n in binding._NATIVE), binding._WRAPPERS, binding.check,
                  binding.qdit_qparams, binding.qdit_epilogue)


@pytest.mark.parametrize("name", list(CALLS))
def test_native_and_wrapper_pass_the_same(recorded, name):
    log, status = recorded
    wrapper = binding._WRAPPERS[binding._NATIVE.index(name)]
    for args in CALLS[name]:
        log.clear()
        assert wrapper(*args) == 0 and getattr(q, name)(*args) == 0
        assert len(log) == 2 and log[0] == log[1]
    # the wrapper's own: keywords, numpy arrays and scalars, booleans, an integer where a float is meant
    args = list(CALLS[name][0])
    for other in (np.zeros(4), np.int64(5)):
        a = list(args)
        a[1 if isinstance(other, np.ndarray) else {"qdit_quantize_act": 3, "qdit_attention": 5, "qdit_adaln_modulate": 2}.get(name, 3)] = other
        log.clear()
        assert wrapper(*a) == 0 and getattr(q, name)(*a) == 0
        assert log[0] == log[1]
    with pytest.raises(TypeError):
        getattr(q, name)(*args[:-1] if name == "qdit_quantize_act" else args[:5])
    with pytest.raises(TypeError):
        getattr(q, name)(*args, 1, 2, 3)
    with pytest.raises((TypeError, C.ArgumentError)):
        getattr(q, name)(*([args[0], "text"] + args[2:]))
    status["now"] = q.QDIT_ERR_SHAPE
    args[0] = None
    with pytest.raises(q.QditError) as e:
        getattr(q, name)(*args)
    assert e.value.status == q.QDIT_ERR_SHAPE


def test_keywords_and_defaults(recorded):
    log, _ = recorded
    q.qdit_attention(77, X, Y, Z, 4, 5, 6, 7, 8, 0.5, X, 2, out_scale_dev=Y)
    q.qdit_attention(77, X, Y, Z, 4, 5, 6, 7, 8, 0.5, X, 2, None, Y)
    q.qdit_w4a8_linear(77, X, Y, 1, 2, 3, QP, X, 1, None, Z, 5, w8_scratch=X)
    q.qdit_w4a8_linear(77, X, Y, 1, 2, 3, QP, X, 1, None, Z, 5, X)
    assert log[0] == log[1] and log[2] == log[3]


@pytest.mark.parametrize("name", list(CALLS))
def test_signatures_are_those_of_the_wrappers(name):
    assert inspect.signature(getattr(q, name)) == inspect.signature(binding._WRAPPERS[binding._NATIVE.index(name)])
