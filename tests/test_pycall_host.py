"""The decode-path calls of the extension module against their ctypes form, without a GPU: both hand the C functions
the same structs and values, refuse the same tensors and pass the status back."""
import ctypes

import pytest
import torch

import paper_2402_18096_gb300 as pkg

pkg.load()
pytestmark = pytest.mark.skipif(pkg._pycall is None, reason="Python headers are not installed")


class FakeTensor:
    """What the binding asks of a tensor."""

    def __init__(self, ptr, is_cuda=True, contiguous=True, dtype=torch.bfloat16, n=64):
        self.ptr, self.is_cuda, self.contiguous, self.dtype, self.n = ptr, is_cuda, contiguous, dtype, n

    def is_contiguous(self):
        return self.contiguous

    def data_ptr(self):
        return self.ptr

    def numel(self):
        return self.n


class FakeCache:
    def __init__(self, shape, **tensors):
        self.shape = shape
        for i, n in enumerate(("k_hi", "v_hi", "hi_tok", "acc", "k_codes", "v_codes", "k_params", "v_params", "lo_tok",
                               "balancer", "k_hi_params", "v_hi_params")):
            setattr(self, n, tensors.get(n, FakeTensor(0x1000 * (i + 1))))

    c = pkg.LayerCache.c


class FakeStream:
    cuda_stream = (1 << 47) + 5


P, I, Z, F = ctypes.c_void_p, ctypes.c_int32, ctypes.c_size_t, ctypes.c_float
STEP = ctypes.CFUNCTYPE(I, P, P, I, P, P, P, I, P, F, P, I, P, Z, P)
ATTENTION = ctypes.CFUNCTYPE(I, P, P, I, P, F, P, I, P, P, P, Z, P)


@pytest.fixture
def calls(monkeypatch):
    """Both paths bound to functions that record their arguments (structs by value) and return the status 3."""
    seen = []

    def record(shape, cache, *rest):
        seen.append((ctypes.string_at(shape, ctypes.sizeof(pkg._Shape)), ctypes.string_at(cache, ctypes.sizeof(pkg._Cache)),
                     *rest))
        return 3

    step, attention = STEP(record), ATTENTION(record)
    lib = pkg.load()

    class Lib:
        mikv_decode_step, mikv_decode_attention = step, attention

    monkeypatch.setattr(pkg, "load", lambda *a, **k: Lib)
    pkg._pycall.bind(ctypes.cast(step, P).value, ctypes.cast(attention, P).value, torch.float32)
    yield seen
    pkg._pycall.bind(ctypes.cast(lib.mikv_decode_step, P).value, ctypes.cast(lib.mikv_decode_attention, P).value,
                     torch.float32)


def both(monkeypatch, seen, call):
    """The recorded arguments of call() through the extension module and through ctypes."""
    got = []
    for native in (True, False):
        with monkeypatch.context() as m:
            if not native:
                m.setattr(pkg, "_pycall", None)
            with pytest.raises(pkg.MikvError) as e:
                call()
            assert e.value.code == 3
            got.append(seen.pop())
            assert not seen
    # ctypes callbacks receive a null pointer as None
    return [[None if x in (0, None) else x for x in g] for g in got]


SHAPES = [pkg.Shape(3, 8, 2, 2, 64, 17, 48), pkg.Shape(1, 4, 4, 3, 128, 5, 64, hi_bits=8),
          pkg.Shape(2, 8, 8, 4, 32, 9, 64, k_channel_group=64), pkg.Shape(2, 8, 8, 0, 32, 9, 0)]


@pytest.mark.parametrize("shape", SHAPES, ids=range(len(SHAPES)))
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_step_arguments(monkeypatch, calls, shape, dtype):
    cache = FakeCache(shape, balancer=None if shape.k_channel_group else FakeTensor(0xABC000), k_hi_params=None)
    out, ws = FakeTensor(0x7F00_0000_1000, dtype=dtype), FakeTensor(0x7F00_0000_2000, n=12345)
    a, b = both(monkeypatch, calls, lambda: pkg.mikv_decode_step(
        cache, 11, FakeTensor(0x10), FakeTensor(0x20), FakeTensor(0x30), -7, FakeTensor(0x40), 0.0883883, out, ws,
        stream=FakeStream))
    assert a == b
    assert a[2:] == [11, 0x10, 0x20, 0x30, -7, 0x40, a[8], 0x7F00_0000_1000, None if dtype != torch.float32 else 1,
                     0x7F00_0000_2000, 12345, FakeStream.cuda_stream]


@pytest.mark.parametrize("logits", [None, FakeTensor(0x50)], ids=["none", "logits"])
def test_attention_arguments(monkeypatch, calls, logits):
    cache = FakeCache(SHAPES[0])
    out, ws = FakeTensor(0x60, dtype=torch.float32), FakeTensor(0x70, n=1 << 33)
    a, b = both(monkeypatch, calls, lambda: pkg.mikv_decode_attention(
        cache, 0, FakeTensor(0x10), 1, out, ws, hi_logits=logits, ml=None, stream=FakeStream))
    assert a == b and a[9] == 0x70 and a[10] == 1 << 33


@pytest.mark.parametrize("bad", [dict(is_cuda=False), dict(contiguous=False)], ids=["host", "strided"])
@pytest.mark.parametrize("where", ["v_codes", "q", "slots", "out", "ws"])
def test_refused_tensors(monkeypatch, calls, bad, where):
    t = {n: FakeTensor(0x100 + i) for i, n in enumerate(("q", "k", "v", "slots", "out", "ws"))}
    cache = FakeCache(SHAPES[0])
    if where in t:
        t[where] = FakeTensor(0x900, **bad)
    else:
        setattr(cache, where, FakeTensor(0x900, **bad))
    said = []
    for native in (True, False):
        with monkeypatch.context() as m:
            if not native:
                m.setattr(pkg, "_pycall", None)
            with pytest.raises(ValueError) as e:
                pkg.mikv_decode_step(cache, 1, t["q"], t["k"], t["v"], 0, t["slots"], 1.0, t["out"], t["ws"],
                                     stream=FakeStream)
            said.append(str(e.value))
    assert said[0] == said[1] and not calls


def test_other_argument_types(monkeypatch, calls):
    """Integers that are not Python ints pass on both paths; a float for an integer is refused on both."""
    import numpy as np
    t = [FakeTensor(0x100 + i) for i in range(6)]
    call = lambda n: pkg.mikv_decode_step(FakeCache(SHAPES[0]), n, t[0], t[1], t[2], 0, t[3], np.float32(0.5), t[4],  # noqa: E731
                                          t[5], stream=FakeStream)
    a, b = both(monkeypatch, calls, lambda: call(1 << 33 | 9))  # the low 32 bits
    assert a == b and a[2] == 9
    for native in (True, False):
        with monkeypatch.context() as m:
            if not native:
                m.setattr(pkg, "_pycall", None)
            with pytest.raises(ctypes.ArgumentError):
                call(2.0)
    assert not calls
