"""The binding's extension module on the CPU: entry points are stand-ins that record what they are given, tensors are objects
with the attributes that the module asks for."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

_I, _P = ctypes.c_int, ctypes.c_void_p
_LINEAR = ctypes.CFUNCTYPE(_I, _P, _I, _I, _I, _P, _I, _P, _I, _P, _P, _I, _I, _P, ctypes.c_size_t, _P, _P)


class FakeTensor:
    is_cuda = True

    def __init__(self, shape, stride, dtype=torch.float16):
        self.shape, self._stride, self.dtype = shape, stride, dtype

    def stride(self):
        return self._stride

    def data_ptr(self):
        return 0x10000

    def numel(self):
        n = 1
        for s in self.shape:
            n *= s
        return n

    def is_contiguous(self):
        return True


@pytest.fixture
def calls():
    from paper_2604_04701_b200 import build
    build.build()
    import paper_2604_04701_b200 as mx
    from paper_2604_04701_b200 import binding
    mx.lib()
    c, seen = binding._calls, []

    @_LINEAR
    def linear(x, M, K, ldx, w, ldw, sw, N, p, y, ldy, out_kind, ws, nbytes, st, s):
        seen.append((M, K, ldx, ldw, N, ldy, out_kind, nbytes))
        return 0

    at = ctypes.cast(linear, _P).value
    c.bind(at, at, at, lambda: 0, lambda d: 0, torch.float16, torch.float32)
    yield c, seen, mx.MuxqParams()
    binding._lib = binding._calls = None  # bound anew on the next use
    mx.lib()


def _args(mx_params, X=None, w_q=None, out=None):
    X = X or FakeTensor((32, 64), (64, 1))
    w_q = w_q or FakeTensor((128, 64), (64, 1), torch.int8)
    out = out or FakeTensor((32, 128), (128, 1))
    ws = FakeTensor((4096,), (1,), torch.uint8)
    return X, w_q, FakeTensor((1,), (1,)), mx_params, ws, FakeTensor((1,), (1,)), 0, out, None


def test_the_library_is_published_after_everything_that_comes_with_it():
    """Threads that make their first call at the same time: whoever finds the library loaded finds the extension module too.
    Looked at between any two instructions of the loading function."""
    import sys

    import paper_2604_04701_b200 as mx
    from paper_2604_04701_b200 import binding
    mx.lib()
    binding._lib = binding._calls = None
    early = []

    def look(code, offset):
        if binding._lib is not None and binding._calls is None:
            early.append(offset)

    mon, tool = sys.monitoring, sys.monitoring.DEBUGGER_ID
    mon.use_tool_id(tool, "order of publication")
    try:
        mon.register_callback(tool, mon.events.INSTRUCTION, look)
        mon.set_local_events(tool, binding.lib.__code__, mon.events.INSTRUCTION)
        binding.lib()
    finally:
        mon.set_local_events(tool, binding.lib.__code__, 0)
        mon.free_tool_id(tool)
    assert binding._lib is not None and binding._calls is not None and not early


def test_linear_passes_sizes_and_pitches(calls):
    c, seen, p = calls
    assert c.linear(*_args(p, X=FakeTensor((32, 64), (80, 1)), w_q=FakeTensor((128, 64), (96, 1)), out=FakeTensor((32, 128), (136, 1)))) == 0
    assert seen == [(32, 64, 80, 96, 128, 136, 0, 4096)]


def test_linear_refuses_operands_without_dimensions(calls):
    """Sizes and pitches come from the shape and the strides; a tensor that has none must not reach the library."""
    c, seen, p = calls
    none = FakeTensor((), ())
    for bad in (dict(w_q=none), dict(out=none)):
        with pytest.raises(IndexError):
            c.linear(*_args(p, **bad))
    for X in (none, FakeTensor((64,), (1,)), FakeTensor((2, 32, 64), (2048, 64, 1)), FakeTensor((32, 64), (1, 32))):
        with pytest.raises((AssertionError, IndexError)):
            c.linear(*_args(p, X=X))
    assert not seen
