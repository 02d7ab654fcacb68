"""The native marshalling of the Python binding (csrc/host/marshal.cpp), as far as it runs without a device."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

import paper_2609_35099_b200 as e3j

e3j._torch()
native = e3j._native
pytestmark = pytest.mark.skipif(native is None, reason="_marshal was not built")


def test_what_is_not_plainly_right_goes_to_the_python_check():
    assert native.dev_ptr(None, torch.float32, (3,), "x") is None
    for t in (torch.zeros(3), [1.0], torch.nn.Parameter(torch.zeros(3)), torch.empty(3, device="meta")):
        with pytest.raises(TypeError, match="x must be a CUDA tensor"):
            native.dev_ptr(t, torch.float32, (3,), "x")


def test_empty_is_torch_empty():
    like = torch.zeros(2)
    for shape in ((3, 4, 5), (0, 7), (9,), 6, (2, 1, 2, 1, 2)):
        a, b = native.empty(shape, torch.float64, like), torch.empty(shape, dtype=torch.float64)
        assert a.shape == b.shape and a.dtype == b.dtype and a.device == like.device and a.is_contiguous() and not a.requires_grad
    with pytest.raises(RuntimeError):
        native.empty((-1, 2), torch.float32, like)
    with pytest.raises(AttributeError):
        native.empty((1, 2), torch.float32, [1.0])


def test_arguments_arrive_as_they_are():
    seen = []
    kinds = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_int] + [ctypes.c_void_p] * 16 + [ctypes.c_size_t, ctypes.c_void_p]
    f = ctypes.CFUNCTYPE(ctypes.c_int, *kinds)(lambda *a: seen.append(a) or -7)
    args = [1 << 47, -5, -2, *range(100, 115), None, (1 << 64) - 1, 9]
    assert native.call(ctypes.cast(f, ctypes.c_void_p).value, *args) == -7
    assert list(seen[0]) == args
    g = ctypes.CFUNCTYPE(ctypes.c_size_t, ctypes.c_int64)(lambda n: (1 << 40) + n)
    assert native.call_size(ctypes.cast(g, ctypes.c_void_p).value, 3) == (1 << 40) + 3
    with pytest.raises(TypeError):
        native.call(ctypes.cast(f, ctypes.c_void_p).value, *range(25))
    with pytest.raises(TypeError):
        native.call(ctypes.cast(f, ctypes.c_void_p).value, 1.5)


def test_sizes_and_refusals_are_those_of_the_library():
    plan = e3j.e3j_plan_create("8x0e+8x1o", 2, None, 2)
    want = e3j._load().e3j_conv_bwd_workspace_bytes(plan.handle, 10, 20)
    assert e3j.e3j_conv_bwd_workspace_bytes(plan, 10, 20) == want > 0
    with pytest.raises(e3j.E3JError, match="e3j_tp_fwd: invalid argument"):
        e3j._run("e3j_tp_fwd", plan.handle.value, 5, None, None, None, None, 0)
