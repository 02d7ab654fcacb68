"""Python binding of libe3j (the sm_100a fused equivariant convolution).

Argument marshalling only: every function below has the name of the C entry point
it calls (see include/e3j.h) and passes device pointers of torch tensors straight
through.  torch is used for device memory and streams, nothing else; there is no
CPU or PyTorch fallback -- if the compiled library is missing, or a call fails,
an exception is raised.

    plan = e3j_plan_create("128x0e+128x1o", 3, None, 3)
    rowptr, sender_perm, colptr = e3j_graph_prepare(n_nodes, senders, receivers)
    out = e3j_conv_fwd(plan, x, sh, w, senders, receivers, rowptr)
    gx, gsh, gw = e3j_conv_bwd(plan, x, sh, w, senders, receivers, grad_out,
                               rowptr, sender_perm, colptr)
"""
from __future__ import annotations

import ctypes
import importlib
import sysconfig
import warnings
from pathlib import Path

__all__ = [
    "E3JError", "Plan", "library_path", "e3j_plan_create", "e3j_plan_destroy", "e3j_plan_info",
    "e3j_plan_paths", "e3j_plan_records", "e3j_plan_signature", "e3j_plan_device_status", "e3j_graph_prepare", "e3j_graph_validate",
    "e3j_conv_fwd_workspace_bytes", "e3j_conv_bwd_workspace_bytes", "e3j_conv_bwd_shares_bytes", "e3j_conv_fwd", "e3j_conv_fwd_noalloc", "e3j_noalloc_status",
    "e3j_conv_bwd", "e3j_graph_prepare_padded", "e3j_conv_fwd_padded", "e3j_conv_bwd_padded",
    "e3j_conv_bwd_bwd_workspace_bytes", "e3j_conv_bwd_bwd",
    "e3j_radial_weights", "e3j_conv_radial_fwd_workspace_bytes", "e3j_conv_radial_fwd_least_workspace_bytes",
    "e3j_conv_radial_bwd_workspace_bytes",
    "e3j_conv_radial_fwd", "e3j_conv_radial_bwd", "e3j_conv_radial_vec_fwd", "e3j_conv_radial_vec_fwd_workspace_bytes", "e3j_conv_radial_vec_fwd_least_workspace_bytes", "e3j_conv_radial_vec_bwd", "e3j_conv_radial_vec_bwd_workspace_bytes",
    "e3j_tp_fwd", "e3j_tp_bwd", "e3j_bwd_schedule_bytes", "e3j_bwd_schedule_build", "e3j_conv_bwd_scheduled", "e3j_harmonics_fwd", "e3j_harmonics_bwd", "e3j_conv_vec_fwd", "e3j_conv_vec_bwd",
    "e3j_conv_vec_fwd_workspace_bytes", "e3j_conv_vec_bwd_workspace_bytes", "e3j_conv_fwd_f64", "e3j_conv_bwd_f64", "e3j_shard_prepare", "e3j_rows_gather", "e3j_rows_add", "e3j_status_string", "e3j_selftest_bounded_wait", "e3j_launch_count", "E3J_PLAN_GENERIC_ONLY",
    "E3J_PLAN_COLLAPSE_OUTPUTS", "E3J_PLAN_RADIAL_MATERIALISE",
]

E3J_PLAN_GENERIC_ONLY = 1
E3J_PLAN_COLLAPSE_OUTPUTS = 2
E3J_PLAN_RADIAL_MATERIALISE = 4
# status codes of include/e3j.h
E3J_OK, E3J_ERR_INVALID_ARG, E3J_ERR_BAD_IRREPS, E3J_ERR_MUL_NOT_UNIFORM = 0, -1, -2, -3
E3J_ERR_UNSUPPORTED, E3J_ERR_WORKSPACE, E3J_ERR_CUDA, E3J_ERR_GRAPH = -4, -5, -6, -7
_LIB_PATH = Path(__file__).resolve().parent / "libe3j.so"
_lib = None


class E3JError(RuntimeError):
    def __init__(self, status: int, where: str):
        lib = _load()
        msg = lib.e3j_status_string(status).decode()
        if status == -6:
            msg += f" (cudaError {lib.e3j_last_cuda_error()})"
        super().__init__(f"{where}: {msg} [status {status}]")
        self.status = status


class _PlanInfo(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in
                ("n_channels", "d_in", "d_sh", "n_paths", "d_out", "nnz", "n_pairs", "specialised")]


class _PathInfo(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in
                ("in_index", "l1", "p1", "l2", "L", "p", "x_off", "y_off", "out_off")]


def library_path() -> Path:
    return _LIB_PATH


def _load():
    """Loads libe3j.so; raises if it has not been built (no fallback exists)."""
    global _lib
    if _lib is not None:
        return _lib
    if not _LIB_PATH.exists():
        raise RuntimeError(
            f"{_LIB_PATH} is missing: build it with `python -m paper_2609_35099_b200.build` "
            "(nvcc, sm_100a). There is no CPU or PyTorch fallback.")
    lib = ctypes.CDLL(str(_LIB_PATH))
    vp, i64, i32, sz, u32 = ctypes.c_void_p, ctypes.c_int64, ctypes.c_int, ctypes.c_size_t, ctypes.c_uint
    lib.e3j_plan_create.argtypes = [ctypes.POINTER(vp), ctypes.c_char_p, i32, ctypes.c_char_p, i32, u32]
    lib.e3j_plan_destroy.argtypes = [vp]
    lib.e3j_plan_info.argtypes = [vp, ctypes.POINTER(_PlanInfo)]
    lib.e3j_plan_paths.argtypes = [vp, ctypes.POINTER(_PathInfo), i32]
    lib.e3j_plan_records.argtypes = [vp, vp, vp, vp, vp, vp, i32]
    lib.e3j_plan_signature.argtypes = [vp]
    lib.e3j_plan_signature.restype = ctypes.c_char_p
    lib.e3j_plan_device_status.argtypes = [vp, ctypes.POINTER(ctypes.c_int32)]
    lib.e3j_plan_device_status.restype = i32
    lib.e3j_graph_prepare.argtypes = [i64, i64, vp, vp, vp, vp, vp, vp]
    lib.e3j_graph_validate.argtypes = [i64, i64, vp, vp, vp, vp]
    lib.e3j_graph_prepare_padded.argtypes = [i64, i64, vp, vp, vp, vp, vp, vp]
    lib.e3j_conv_fwd_workspace_bytes.argtypes = [vp, i64, i64]
    lib.e3j_conv_fwd_workspace_bytes.restype = sz
    lib.e3j_conv_bwd_workspace_bytes.argtypes = [vp, i64, i64]
    lib.e3j_conv_bwd_workspace_bytes.restype = sz
    lib.e3j_conv_bwd_shares_bytes.argtypes = [vp, i64, i32]
    lib.e3j_conv_bwd_shares_bytes.restype = sz
    lib.e3j_conv_fwd.argtypes = [vp, i64, i64] + [vp] * 8 + [sz, vp]
    lib.e3j_conv_bwd.argtypes = [vp, i64, i64] + [vp] * 13 + [sz, vp]
    lib.e3j_conv_fwd_padded.argtypes = [vp, i64, i64] + [vp] * 8 + [sz, vp]
    lib.e3j_conv_bwd_bwd_workspace_bytes.argtypes = [vp, i64, i64]
    lib.e3j_conv_bwd_bwd_workspace_bytes.restype = sz
    lib.e3j_conv_bwd_bwd.argtypes = [vp, i64, i64] + [vp] * 17 + [sz, vp]
    lib.e3j_conv_bwd_padded.argtypes = [vp, i64, i64] + [vp] * 13 + [sz, vp]
    lib.e3j_conv_fwd_noalloc.argtypes = [vp, i64, i64] + [vp] * 7
    lib.e3j_conv_fwd_noalloc.restype = i32
    lib.e3j_noalloc_status.argtypes = [ctypes.POINTER(ctypes.c_int32)]
    lib.e3j_noalloc_status.restype = i32
    lib.e3j_radial_weights.argtypes = [vp, i64, i32] + [vp] * 4
    lib.e3j_radial_weights.restype = i32
    lib.e3j_conv_radial_fwd_workspace_bytes.argtypes = [vp, i64, i64, i32]
    lib.e3j_conv_radial_fwd_workspace_bytes.restype = sz
    for name in ("e3j_conv_radial_fwd_least_workspace_bytes", "e3j_conv_radial_vec_fwd_least_workspace_bytes"):
        getattr(lib, name).argtypes = [vp, i64, i64, i32]
        getattr(lib, name).restype = sz
    lib.e3j_conv_radial_bwd_workspace_bytes.argtypes = [vp, i64, i64, i32]
    lib.e3j_conv_radial_bwd_workspace_bytes.restype = sz
    lib.e3j_conv_radial_fwd.argtypes = [vp, i64, i64, i32] + [vp] * 9 + [sz, vp]
    lib.e3j_conv_radial_fwd.restype = i32
    lib.e3j_conv_radial_vec_fwd_workspace_bytes.argtypes = [vp, i64, i64, i32]
    lib.e3j_conv_radial_vec_fwd_workspace_bytes.restype = sz
    lib.e3j_conv_radial_vec_fwd.argtypes = [vp, i64, i64, i32] + [vp] * 9 + [sz, vp]
    lib.e3j_conv_radial_vec_fwd.restype = i32
    lib.e3j_conv_radial_vec_bwd_workspace_bytes.argtypes = [vp, i64, i64, i32]
    lib.e3j_conv_radial_vec_bwd_workspace_bytes.restype = sz
    lib.e3j_conv_radial_vec_bwd.argtypes = [vp, i64, i64, i32] + [vp] * 15 + [sz, vp]
    lib.e3j_conv_radial_vec_bwd.restype = i32
    lib.e3j_conv_radial_bwd.argtypes = [vp, i64, i64, i32] + [vp] * 15 + [sz, vp]
    lib.e3j_conv_radial_bwd.restype = i32
    lib.e3j_tp_fwd.argtypes = [vp, i64] + [vp] * 5
    lib.e3j_tp_bwd.argtypes = [vp, i64] + [vp] * 8
    lib.e3j_harmonics_fwd.argtypes = [i32, i64, vp, vp, vp]
    lib.e3j_harmonics_fwd.restype = i32
    lib.e3j_harmonics_bwd.argtypes = [i32, i64, vp, vp, vp, vp]
    lib.e3j_harmonics_bwd.restype = i32
    for name in ("e3j_conv_vec_fwd_workspace_bytes", "e3j_conv_vec_bwd_workspace_bytes"):
        getattr(lib, name).argtypes = [vp, i64, i64]
        getattr(lib, name).restype = sz
    lib.e3j_conv_vec_fwd.argtypes = [vp, i64, i64] + [vp] * 8 + [sz, vp]
    lib.e3j_conv_vec_fwd.restype = i32
    lib.e3j_conv_vec_bwd.argtypes = [vp, i64, i64] + [vp] * 13 + [sz, vp]
    lib.e3j_conv_vec_bwd.restype = i32
    lib.e3j_bwd_schedule_bytes.argtypes = [vp, i64, i64]
    lib.e3j_bwd_schedule_bytes.restype = sz
    lib.e3j_bwd_schedule_build.argtypes = [vp, i64, i64, vp, vp, vp, sz, vp]
    lib.e3j_bwd_schedule_build.restype = i32
    lib.e3j_conv_bwd_scheduled.argtypes = [vp, i64, i64] + [vp] * 9 + [sz, vp]
    lib.e3j_conv_bwd_scheduled.restype = i32
    lib.e3j_conv_f64_workspace_bytes.argtypes = [vp, i64, i64]
    lib.e3j_conv_f64_workspace_bytes.restype = sz
    lib.e3j_conv_fwd_f64.argtypes = [vp, i64, i64] + [vp] * 8 + [sz, vp]
    lib.e3j_conv_fwd_f64.restype = i32
    lib.e3j_conv_bwd_f64.argtypes = [vp, i64, i64] + [vp] * 12 + [sz, vp]
    lib.e3j_conv_bwd_f64.restype = i32
    lib.e3j_shard_prepare_workspace_bytes.argtypes = [i64]
    lib.e3j_shard_prepare_workspace_bytes.restype = sz
    lib.e3j_shard_prepare.argtypes = [i64, i64, i32, i32] + [vp] * 7 + [sz, vp]
    lib.e3j_shard_prepare.restype = i32
    lib.e3j_rows_gather.argtypes = [vp, vp, vp, i64, i64, vp]
    lib.e3j_rows_gather.restype = i32
    lib.e3j_rows_add.argtypes = [vp, vp, vp, i64, i64, vp]
    lib.e3j_rows_add.restype = i32
    lib.e3j_selftest_bounded_wait.argtypes = [vp, u32, ctypes.POINTER(ctypes.c_int32), ctypes.POINTER(ctypes.c_int32)]
    lib.e3j_selftest_bounded_wait.restype = i32
    lib.e3j_status_string.argtypes = [i32]
    lib.e3j_status_string.restype = ctypes.c_char_p
    lib.e3j_last_cuda_error.restype = i32
    lib.e3j_launch_count.restype = i64
    for name in ("e3j_plan_create", "e3j_plan_destroy", "e3j_plan_info", "e3j_plan_paths", "e3j_plan_records",
                 "e3j_graph_prepare", "e3j_graph_validate", "e3j_conv_fwd", "e3j_conv_bwd", "e3j_tp_fwd",
                 "e3j_tp_bwd"):
        getattr(lib, name).restype = i32
    _lib = lib
    return lib


def _check(status: int, where: str) -> int:
    if status < 0:
        raise E3JError(status, where)
    return status


_native = None      # the marshalling in native code (csrc/host/marshal.cpp), where it has been built
_addresses = {}     # of the entry points it has called


def _address(entry: str) -> int:
    address = _addresses[entry] = ctypes.cast(getattr(_load(), entry), ctypes.c_void_p).value
    return address


def _run(entry: str, *args) -> None:
    """Calls an entry point with integers and addresses (None: NULL); raises on a negative status."""
    if _native is None:
        status = getattr(_load(), entry)(*args)
    else:
        status = _native.call(_addresses.get(entry) or _address(entry), *args)
    if status < 0:
        raise E3JError(status, entry)


def _bytes(entry: str, *args) -> int:
    """The same for the functions that return a size."""
    if _native is None:
        return int(getattr(_load(), entry)(*args))
    return _native.call_size(_addresses.get(entry) or _address(entry), *args)


class Plan:
    """Owner of one e3j_plan handle (released when the object is collected)."""

    def __init__(self, handle: int):
        self.handle = ctypes.c_void_p(handle)
        info = _PlanInfo()
        _check(_load().e3j_plan_info(self.handle, ctypes.byref(info)), "e3j_plan_info")
        for name, _ in _PlanInfo._fields_:
            setattr(self, name, getattr(info, name))

    def __del__(self):
        try:
            e3j_plan_destroy(self)
        except Exception:
            pass


def e3j_plan_create(irreps_in: str, sh_lmax: int, irreps_out: str | None = None, out_lmax: int = -1,
                    flags: int = 0) -> Plan:
    h = ctypes.c_void_p()
    out = irreps_out.encode() if irreps_out is not None else None
    _check(_load().e3j_plan_create(ctypes.byref(h), irreps_in.encode(), sh_lmax, out, out_lmax, flags),
           "e3j_plan_create")
    return Plan(h.value)


def e3j_plan_destroy(plan: Plan) -> None:
    if plan.handle is not None and plan.handle.value:
        _load().e3j_plan_destroy(plan.handle)
        plan.handle = ctypes.c_void_p()


def e3j_plan_info(plan: Plan) -> dict:
    return {name: getattr(plan, name) for name, _ in _PlanInfo._fields_}


def e3j_plan_signature(plan: Plan) -> str:
    return _load().e3j_plan_signature(plan.handle).decode()


def e3j_plan_device_status(plan: Plan) -> int:
    """Sticky device status of the plan on the current device (0 = fine); synchronises."""
    st = ctypes.c_int32(0)
    _check(_load().e3j_plan_device_status(plan.handle, ctypes.byref(st)), "e3j_plan_device_status")
    return int(st.value)


def e3j_plan_paths(plan: Plan) -> list[dict]:
    arr = (_PathInfo * plan.n_paths)()
    _check(_load().e3j_plan_paths(plan.handle, arr, plan.n_paths), "e3j_plan_paths")
    return [{name: getattr(p, name) for name, _ in _PathInfo._fields_} for p in arr]


def e3j_plan_records(plan: Plan):
    """(i0, i1, i2, i3, val) numpy arrays of the coefficient records (host side)."""
    import numpy as np
    n = plan.nnz
    idx = [np.zeros(n, dtype=np.int32) for _ in range(4)]
    val = np.zeros(n, dtype=np.float64)
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    _check(_load().e3j_plan_records(plan.handle, *map(ptr, idx), ptr(val), n), "e3j_plan_records")
    return (*idx, val)


# ----------------------------------------------------------------- marshalling
# A call's arguments are checked and converted in a few microseconds: with small graphs that is what a call costs.
_torch_module = _current_stream = None


def _stream_reader(torch):
    """A function that gives the current stream's handle: what torch.cuda.current_stream() does without building the
    object, where torch has the (undocumented) calls for it."""
    raw, device = (getattr(torch._C, name, None) for name in ("_cuda_getCurrentRawStream", "_cuda_getDevice"))
    return (lambda: raw(device())) if raw and device else lambda: torch.cuda.current_stream().cuda_stream


def _marshal_abi(torch) -> str:
    """What the native marshalling is compiled against: it reads the objects of this torch and this interpreter directly."""
    return f"torch {torch.__version__} ({torch.version.git_version}), {sysconfig.get_config_var('EXT_SUFFIX')}"


def _native_marshalling(torch):
    """The module built from csrc/host/marshal.cpp, or None where there is none for this torch and interpreter."""
    try:
        native = importlib.import_module("._marshal", __package__)   # (linked against torch's libraries)
        built_for = getattr(native, "built_for", "unknown")
        if built_for == _marshal_abi(torch):
            return native
        reason = f"built for {built_for}, this is {_marshal_abi(torch)}"
    except ModuleNotFoundError:
        return None
    except ImportError as error:
        reason = str(error)
    warnings.warn(f"native marshalling not used, calls convert their arguments in Python until the next build: {reason}",
                  RuntimeWarning, stacklevel=4)
    return None


def _torch():
    global _torch_module, _current_stream, _native, _dev_ptr, _empty
    if _torch_module is None:
        import torch
        _current_stream = _stream_reader(torch)
        native = _native_marshalling(torch)
        if native is not None:   # several threads may come here together: each leaves the same behind, and no name changes that is read here
            native.set_slow(_dev_ptr_in_python, _empty_in_python)
            _native, _dev_ptr, _empty = native, native.dev_ptr, native.empty
        _torch_module = torch
    return _torch_module


def _dev_ptr_in_python(t, dtype, shape, name):
    """Device address of a contiguous CUDA tensor of that type (and shape, if given); None stays None."""
    if t is None:
        return None
    if not isinstance(t, _torch().Tensor) or not t.is_cuda:
        raise TypeError(f"{name} must be a CUDA tensor")
    if t.dtype != dtype or not t.is_contiguous():
        raise TypeError(f"{name} must be contiguous {dtype}")
    if shape is not None and t.shape != shape:
        raise ValueError(f"{name} has shape {tuple(t.shape)}, expected {tuple(shape)}")
    return t.data_ptr()


def _empty_in_python(shape, dtype, like):
    """An uninitialised tensor on the device of `like`."""
    return _torch().empty(shape, dtype=dtype, device=like.device)


_dev_ptr, _empty = _dev_ptr_in_python, _empty_in_python   # replaced by the native functions where there are any


def _stream(stream):
    if stream is not None:
        return stream.cuda_stream
    _torch()
    return _current_stream()


def _as_torch_stream(stream):
    """stream itself, or torch's view of another library's object with a cuda_stream."""
    torch = _torch()
    return stream if isinstance(stream, torch.cuda.Stream) else torch.cuda.ExternalStream(stream.cuda_stream)


def _workspace(nbytes: int, like, workspace, stream, least=None):
    """The caller's workspace, or a new one of nbytes.  least(): the bytes a call also runs with, where that is less."""
    torch = _torch()
    if workspace is None:
        workspace = _empty((max(nbytes, 256),), torch.uint8, like)
        if stream is not None:   # released when the call returns: not to be used again before that stream is done with it
            workspace.record_stream(_as_torch_stream(stream))
        return workspace
    if workspace.dtype != torch.uint8 or not workspace.is_cuda or \
            workspace.numel() < nbytes and (least is None or workspace.numel() < least()):
        raise ValueError("workspace must be a CUDA uint8 tensor of sufficient size")
    return workspace


def _bwd_workspace(nbytes: int, plan, n_edges: int, like, workspace, stream, want_x: bool):
    """_workspace of a call with a backward: nbytes less the room for shares of grad_x where that gradient is not wanted, and a
    caller's workspace may be without that room."""
    if want_x and workspace is None:
        return _workspace(nbytes, like, None, stream)
    least = nbytes - e3j_conv_bwd_shares_bytes(plan, n_edges)
    return _workspace(nbytes if want_x else least, like, workspace, stream, lambda: least)


def e3j_graph_prepare(n_nodes: int, senders, receivers, want_transpose: bool = True, stream=None,
                      _entry: str = "e3j_graph_prepare"):
    """(rowptr, sender_perm, colptr) int32 CUDA tensors; the last two are None unless want_transpose."""
    torch = _torch()
    e = senders.numel()
    rowptr = _empty((n_nodes + 1,), torch.int32, senders)
    perm = _empty((max(e, 1),), torch.int32, senders) if want_transpose else None
    colptr = _empty((n_nodes + 1,), torch.int32, senders) if want_transpose else None
    _run(_entry, n_nodes, e, _dev_ptr(senders, torch.int32, (e,), "senders"),
                                    _dev_ptr(receivers, torch.int32, (e,), "receivers"),
                                    _dev_ptr(rowptr, torch.int32, None, "rowptr"),
                                    _dev_ptr(perm, torch.int32, None, "sender_perm"),
                                    _dev_ptr(colptr, torch.int32, None, "colptr"), _stream(stream))
    if perm is not None:
        perm = perm[:e]
    return rowptr, perm, colptr


def e3j_graph_prepare_padded(n_nodes: int, senders, receivers, want_transpose: bool = True, stream=None):
    """As e3j_graph_prepare for a padded edge list (edges with receiver >= n_nodes are padding and come last):
    rowptr[n_nodes] is the number of real edges, of sender_perm only that many entries are written."""
    return e3j_graph_prepare(n_nodes, senders, receivers, want_transpose, stream, "e3j_graph_prepare_padded")


def e3j_graph_validate(n_nodes: int, senders, receivers, stream=None) -> int:
    """0 if the graph is usable, else the (negative) E3J_ERR_GRAPH status.  Synchronises."""
    torch = _torch()
    if stream is not None:   # the status is cleared, written and read on that stream
        with torch.cuda.stream(_as_torch_stream(stream)):
            return e3j_graph_validate(n_nodes, senders, receivers)
    e = senders.numel()
    status = torch.zeros(1, dtype=torch.int32, device=senders.device)
    _check(_load().e3j_graph_validate(n_nodes, e, _dev_ptr(senders, torch.int32, (e,), "senders"),
                                      _dev_ptr(receivers, torch.int32, (e,), "receivers"),
                                      _dev_ptr(status, torch.int32, None, "status"), _stream(stream)),
           "e3j_graph_validate")
    return int(status.item())


def e3j_conv_fwd_workspace_bytes(plan: Plan, n_nodes: int, n_edges: int) -> int:
    return _bytes("e3j_conv_fwd_workspace_bytes", plan.handle.value, n_nodes, n_edges)


def e3j_conv_bwd_workspace_bytes(plan: Plan, n_nodes: int, n_edges: int) -> int:
    return _bytes("e3j_conv_bwd_workspace_bytes", plan.handle.value, n_nodes, n_edges)


def e3j_conv_bwd_shares_bytes(plan: Plan, n_edges: int, element_bytes: int = 4) -> int:
    """The part of the workspace queries of calls with a backward (element_bytes 8: in float64) that these also run
    without: slower, and with grad_x summed in another order."""
    return _bytes("e3j_conv_bwd_shares_bytes", plan.handle.value, n_edges, element_bytes)


def e3j_conv_fwd(plan: Plan, x, sh, w, senders, receivers, rowptr=None, out=None, workspace=None,
                 stream=None, _entry: str = "e3j_conv_fwd"):
    torch = _torch()
    n, e = x.shape[0], senders.numel()
    f32, i32 = torch.float32, torch.int32
    if out is None:
        out = _empty((n, plan.d_out, plan.n_channels), f32, x)
    nbytes = e3j_conv_fwd_workspace_bytes(plan, n, e)
    workspace = _workspace(nbytes, x, workspace, stream)
    _run(_entry, plan.handle.value, n, e,
        _dev_ptr(x, f32, (n, plan.d_in, plan.n_channels), "x"),
        _dev_ptr(sh, f32, (e, plan.d_sh), "sh"),
        _dev_ptr(w, f32, (e, plan.n_paths, plan.n_channels), "w"),
        _dev_ptr(senders, i32, (e,), "senders"), _dev_ptr(receivers, i32, (e,), "receivers"),
        _dev_ptr(rowptr, i32, (n + 1,), "rowptr"),
        _dev_ptr(out, f32, (n, plan.d_out, plan.n_channels), "out"),
        workspace.data_ptr(), workspace.numel(), _stream(stream))
    return out


def e3j_conv_fwd_padded(plan: Plan, x, sh, w, senders, receivers, rowptr, out=None, workspace=None, stream=None):
    """Forward convolution over a padded edge list; rowptr (from e3j_graph_prepare_padded) is required."""
    return e3j_conv_fwd(plan, x, sh, w, senders, receivers, rowptr, out, workspace, stream, "e3j_conv_fwd_padded")


def e3j_conv_fwd_noalloc(plan: Plan, x, sh, w, senders, receivers, out, stream=None):
    """Forward convolution through the allocation-free entry point.

    For callers that must not allocate device memory at call time (engines that reserve everything at
    start-up, plug-ins without an allocator): the kernel's scratch lives inside the library, and this
    wrapper allocates nothing either, so `out` must be passed in.  Calls on one device share that scratch and
    must not overlap on the GPU."""
    torch = _torch()
    n, e = x.shape[0], senders.numel()
    f32, i32 = torch.float32, torch.int32
    _run("e3j_conv_fwd_noalloc", plan.handle.value, n, e,
        _dev_ptr(x, f32, (n, plan.d_in, plan.n_channels), "x"),
        _dev_ptr(sh, f32, (e, plan.d_sh), "sh"),
        _dev_ptr(w, f32, (e, plan.n_paths, plan.n_channels), "w"),
        _dev_ptr(senders, i32, (e,), "senders"), _dev_ptr(receivers, i32, (e,), "receivers"),
        _dev_ptr(out, f32, (n, plan.d_out, plan.n_channels), "out"), _stream(stream))
    return out


def e3j_noalloc_status() -> int:
    """Status word of the allocation-free entry point on the current device (0 = fine; non-zero: a bounded wait
    inside its kernel gave up and the output of that call is invalid).  Reads and clears; synchronises."""
    st = ctypes.c_int32(0)
    _check(_load().e3j_noalloc_status(ctypes.byref(st)), "e3j_noalloc_status")
    return int(st.value)


def e3j_conv_bwd(plan: Plan, x, sh, w, senders, receivers, grad_out, rowptr=None, sender_perm=None,
                 colptr=None, grad_x=True, grad_sh=True, grad_w=True, workspace=None, stream=None,
                 _entry: str = "e3j_conv_bwd"):
    """Returns (grad_x, grad_sh, grad_w).  Each grad_* argument is True (allocate), False/None
    (not wanted) or a preallocated tensor."""
    torch = _torch()
    n, e = x.shape[0], senders.numel()
    f32, i32 = torch.float32, torch.int32

    def alloc(flag, shape):
        if flag is True:
            return _empty(shape, f32, x)
        return flag if isinstance(flag, torch.Tensor) else None

    grad_x = alloc(grad_x, (n, plan.d_in, plan.n_channels))
    grad_sh = alloc(grad_sh, (e, plan.d_sh))
    grad_w = alloc(grad_w, (e, plan.n_paths, plan.n_channels))
    workspace = _bwd_workspace(e3j_conv_bwd_workspace_bytes(plan, n, e), plan, e, x, workspace, stream, grad_x is not None)
    _run(_entry, plan.handle.value, n, e,
        _dev_ptr(x, f32, (n, plan.d_in, plan.n_channels), "x"),
        _dev_ptr(sh, f32, (e, plan.d_sh), "sh"),
        _dev_ptr(w, f32, (e, plan.n_paths, plan.n_channels), "w"),
        _dev_ptr(senders, i32, (e,), "senders"), _dev_ptr(receivers, i32, (e,), "receivers"),
        _dev_ptr(rowptr, i32, (n + 1,), "rowptr"),
        _dev_ptr(sender_perm, i32, (e,), "sender_perm"), _dev_ptr(colptr, i32, (n + 1,), "colptr"),
        _dev_ptr(grad_out, f32, (n, plan.d_out, plan.n_channels), "grad_out"),
        _dev_ptr(grad_x, f32, (n, plan.d_in, plan.n_channels), "grad_x"),
        _dev_ptr(grad_sh, f32, (e, plan.d_sh), "grad_sh"),
        _dev_ptr(grad_w, f32, (e, plan.n_paths, plan.n_channels), "grad_w"),
        workspace.data_ptr(), workspace.numel(), _stream(stream))
    return grad_x, grad_sh, grad_w


def e3j_conv_bwd_padded(plan: Plan, x, sh, w, senders, receivers, grad_out, rowptr, sender_perm=None,
                        colptr=None, grad_x=True, grad_sh=True, grad_w=True, workspace=None, stream=None):
    """Backward convolution over a padded edge list; rowptr (from e3j_graph_prepare_padded) is required.
    The grad_sh / grad_w rows of padding edges come back as zeros."""
    return e3j_conv_bwd(plan, x, sh, w, senders, receivers, grad_out, rowptr, sender_perm, colptr, grad_x,
                        grad_sh, grad_w, workspace, stream, "e3j_conv_bwd_padded")


def e3j_conv_bwd_bwd_workspace_bytes(plan: Plan, n_nodes: int, n_edges: int) -> int:
    return _bytes("e3j_conv_bwd_bwd_workspace_bytes", plan.handle.value, n_nodes, n_edges)


def e3j_conv_bwd_bwd(plan: Plan, x, sh, w, senders, receivers, grad_out, rowptr, sender_perm, colptr,
                     ct_x=None, ct_sh=None, ct_w=None, gg_out=True, g_x=True, g_sh=True, g_w=True,
                     workspace=None, stream=None):
    """Double backward: cotangents (ct_x, ct_sh, ct_w) of the backward's results -> cotangents
    (gg_out, g_x, g_sh, g_w) of the backward's inputs (grad_out, x, sh, w).  A missing ct_* is zero; each
    output argument is True (allocate), False/None (not wanted) or a preallocated tensor."""
    torch = _torch()
    n, e = x.shape[0], senders.numel()
    f32, i32 = torch.float32, torch.int32

    def alloc(flag, shape):
        if flag is True:
            return _empty(shape, f32, x)
        return flag if isinstance(flag, torch.Tensor) else None

    s_x, s_sh = (n, plan.d_in, plan.n_channels), (e, plan.d_sh)
    s_w, s_out = (e, plan.n_paths, plan.n_channels), (n, plan.d_out, plan.n_channels)
    gg_out, g_x, g_sh, g_w = alloc(gg_out, s_out), alloc(g_x, s_x), alloc(g_sh, s_sh), alloc(g_w, s_w)
    workspace = _bwd_workspace(e3j_conv_bwd_bwd_workspace_bytes(plan, n, e), plan, e, x, workspace, stream, True)
    _run("e3j_conv_bwd_bwd", plan.handle.value, n, e, _dev_ptr(x, f32, s_x, "x"), _dev_ptr(sh, f32, s_sh, "sh"), _dev_ptr(w, f32, s_w, "w"),
        _dev_ptr(senders, i32, (e,), "senders"), _dev_ptr(receivers, i32, (e,), "receivers"),
        _dev_ptr(rowptr, i32, (n + 1,), "rowptr"), _dev_ptr(sender_perm, i32, (e,), "sender_perm"),
        _dev_ptr(colptr, i32, (n + 1,), "colptr"), _dev_ptr(grad_out, f32, s_out, "grad_out"),
        _dev_ptr(ct_x, f32, s_x, "ct_x"), _dev_ptr(ct_sh, f32, s_sh, "ct_sh"), _dev_ptr(ct_w, f32, s_w, "ct_w"),
        _dev_ptr(gg_out, f32, s_out, "gg_out"), _dev_ptr(g_x, f32, s_x, "g_x"), _dev_ptr(g_sh, f32, s_sh, "g_sh"),
        _dev_ptr(g_w, f32, s_w, "g_w"),
        workspace.data_ptr(), workspace.numel(), _stream(stream))
    return gg_out, g_x, g_sh, g_w


def e3j_radial_weights(plan: Plan, h, W, out=None, stream=None):
    """w[E, P, N_q] = h W (the radial network's last layer), materialised."""
    torch = _torch()
    e, hidden = h.shape
    f32 = torch.float32
    if out is None:
        out = _empty((e, plan.n_paths, plan.n_channels), f32, h)
    _run("e3j_radial_weights", plan.handle.value, e, hidden, _dev_ptr(h, f32, (e, hidden), "h"),
        _dev_ptr(W, f32, (hidden, plan.n_paths * plan.n_channels), "W"),
        _dev_ptr(out, f32, (e, plan.n_paths, plan.n_channels), "out"), _stream(stream))
    return out


def e3j_conv_radial_fwd_workspace_bytes(plan: Plan, n_nodes: int, n_edges: int, hidden: int) -> int:
    return _bytes("e3j_conv_radial_fwd_workspace_bytes", plan.handle.value, n_nodes, n_edges, hidden)


def e3j_conv_radial_fwd_least_workspace_bytes(plan: Plan, n_nodes: int, n_edges: int, hidden: int) -> int:
    """The smallest workspace e3j_conv_radial_fwd runs with: where the plan has the kernel for it, without room for the
    edge weights, which are then formed inside the kernel (slower below 2 GiB of them)."""
    return _bytes("e3j_conv_radial_fwd_least_workspace_bytes", plan.handle.value, n_nodes, n_edges, hidden)


def e3j_conv_radial_bwd_workspace_bytes(plan: Plan, n_nodes: int, n_edges: int, hidden: int) -> int:
    return _bytes("e3j_conv_radial_bwd_workspace_bytes", plan.handle.value, n_nodes, n_edges, hidden)


def e3j_conv_radial_fwd(plan: Plan, x, sh, h, W, senders, receivers, rowptr=None, out=None, workspace=None,
                        stream=None):
    """Forward convolution with the edge weights given as (h [E, hidden], W [hidden, P * N_q])."""
    torch = _torch()
    n, e, hidden = x.shape[0], senders.numel(), W.shape[0]
    f32, i32 = torch.float32, torch.int32
    if out is None:
        out = _empty((n, plan.d_out, plan.n_channels), f32, x)
    workspace = _workspace(e3j_conv_radial_fwd_workspace_bytes(plan, n, e, hidden), x, workspace, stream,
                           lambda: e3j_conv_radial_fwd_least_workspace_bytes(plan, n, e, hidden))
    _run("e3j_conv_radial_fwd", plan.handle.value, n, e, hidden,
        _dev_ptr(x, f32, (n, plan.d_in, plan.n_channels), "x"), _dev_ptr(sh, f32, (e, plan.d_sh), "sh"),
        _dev_ptr(h, f32, (e, hidden), "h"), _dev_ptr(W, f32, (hidden, plan.n_paths * plan.n_channels), "W"),
        _dev_ptr(senders, i32, (e,), "senders"), _dev_ptr(receivers, i32, (e,), "receivers"),
        _dev_ptr(rowptr, i32, (n + 1,), "rowptr"),
        _dev_ptr(out, f32, (n, plan.d_out, plan.n_channels), "out"),
        workspace.data_ptr(), workspace.numel(), _stream(stream))
    return out


def e3j_conv_radial_vec_fwd_workspace_bytes(plan: Plan, n_nodes: int, n_edges: int, hidden: int) -> int:
    return _bytes("e3j_conv_radial_vec_fwd_workspace_bytes", plan.handle.value, n_nodes, n_edges, hidden)


def e3j_conv_radial_vec_fwd_least_workspace_bytes(plan: Plan, n_nodes: int, n_edges: int, hidden: int) -> int:
    """As e3j_conv_radial_fwd_least_workspace_bytes, for the call on edge vectors."""
    return _bytes("e3j_conv_radial_vec_fwd_least_workspace_bytes", plan.handle.value, n_nodes, n_edges, hidden)


def e3j_conv_radial_vec_fwd(plan: Plan, x, edge_vec, h, W, senders, receivers, rowptr=None, out=None, workspace=None,
                            stream=None):
    """Forward convolution from edge vectors [E, 3] and the radial layer (h, W): where the plan has the kernels for it
    the harmonics never exist as an array, nor do the edge weights once they would take more than 2 GiB."""
    torch = _torch()
    n, e, hidden = x.shape[0], senders.numel(), W.shape[0]
    f32, i32 = torch.float32, torch.int32
    if out is None:
        out = _empty((n, plan.d_out, plan.n_channels), f32, x)
    workspace = _workspace(e3j_conv_radial_vec_fwd_workspace_bytes(plan, n, e, hidden), x, workspace, stream,
                           lambda: e3j_conv_radial_vec_fwd_least_workspace_bytes(plan, n, e, hidden))
    _run("e3j_conv_radial_vec_fwd", plan.handle.value, n, e, hidden,
        _dev_ptr(x, f32, (n, plan.d_in, plan.n_channels), "x"), _dev_ptr(edge_vec, f32, (e, 3), "edge_vec"),
        _dev_ptr(h, f32, (e, hidden), "h"), _dev_ptr(W, f32, (hidden, plan.n_paths * plan.n_channels), "W"),
        _dev_ptr(senders, i32, (e,), "senders"), _dev_ptr(receivers, i32, (e,), "receivers"),
        _dev_ptr(rowptr, i32, (n + 1,), "rowptr"),
        _dev_ptr(out, f32, (n, plan.d_out, plan.n_channels), "out"),
        workspace.data_ptr(), workspace.numel(), _stream(stream))
    return out


def e3j_conv_radial_bwd(plan: Plan, x, sh, h, W, senders, receivers, grad_out, rowptr=None, sender_perm=None,
                        colptr=None, grad_x=True, grad_sh=True, grad_h=True, grad_W=True, workspace=None,
                        stream=None):
    """Returns (grad_x, grad_sh, grad_h, grad_W); each grad_* argument is True (allocate), False/None (not
    wanted) or a preallocated tensor."""
    torch = _torch()
    n, e, hidden = x.shape[0], senders.numel(), W.shape[0]
    f32, i32 = torch.float32, torch.int32

    def alloc(flag, shape):
        if flag is True:
            return _empty(shape, f32, x)
        return flag if isinstance(flag, torch.Tensor) else None

    s_w = (hidden, plan.n_paths * plan.n_channels)
    grad_x = alloc(grad_x, (n, plan.d_in, plan.n_channels))
    grad_sh = alloc(grad_sh, (e, plan.d_sh))
    grad_h = alloc(grad_h, (e, hidden))
    grad_W = alloc(grad_W, s_w)
    workspace = _bwd_workspace(e3j_conv_radial_bwd_workspace_bytes(plan, n, e, hidden), plan, e, x, workspace, stream, grad_x is not None)
    _run("e3j_conv_radial_bwd", plan.handle.value, n, e, hidden,
        _dev_ptr(x, f32, (n, plan.d_in, plan.n_channels), "x"), _dev_ptr(sh, f32, (e, plan.d_sh), "sh"),
        _dev_ptr(h, f32, (e, hidden), "h"), _dev_ptr(W, f32, s_w, "W"),
        _dev_ptr(senders, i32, (e,), "senders"), _dev_ptr(receivers, i32, (e,), "receivers"),
        _dev_ptr(rowptr, i32, (n + 1,), "rowptr"),
        _dev_ptr(sender_perm, i32, (e,), "sender_perm"), _dev_ptr(colptr, i32, (n + 1,), "colptr"),
        _dev_ptr(grad_out, f32, (n, plan.d_out, plan.n_channels), "grad_out"),
        _dev_ptr(grad_x, f32, (n, plan.d_in, plan.n_channels), "grad_x"),
        _dev_ptr(grad_sh, f32, (e, plan.d_sh), "grad_sh"),
        _dev_ptr(grad_h, f32, (e, hidden), "grad_h"), _dev_ptr(grad_W, f32, s_w, "grad_W"),
        workspace.data_ptr(), workspace.numel(), _stream(stream))
    return grad_x, grad_sh, grad_h, grad_W


def e3j_conv_radial_vec_bwd_workspace_bytes(plan: Plan, n_nodes: int, n_edges: int, hidden: int) -> int:
    return _bytes("e3j_conv_radial_vec_bwd_workspace_bytes", plan.handle.value, n_nodes, n_edges, hidden)


def e3j_conv_radial_vec_bwd(plan: Plan, x, edge_vec, h, W, senders, receivers, grad_out, rowptr=None, sender_perm=None,
                            colptr=None, grad_x=True, grad_vec=True, grad_h=True, grad_W=True, workspace=None,
                            stream=None):
    """Backward of e3j_conv_radial_vec_fwd: (grad_x, grad_vec, grad_h, grad_W); each grad_* argument is True
    (allocate), False/None (not wanted) or a preallocated tensor."""
    torch = _torch()
    n, e, hidden = x.shape[0], senders.numel(), W.shape[0]
    f32, i32 = torch.float32, torch.int32

    def alloc(flag, shape):
        if flag is True:
            return _empty(shape, f32, x)
        return flag if isinstance(flag, torch.Tensor) else None

    s_w = (hidden, plan.n_paths * plan.n_channels)
    grad_x = alloc(grad_x, (n, plan.d_in, plan.n_channels))
    grad_vec = alloc(grad_vec, (e, 3))
    grad_h = alloc(grad_h, (e, hidden))
    grad_W = alloc(grad_W, s_w)
    workspace = _bwd_workspace(e3j_conv_radial_vec_bwd_workspace_bytes(plan, n, e, hidden), plan, e, x, workspace, stream, grad_x is not None)
    _run("e3j_conv_radial_vec_bwd", plan.handle.value, n, e, hidden,
        _dev_ptr(x, f32, (n, plan.d_in, plan.n_channels), "x"), _dev_ptr(edge_vec, f32, (e, 3), "edge_vec"),
        _dev_ptr(h, f32, (e, hidden), "h"), _dev_ptr(W, f32, s_w, "W"),
        _dev_ptr(senders, i32, (e,), "senders"), _dev_ptr(receivers, i32, (e,), "receivers"),
        _dev_ptr(rowptr, i32, (n + 1,), "rowptr"),
        _dev_ptr(sender_perm, i32, (e,), "sender_perm"), _dev_ptr(colptr, i32, (n + 1,), "colptr"),
        _dev_ptr(grad_out, f32, (n, plan.d_out, plan.n_channels), "grad_out"),
        _dev_ptr(grad_x, f32, (n, plan.d_in, plan.n_channels), "grad_x"), _dev_ptr(grad_vec, f32, (e, 3), "grad_vec"),
        _dev_ptr(grad_h, f32, (e, hidden), "grad_h"), _dev_ptr(grad_W, f32, s_w, "grad_W"),
        workspace.data_ptr(), workspace.numel(), _stream(stream))
    return grad_x, grad_vec, grad_h, grad_W


def e3j_tp_fwd(plan: Plan, x1, x2, w, out=None, stream=None):
    torch = _torch()
    rows, f32 = x1.shape[0], torch.float32
    if out is None:
        out = _empty((rows, plan.d_out, plan.n_channels), f32, x1)
    _run("e3j_tp_fwd", plan.handle.value, rows, _dev_ptr(x1, f32, (rows, plan.d_in, plan.n_channels), "x1"),
        _dev_ptr(x2, f32, (rows, plan.d_sh), "x2"),
        _dev_ptr(w, f32, (rows, plan.n_paths, plan.n_channels), "w"),
        _dev_ptr(out, f32, (rows, plan.d_out, plan.n_channels), "out"), _stream(stream))
    return out


def e3j_tp_bwd(plan: Plan, x1, x2, w, grad_out, grad_x1=True, grad_x2=True, grad_w=True, stream=None):
    torch = _torch()
    rows, f32 = x1.shape[0], torch.float32

    def alloc(flag, shape):
        if flag is True:
            return _empty(shape, f32, x1)
        return flag if isinstance(flag, torch.Tensor) else None

    grad_x1 = alloc(grad_x1, (rows, plan.d_in, plan.n_channels))
    grad_x2 = alloc(grad_x2, (rows, plan.d_sh))
    grad_w = alloc(grad_w, (rows, plan.n_paths, plan.n_channels))
    _run("e3j_tp_bwd", plan.handle.value, rows, _dev_ptr(x1, f32, (rows, plan.d_in, plan.n_channels), "x1"),
        _dev_ptr(x2, f32, (rows, plan.d_sh), "x2"),
        _dev_ptr(w, f32, (rows, plan.n_paths, plan.n_channels), "w"),
        _dev_ptr(grad_out, f32, (rows, plan.d_out, plan.n_channels), "grad_out"),
        _dev_ptr(grad_x1, f32, None, "grad_x1"), _dev_ptr(grad_x2, f32, None, "grad_x2"),
        _dev_ptr(grad_w, f32, None, "grad_w"), _stream(stream))
    return grad_x1, grad_x2, grad_w


def e3j_bwd_schedule_bytes(plan: Plan, n_nodes: int, n_edges: int) -> int:
    """Device bytes a backward schedule may need; 0 if the plan has no scheduled kernel."""
    return int(_load().e3j_bwd_schedule_bytes(plan.handle, n_nodes, n_edges))


def e3j_bwd_schedule_build(plan: Plan, n_nodes: int, senders, receivers, stream=None):
    """The processing order of e3j_conv_bwd_scheduled for this graph (a device uint8 tensor).  The graph arrays may
    live on the device or the host; the order is computed on the host."""
    torch = _torch()
    e = senders.numel()
    dev = senders.device if senders.is_cuda else torch.device("cuda", torch.cuda.current_device())
    nbytes = e3j_bwd_schedule_bytes(plan, n_nodes, e)
    if nbytes == 0:
        raise RuntimeError("e3j_bwd_schedule_build: the plan has no scheduled backward kernel")
    snd = senders.detach().to("cpu", torch.int32).contiguous()
    rcv = receivers.detach().to("cpu", torch.int32).contiguous()
    sched = torch.empty(nbytes, dtype=torch.uint8, device=dev)
    with torch.cuda.device(dev):
        _check(_load().e3j_bwd_schedule_build(plan.handle, n_nodes, e, ctypes.c_void_p(snd.data_ptr()),
                                              ctypes.c_void_p(rcv.data_ptr()), ctypes.c_void_p(sched.data_ptr()), nbytes,
                                              _stream(stream)), "e3j_bwd_schedule_build")
    return sched


def e3j_conv_bwd_scheduled(plan: Plan, x, sh, w, schedule, grad_out, grad_x=None, grad_sh=None, grad_w=None,
                           workspace=None, stream=None):
    """e3j_conv_bwd over a schedule from e3j_bwd_schedule_build: (grad_x, grad_sh, grad_w), all three always."""
    torch = _torch()
    n, e = x.shape[0], w.shape[0]
    f32 = torch.float32
    if grad_x is None:
        grad_x = _empty((n, plan.d_in, plan.n_channels), f32, x)
    if grad_sh is None:
        grad_sh = _empty((e, plan.d_sh), f32, x)
    if grad_w is None:
        grad_w = _empty((e, plan.n_paths, plan.n_channels), f32, x)
    workspace = _workspace(e3j_conv_bwd_workspace_bytes(plan, n, e), x, workspace, stream)
    if schedule.dtype != torch.uint8 or not schedule.is_cuda:
        raise ValueError("schedule must be the CUDA uint8 tensor returned by e3j_bwd_schedule_build")
    _run("e3j_conv_bwd_scheduled", plan.handle.value, n, e, _dev_ptr(x, f32, (n, plan.d_in, plan.n_channels), "x"), _dev_ptr(sh, f32, (e, plan.d_sh), "sh"),
        _dev_ptr(w, f32, (e, plan.n_paths, plan.n_channels), "w"), schedule.data_ptr(),
        _dev_ptr(grad_out, f32, (n, plan.d_out, plan.n_channels), "grad_out"),
        _dev_ptr(grad_x, f32, (n, plan.d_in, plan.n_channels), "grad_x"), _dev_ptr(grad_sh, f32, (e, plan.d_sh), "grad_sh"),
        _dev_ptr(grad_w, f32, (e, plan.n_paths, plan.n_channels), "grad_w"),
        workspace.data_ptr(), workspace.numel(), _stream(stream))
    return grad_x, grad_sh, grad_w


def e3j_harmonics_fwd(lmax: int, edge_vec, out=None, stream=None):
    """sh[E, (lmax+1)^2] = Y(edge_vec / |edge_vec|), component-normalised real harmonics."""
    torch = _torch()
    e, f32 = edge_vec.shape[0], torch.float32
    if out is None:
        out = _empty((e, (lmax + 1) ** 2), f32, edge_vec)
    _run("e3j_harmonics_fwd", lmax, e, _dev_ptr(edge_vec, f32, (e, 3), "edge_vec"),
                                     _dev_ptr(out, f32, (e, (lmax + 1) ** 2), "sh"), _stream(stream))
    return out


def e3j_harmonics_bwd(lmax: int, edge_vec, grad_sh, out=None, stream=None):
    """grad_vec[E, 3] of e3j_harmonics_fwd."""
    torch = _torch()
    e, f32 = edge_vec.shape[0], torch.float32
    if out is None:
        out = _empty((e, 3), f32, edge_vec)
    _run("e3j_harmonics_bwd", lmax, e, _dev_ptr(edge_vec, f32, (e, 3), "edge_vec"),
                                     _dev_ptr(grad_sh, f32, (e, (lmax + 1) ** 2), "grad_sh"),
                                     _dev_ptr(out, f32, (e, 3), "grad_vec"), _stream(stream))
    return out


def e3j_conv_vec_fwd_workspace_bytes(plan: Plan, n_nodes: int, n_edges: int) -> int:
    return _bytes("e3j_conv_vec_fwd_workspace_bytes", plan.handle.value, n_nodes, n_edges)


def e3j_conv_vec_bwd_workspace_bytes(plan: Plan, n_nodes: int, n_edges: int) -> int:
    return _bytes("e3j_conv_vec_bwd_workspace_bytes", plan.handle.value, n_nodes, n_edges)


def e3j_conv_vec_fwd(plan: Plan, x, edge_vec, w, senders, receivers, rowptr=None, out=None, workspace=None,
                     stream=None):
    """Forward convolution with the harmonics formed from the edge vectors [E, 3]."""
    torch = _torch()
    n, e = x.shape[0], senders.numel()
    f32, i32 = torch.float32, torch.int32
    if out is None:
        out = _empty((n, plan.d_out, plan.n_channels), f32, x)
    workspace = _workspace(e3j_conv_vec_fwd_workspace_bytes(plan, n, e), x, workspace, stream)
    _run("e3j_conv_vec_fwd", plan.handle.value, n, e, _dev_ptr(x, f32, (n, plan.d_in, plan.n_channels), "x"),
        _dev_ptr(edge_vec, f32, (e, 3), "edge_vec"), _dev_ptr(w, f32, (e, plan.n_paths, plan.n_channels), "w"),
        _dev_ptr(senders, i32, (e,), "senders"), _dev_ptr(receivers, i32, (e,), "receivers"),
        _dev_ptr(rowptr, i32, (n + 1,), "rowptr"), _dev_ptr(out, f32, (n, plan.d_out, plan.n_channels), "out"),
        workspace.data_ptr(), workspace.numel(), _stream(stream))
    return out


def e3j_conv_vec_bwd(plan: Plan, x, edge_vec, w, senders, receivers, grad_out, rowptr=None, sender_perm=None,
                     colptr=None, grad_x=True, grad_vec=True, grad_w=True, workspace=None, stream=None):
    """Returns (grad_x, grad_vec, grad_w); each grad_* argument is True (allocate), False/None or a tensor."""
    torch = _torch()
    n, e = x.shape[0], senders.numel()
    f32, i32 = torch.float32, torch.int32

    def alloc(flag, shape):
        if flag is True:
            return _empty(shape, f32, x)
        return flag if isinstance(flag, torch.Tensor) else None

    grad_x = alloc(grad_x, (n, plan.d_in, plan.n_channels))
    grad_vec = alloc(grad_vec, (e, 3))
    grad_w = alloc(grad_w, (e, plan.n_paths, plan.n_channels))
    workspace = _bwd_workspace(e3j_conv_vec_bwd_workspace_bytes(plan, n, e), plan, e, x, workspace, stream, grad_x is not None)
    _run("e3j_conv_vec_bwd", plan.handle.value, n, e, _dev_ptr(x, f32, (n, plan.d_in, plan.n_channels), "x"),
        _dev_ptr(edge_vec, f32, (e, 3), "edge_vec"), _dev_ptr(w, f32, (e, plan.n_paths, plan.n_channels), "w"),
        _dev_ptr(senders, i32, (e,), "senders"), _dev_ptr(receivers, i32, (e,), "receivers"),
        _dev_ptr(rowptr, i32, (n + 1,), "rowptr"), _dev_ptr(sender_perm, i32, (e,), "sender_perm"),
        _dev_ptr(colptr, i32, (n + 1,), "colptr"),
        _dev_ptr(grad_out, f32, (n, plan.d_out, plan.n_channels), "grad_out"),
        _dev_ptr(grad_x, f32, (n, plan.d_in, plan.n_channels), "grad_x"), _dev_ptr(grad_vec, f32, (e, 3), "grad_vec"),
        _dev_ptr(grad_w, f32, (e, plan.n_paths, plan.n_channels), "grad_w"),
        workspace.data_ptr(), workspace.numel(), _stream(stream))
    return grad_x, grad_vec, grad_w


def e3j_conv_fwd_f64(plan: Plan, x, sh, w, senders, receivers, rowptr=None, out=None, stream=None):
    """Float64 forward convolution (per-path kernels; odd channel counts and l > 3 on table-driven ones)."""
    torch = _torch()
    n, e, f64, i32 = x.shape[0], senders.numel(), torch.float64, torch.int32
    if out is None:
        out = _empty((n, plan.d_out, plan.n_channels), f64, x)
    ws = _workspace(_bytes("e3j_conv_f64_workspace_bytes", plan.handle.value, n, e) - e3j_conv_bwd_shares_bytes(plan, e, 8),
                    x, None, stream)
    _run("e3j_conv_fwd_f64", plan.handle.value, n, e, _dev_ptr(x, f64, (n, plan.d_in, plan.n_channels), "x"), _dev_ptr(sh, f64, (e, plan.d_sh), "sh"),
        _dev_ptr(w, f64, (e, plan.n_paths, plan.n_channels), "w"), _dev_ptr(senders, i32, (e,), "senders"),
        _dev_ptr(receivers, i32, (e,), "receivers"), _dev_ptr(rowptr, i32, (n + 1,), "rowptr"),
        _dev_ptr(out, f64, (n, plan.d_out, plan.n_channels), "out"), ws.data_ptr(), ws.numel(),
        _stream(stream))
    return out


def e3j_conv_bwd_f64(plan: Plan, x, sh, w, senders, receivers, grad_out, sender_perm=None, colptr=None, stream=None):
    """Float64 backward convolution: (grad_x, grad_sh, grad_w)."""
    torch = _torch()
    n, e, f64, i32 = x.shape[0], senders.numel(), torch.float64, torch.int32
    gx = _empty((n, plan.d_in, plan.n_channels), f64, x)
    gsh = _empty((e, plan.d_sh), f64, x)
    gw = _empty((e, plan.n_paths, plan.n_channels), f64, x)
    ws = _workspace(_bytes("e3j_conv_f64_workspace_bytes", plan.handle.value, n, e), x, None, stream)
    _run("e3j_conv_bwd_f64", plan.handle.value, n, e, _dev_ptr(x, f64, (n, plan.d_in, plan.n_channels), "x"), _dev_ptr(sh, f64, (e, plan.d_sh), "sh"),
        _dev_ptr(w, f64, (e, plan.n_paths, plan.n_channels), "w"), _dev_ptr(senders, i32, (e,), "senders"),
        _dev_ptr(receivers, i32, (e,), "receivers"), _dev_ptr(sender_perm, i32, (e,), "sender_perm"),
        _dev_ptr(colptr, i32, (n + 1,), "colptr"), _dev_ptr(grad_out, f64, (n, plan.d_out, plan.n_channels), "grad_out"),
        _dev_ptr(gx, f64, None, "grad_x"), _dev_ptr(gsh, f64, None, "grad_sh"), _dev_ptr(gw, f64, None, "grad_w"),
        ws.data_ptr(), ws.numel(), _stream(stream))
    return gx, gsh, gw


def e3j_shard_prepare(n_nodes: int, node_lo: int, node_hi: int, senders, receivers, stream=None):
    """Local problem of the rank that owns receivers [node_lo, node_hi): (local_senders, local_receivers, halo_ids)
    for its slice of the edge list (global ids in).  halo_ids (ascending global ids) is cut to its length, which
    costs one device-to-host read of the count."""
    torch = _torch()
    if stream is not None:   # the count is cleared, written and read on that stream
        with torch.cuda.stream(_as_torch_stream(stream)):
            return e3j_shard_prepare(n_nodes, node_lo, node_hi, senders, receivers)
    e, i32 = senders.numel(), torch.int32
    dev = senders.device
    ls = torch.empty(max(e, 1), dtype=i32, device=dev)
    lr = torch.empty(max(e, 1), dtype=i32, device=dev)
    halo = torch.empty(max(n_nodes, 1), dtype=i32, device=dev)
    count = torch.zeros(1, dtype=i32, device=dev)
    ws = torch.empty(max(int(_load().e3j_shard_prepare_workspace_bytes(n_nodes)), 256), dtype=torch.uint8, device=dev)
    _check(_load().e3j_shard_prepare(n_nodes, e, node_lo, node_hi, _dev_ptr(senders, i32, (e,), "senders"),
                                     _dev_ptr(receivers, i32, (e,), "receivers"), _dev_ptr(ls, i32, None, "local_senders"),
                                     _dev_ptr(lr, i32, None, "local_receivers"), _dev_ptr(halo, i32, None, "halo_ids"),
                                     _dev_ptr(count, i32, None, "n_halo"), ws.data_ptr(), ws.numel(),
                                     _stream(stream)), "e3j_shard_prepare")
    return ls[:e], lr[:e], halo[:int(count.item())]


def e3j_rows_gather(dst, src, ids, stream=None):
    """dst[i] = src[ids[i]] for float32 tensors whose trailing dimensions form the row."""
    torch = _torch()
    n = ids.numel()
    row = src[0].numel() if src.shape[0] else 0
    if n:
        _check(_load().e3j_rows_gather(_dev_ptr(dst, torch.float32, None, "dst"), _dev_ptr(src, torch.float32, None, "src"),
                                       _dev_ptr(ids, torch.int32, (n,), "ids"), n, row, _stream(stream)), "e3j_rows_gather")
    return dst


def e3j_rows_add(dst, src, ids, stream=None):
    """dst[ids[i]] += src[i]; ids must not repeat within the call."""
    torch = _torch()
    n = ids.numel()
    row = dst[0].numel() if dst.shape[0] else 0
    if n:
        _check(_load().e3j_rows_add(_dev_ptr(dst, torch.float32, None, "dst"), _dev_ptr(src, torch.float32, None, "src"),
                                    _dev_ptr(ids, torch.int32, (n,), "ids"), n, row, _stream(stream)), "e3j_rows_add")
    return dst


def e3j_selftest_bounded_wait(plan: Plan, spin_limit: int = 1000):
    """(returned, abort_flag) of a wait that is made to run out after spin_limit polls; sets the plan's status word."""
    a, b = ctypes.c_int32(-1), ctypes.c_int32(-1)
    _check(_load().e3j_selftest_bounded_wait(plan.handle, spin_limit, ctypes.byref(a), ctypes.byref(b)),
           "e3j_selftest_bounded_wait")
    return int(a.value), int(b.value)


def e3j_status_string(status: int) -> str:
    return _load().e3j_status_string(status).decode()


def e3j_launch_count() -> int:
    return int(_load().e3j_launch_count())
