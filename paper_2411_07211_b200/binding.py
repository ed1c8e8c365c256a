"""Python binding of libb2blas.so: argument marshalling only.

Every routine of ``include/b2blas.h`` is exposed twice:

* ``lib().b2_saxpy`` etc. -- the raw C symbols through ctypes, with their prototypes set;
* ``axpy``, ``scal``, ... -- callables of the compiled module ``_binding`` that pick the s/d symbol
  from the tensor dtype, pass the tensors' addresses and torch's current stream, and raise
  :class:`B2Error` on a non-zero status.

PyTorch is used for device memory and streams only.  There is no CPU path: if the compiled
CUDA library is missing the import of the symbols fails loudly.
"""
from __future__ import annotations

import ctypes
import inspect
import os

import torch

try:
    from . import _binding as _native  # (built with the library; what keeps it from loading is reported at the first call)
    _native_error = None
except ImportError as e:
    _native, _native_error = None, e

ROW_MAJOR, COL_MAJOR = 101, 102
NO_TRANS, TRANS = 111, 112
UPPER, LOWER = 121, 122
NON_UNIT, UNIT = 131, 132

STATUS_OK, STATUS_LAUNCH_FAILED, STATUS_WORKSPACE_TOO_SMALL = 0, 1, 2
STATUS_NOT_IMPLEMENTED, STATUS_TIMEOUT, STATUS_BAD_CONTEXT = 3, 4, 5
STATUS_TOO_LARGE = 6

KNOB_L1_BLOCKS_PER_SM, KNOB_GEMV_N_TILE_BYTES, KNOB_GEMV_T_ROWS, KNOB_TRI_ROWS = 0, 1, 2, 3
KNOB_GER_ROWS, KNOB_USE_PDL, KNOB_TRSV_DEBUG_SKIP, KNOB_TRI_WIDE = 4, 5, 6, 7
KNOB_TRSV_PREFETCH_BYTES = 8
KNOB_TRSV_FRONT, KNOB_TRSV_CLUSTER = 9, 10
KNOB_TRSV_PM_FROM, KNOB_TRI_TILE, KNOB_TRI_TILE_UNIT, KNOB_NARROW_BLOCK = 11, 12, 13, 14
KNOB_TRI_BULK, KNOB_TRSV_STREAMS, KNOB_GATHER, KNOB_TRSV_DEBUG_LATE, KNOB_TRSV_SHORT_ROWS = 15, 16, 17, 18, 19

# B2BLAS_LIB selects another build of the same library (the bounds-checking one, libb2blas_dbg.so)
LIB_PATH = os.environ.get("B2BLAS_LIB") or os.path.join(os.path.dirname(os.path.abspath(__file__)), "libb2blas.so")

_i64, _int, _vp, _f, _d = ctypes.c_int64, ctypes.c_int, ctypes.c_void_p, ctypes.c_float, ctypes.c_double


class B2Ctx(ctypes.Structure):
    _fields_ = [("stream", _vp), ("workspace", _vp), ("workspace_bytes", ctypes.c_size_t),
                ("device_status", _vp), ("wait_limit", ctypes.c_ulonglong)]


class B2Error(RuntimeError):
    def __init__(self, name, status):
        self.status = status
        msg = lib().b2_status_string(status).decode()
        super().__init__(f"{name} returned {status}: {msg}")


def _protos():
    cp = ctypes.POINTER(B2Ctx)
    out = {}
    for p, sc in (("s", _f), ("d", _d)):
        out[f"b2_{p}axpy"] = [cp, _i64, sc, _vp, _i64, _vp, _i64]
        out[f"b2_{p}scal"] = [cp, _i64, sc, _vp, _i64]
        out[f"b2_{p}copy"] = [cp, _i64, _vp, _i64, _vp, _i64]
        out[f"b2_{p}swap"] = [cp, _i64, _vp, _i64, _vp, _i64]
        out[f"b2_{p}rot"] = [cp, _i64, _vp, _i64, _vp, _i64, sc, sc]
        out[f"b2_{p}rotm"] = [cp, _i64, _vp, _i64, _vp, _i64, _vp]
        out[f"b2_{p}dot"] = [cp, _i64, _vp, _i64, _vp, _i64, _vp]
        out[f"b2_{p}asum"] = [cp, _i64, _vp, _i64, _vp]
        out[f"b2_{p}nrm2"] = [cp, _i64, _vp, _i64, _vp]
        out[f"b2_i{p}amax"] = [cp, _i64, _vp, _i64, _vp]
        out[f"b2_{p}gemv"] = [cp, _int, _int, _i64, _i64, sc, _vp, _i64, _vp, _i64, sc, _vp, _i64]
        out[f"b2_{p}ger"] = [cp, _int, _i64, _i64, sc, _vp, _i64, _vp, _i64, _vp, _i64]
        out[f"b2_{p}symv"] = [cp, _int, _int, _i64, sc, _vp, _i64, _vp, _i64, sc, _vp, _i64]
        out[f"b2_{p}syr"] = [cp, _int, _int, _i64, sc, _vp, _i64, _vp, _i64]
        out[f"b2_{p}syr2"] = [cp, _int, _int, _i64, sc, _vp, _i64, _vp, _i64, _vp, _i64]
        out[f"b2_{p}trmv"] = [cp, _int, _int, _int, _int, _i64, _vp, _i64, _vp, _i64]
        out[f"b2_{p}trsv"] = [cp, _int, _int, _int, _int, _i64, _vp, _i64, _vp, _i64]
    out["b2_dsdot"] = [cp, _i64, _vp, _i64, _vp, _i64, _vp]
    out["b2_sdsdot"] = [cp, _i64, _f, _vp, _i64, _vp, _i64, _vp]
    out["b2_sdot_noalloc"] = [_vp, _i64, _vp, _i64, _vp, _i64, _vp]
    out["b2_workspace_reset"] = [cp]
    return out


_lib = None


def lib():
    """The loaded library; raises if it has not been built (no fallback exists)."""
    global _lib
    if _lib is None:
        if not os.path.exists(LIB_PATH):
            raise ImportError(
                f"{LIB_PATH} is missing: build it with `python -m paper_2411_07211_b200.build` "
                "(there is no CPU fallback)")
        h = ctypes.CDLL(LIB_PATH)
        for name, args in _protos().items():
            fn = getattr(h, name)
            fn.argtypes = args
            fn.restype = _int
        h.b2_workspace_min_bytes.restype = ctypes.c_size_t
        h.b2_workspace_bytes.restype = ctypes.c_size_t
        h.b2_workspace_query.restype = ctypes.c_size_t
        h.b2_workspace_query.argtypes = [_i64, _i64, ctypes.c_size_t]
        h.b2_status_string.restype = ctypes.c_char_p
        h.b2_status_string.argtypes = [_int]
        h.b2_version.restype = _int
        h.b2_launch_count.restype = ctypes.c_ulonglong
        h.b2_set_tuning.argtypes = [_int, _i64]
        h.b2_set_tuning.restype = _int
        h.b2_get_tuning.argtypes = [_int]
        h.b2_get_tuning.restype = _i64
        h.b2_debug_bounds_report.argtypes = [ctypes.POINTER(ctypes.c_ulonglong)]
        h.b2_debug_bounds_report.restype = _int
        h.b2_debug_bounds_shrink.argtypes = [_int]
        h.b2_debug_bounds_shrink.restype = _int
        _lib = h
    return _lib


def exported_symbols():
    return sorted(_protos().keys()) + ["b2_workspace_min_bytes", "b2_workspace_bytes", "b2_workspace_query", "b2_status_string",
                                       "b2_version", "b2_launch_count", "b2_set_tuning", "b2_get_tuning",
                                       "b2_debug_bounds_report", "b2_debug_bounds_shrink"]


class Context(_native.ContextBase if _native else object):
    """Owns the workspace and status word (torch tensors); the calls build the b2_ctx from it and from
    torch's current stream."""

    def __init__(self, device="cuda", workspace_bytes: int | None = None, wait_limit: int = 0):
        h = lib()
        self.device = torch.device(device)
        self._device_index = -1 if self.device.index is None else self.device.index  # -1: the current device
        nbytes = int(workspace_bytes if workspace_bytes is not None else h.b2_workspace_bytes())
        self.workspace = torch.zeros(nbytes + 256, dtype=torch.uint8, device=self.device)
        off = (-self.workspace.data_ptr()) % 256
        self._ws_ptr = self.workspace.data_ptr() + off
        self._ws_bytes = nbytes
        self.status = torch.zeros(1, dtype=torch.int32, device=self.device)
        self.wait_limit = wait_limit

    def struct(self) -> B2Ctx:
        stream = torch.cuda.current_stream(self.device).cuda_stream
        return B2Ctx(stream, self._ws_ptr, self._ws_bytes, self.status.data_ptr(), self.wait_limit)

    def reset(self):
        c = self.struct()
        st = lib().b2_workspace_reset(ctypes.byref(c))
        if st:
            raise B2Error("b2_workspace_reset", st)
        self.status.zero_()

    def device_status(self) -> int:
        return int(self.status.item())


def _p(t):
    if t is None:
        return None
    if isinstance(t, int):
        return t
    assert t.is_cuda, "b2blas routines take device tensors"
    return t.data_ptr()


def _need_native():
    """The compiled module, or an ImportError that says why there is none."""
    if _native is None:
        lib()
        raise ImportError(f"the compiled module paper_2411_07211_b200._binding does not load ({_native_error}): build it "
                          "with `python -m paper_2411_07211_b200.build`") from _native_error
    return _native


def _missing(name):
    def call(*args, **kwargs):
        _need_native()
    call.__name__ = name
    return call


_NAMES = ("axpy", "scal", "copy", "swap", "rot", "rotm", "dot", "dsdot", "sdsdot", "asum", "nrm2", "iamax",
          "gemv", "ger", "syr", "syr2", "symv", "trmv", "trsv")


def _signature(params):
    kind = inspect.Parameter.POSITIONAL_OR_KEYWORD
    return inspect.Signature([inspect.Parameter(p, kind) for p in params.split()] + [inspect.Parameter("check", kind, default=True)])


def _routine(name):
    return _routines[name]


_routines = _native.routines(LIB_PATH, B2Error, lib, _signature, _routine) if _native else {name: _missing(name) for name in _NAMES}


def prepare(thunk):
    """Runs `thunk` (calls of this module) once and returns a callable that repeats exactly those
    library calls with the arguments marshalled then -- same stream, same pointers -- without
    going through the interpreter for each of them.  For timing loops over small problems; the
    returned callable returns the last status.  What is recorded are the calls that the thunk makes
    on the thread that runs it; any number of threads may be inside prepare()."""
    return _need_native().record(thunk)


# help() of a routine tells its parameters.  Every one ends with `check=True`: raise B2Error on a non-zero status
# instead of returning it.
# ---- level 1 ----------------------------------------------------------------------------
axpy = _routines["axpy"]
scal = _routines["scal"]
copy = _routines["copy"]
swap = _routines["swap"]
rot = _routines["rot"]
dsdot = _routines["dsdot"]
sdsdot = _routines["sdsdot"]
dot = _routines["dot"]
asum = _routines["asum"]
nrm2 = _routines["nrm2"]
iamax = _routines["iamax"]


def rotm(ctx, n, x, incx, y, incy, param, check=True):
    """param: 5 host values [flag, h11, h21, h12, h22] (any sequence); None passes a NULL pointer."""
    if param is None:
        return _routines["rotm"](ctx, n, x, incx, y, incy, None, check)
    ctype = ctypes.c_float if x.dtype == torch.float32 else ctypes.c_double
    host = (ctype * 5)(*[float(v) for v in param])
    _need_native().keep(host)
    return _routines["rotm"](ctx, n, x, incx, y, incy, ctypes.addressof(host), check)


# ---- level 2 ----------------------------------------------------------------------------
gemv = _routines["gemv"]
ger = _routines["ger"]
syr = _routines["syr"]
syr2 = _routines["syr2"]
symv = _routines["symv"]
trmv = _routines["trmv"]
trsv = _routines["trsv"]


def set_tuning(knob: int, value: int):
    if lib().b2_set_tuning(knob, value) != 0:
        raise ValueError(f"unknown tuning knob {knob}")


def get_tuning(knob: int) -> int:
    return int(lib().b2_get_tuning(knob))


def debug_bounds_report():
    """(violations since the last report, first offending address, its size) of the bounds-checking
    build; None in the ordinary build."""
    out = (ctypes.c_ulonglong * 3)()
    st = lib().b2_debug_bounds_report(out)
    if st == STATUS_NOT_IMPLEMENTED:
        return None
    if st:
        raise B2Error("b2_debug_bounds_report", st)
    return int(out[0]), int(out[1]), int(out[2])


def debug_bounds_shrink(nbytes: int) -> bool:
    """Test hook of the bounds-checking build; False in the ordinary build."""
    return lib().b2_debug_bounds_shrink(int(nbytes)) == 0


def launch_count() -> int:
    return int(lib().b2_launch_count())


def sdot_noalloc(n, x, incx, y, incy, result, stream=None, check=True):
    """b2_sdot_noalloc: float dot product that needs no Context (no workspace): its scratch is a
    fixed array inside the library.  For callers that cannot get device memory when they call;
    calls must not overlap on the GPU."""
    if stream is None:
        stream = torch.cuda.current_stream(x.device).cuda_stream
    st = lib().b2_sdot_noalloc(stream, n, _p(x), incx, _p(y), incy, _p(result))
    if check and st != 0:
        raise B2Error("b2_sdot_noalloc", st)
    return st
