"""Python binding of the C-ABI library declared in include/tvm_attn.h.

Argument marshalling only: every step of the path runs in the CUDA kernels of the library.
PyTorch provides device memory and streams.  The tensor functions go through a native module
(csrc/torch_binding.cpp: a call on a small problem is over on the GPU before Python has compared
its arguments' shapes), the rest through ctypes.  There is no CPU or library fallback: if a
shared object is missing or a call fails, an exception is raised.
"""
import ctypes
import importlib.util
import os

import torch

from . import build as _build

BF16 = 0
FP32 = 1
FLAG_CUDA_CORES = 1

_STATUS_NAMES = {0: "OK", -1: "INVALID_ARG", -2: "UNSUPPORTED", -3: "WORKSPACE_TOO_SMALL", -4: "CUDA_ERROR",
                 -5: "DEVICE_TIMEOUT", -6: "TOO_LARGE"}
NOALLOC_MAX_ROWS = 262144


class TvmAttnError(RuntimeError):
    def __init__(self, where, code, text):
        super().__init__("%s failed: %s (%d): %s" % (where, _STATUS_NAMES.get(code, "?"), code, text))
        self.code = code


class Params(ctypes.Structure):
    _fields_ = [("B", ctypes.c_int32), ("H", ctypes.c_int32), ("N", ctypes.c_int32), ("d", ctypes.c_int32),
                ("scale", ctypes.c_float), ("dtype", ctypes.c_int32), ("flags", ctypes.c_uint32), ("M", ctypes.c_int32),
                ("q_strides", ctypes.c_int64 * 3), ("k_strides", ctypes.c_int64 * 3)]


_lib = None
_native = None
_BOUND = ("tvm_attn_jvp_fwd", "tvm_attn_jvp_bwd", "tvm_attn_jvp_bwd_noalloc", "tvm_attn_jvp_workspace_bytes",
          "tvm_qk_rmsnorm_jvp_fwd", "tvm_qk_rmsnorm_jvp_bwd", "tvm_qk_rmsnorm_jvp_workspace_bytes")
EXPORTS = ("tvm_attn_jvp_workspace_bytes", "tvm_attn_jvp_fwd", "tvm_attn_jvp_bwd", "tvm_attn_jvp_bwd_noalloc",
           "tvm_attn_check_status", "tvm_attn_selftest_timeout",
           "tvm_qk_rmsnorm_jvp_fwd", "tvm_qk_rmsnorm_jvp_bwd", "tvm_qk_rmsnorm_jvp_workspace_bytes",
           "tvm_attn_launch_count", "tvm_attn_strerror", "tvm_attn_version", "tvm_attn_set_profiling",
           "tvm_attn_get_profile")


def library_path():
    """Path of the shared object; the environment variable TVM_ATTN_LIBRARY selects another build."""
    return os.environ.get("TVM_ATTN_LIBRARY") or _build.LIB_PATH


def load(build_if_missing=False):
    """Loads libtvm_attn.so (built in-tree by build.py).  Raises if it is not there; with build_if_missing it is built
    first, as is the native half of this binding, which the tensor functions load on their first call."""
    global _lib
    if build_if_missing and not os.path.exists(_build.binding_path()):
        _build.build_binding()
    if _lib is not None:
        return _lib
    path = library_path()
    if not os.path.exists(path):
        if not build_if_missing:
            raise FileNotFoundError("%s is missing: run paper_2511_19797_b200/build.py (nvcc, sm_100a) first" % path)
        _build.build()
    lib = ctypes.CDLL(path)
    vp, pp = ctypes.c_void_p, ctypes.POINTER(Params)
    lib.tvm_attn_jvp_workspace_bytes.restype = ctypes.c_size_t
    lib.tvm_attn_jvp_workspace_bytes.argtypes = [pp, ctypes.c_int]
    lib.tvm_attn_jvp_fwd.restype = ctypes.c_int
    lib.tvm_attn_jvp_fwd.argtypes = [pp] + [vp] * 10 + [vp, ctypes.c_size_t, vp]
    lib.tvm_attn_jvp_bwd.restype = ctypes.c_int
    lib.tvm_attn_jvp_bwd.argtypes = [pp] + [vp] * 18 + [vp, ctypes.c_size_t, vp]
    lib.tvm_attn_jvp_bwd_noalloc.restype = ctypes.c_int
    lib.tvm_attn_jvp_bwd_noalloc.argtypes = [pp] + [vp] * 18 + [vp]
    lib.tvm_attn_check_status.restype = ctypes.c_int
    lib.tvm_attn_check_status.argtypes = [vp]
    lib.tvm_qk_rmsnorm_jvp_workspace_bytes.restype = ctypes.c_size_t
    lib.tvm_qk_rmsnorm_jvp_workspace_bytes.argtypes = [pp]
    lib.tvm_qk_rmsnorm_jvp_fwd.restype = ctypes.c_int
    lib.tvm_qk_rmsnorm_jvp_fwd.argtypes = [pp, ctypes.c_float] + [vp] * 10 + [vp]
    lib.tvm_qk_rmsnorm_jvp_bwd.restype = ctypes.c_int
    lib.tvm_qk_rmsnorm_jvp_bwd.argtypes = [pp, ctypes.c_float] + [vp] * 16 + [vp, ctypes.c_size_t, vp]
    lib.tvm_attn_selftest_timeout.restype = ctypes.c_int
    lib.tvm_attn_selftest_timeout.argtypes = [ctypes.c_uint64, vp]
    lib.tvm_attn_launch_count.restype = ctypes.c_uint64
    lib.tvm_attn_launch_count.argtypes = []
    lib.tvm_attn_strerror.restype = ctypes.c_char_p
    lib.tvm_attn_strerror.argtypes = [ctypes.c_int]
    lib.tvm_attn_version.restype = ctypes.c_int
    lib.tvm_attn_version.argtypes = []
    lib.tvm_attn_set_profiling.restype = ctypes.c_int
    lib.tvm_attn_set_profiling.argtypes = [ctypes.c_int]
    lib.tvm_attn_get_profile.restype = ctypes.c_int
    lib.tvm_attn_get_profile.argtypes = [ctypes.POINTER(ctypes.c_float), ctypes.c_int]
    _lib = lib
    return lib


def _raise(where, code):
    raise TvmAttnError(where, code, load().tvm_attn_strerror(code).decode())


def _load_native():
    """The native half of the binding, bound to the library's entry points.  Raises if it is not built."""
    global _native
    lib = load()
    path = _build.binding_path()
    if not os.path.exists(path):
        raise FileNotFoundError("%s is missing: run paper_2511_19797_b200/build.py first (it is built for one PyTorch)" % path)
    spec = importlib.util.spec_from_file_location("_tvm_binding", path)
    native = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(native)
    native.bind(*[ctypes.cast(getattr(lib, name), ctypes.c_void_p).value for name in _BOUND])
    _native = native
    return native


def _stream_ptr(stream):
    s = stream if stream is not None else torch.cuda.current_stream()
    return ctypes.c_void_p(s.cuda_stream)


def tvm_attn_jvp_workspace_bytes(B, H, N, d, dtype=BF16, is_bwd=True, scale=0.0, flags=0):
    p = Params(B, H, N, d, float(scale), dtype, flags)
    return int(load().tvm_attn_jvp_workspace_bytes(ctypes.byref(p), 1 if is_bwd else 0))


def tvm_attn_jvp_fwd(Q, K, V, tQ, tK, tV, scale=0.0, flags=0, out=None, stream=None):
    """Forward: returns (O, tO, lse, mu).  `out` may hold preallocated (O, tO, lse, mu)."""
    r = (_native or _load_native()).fwd(Q, K, V, tQ, tK, tV, scale, flags, out, None if stream is None else stream.cuda_stream)
    if r.__class__ is int:
        _raise("tvm_attn_jvp_fwd", r)
    return r


def tvm_attn_jvp_bwd(Q, K, V, tQ, tK, tV, O, tO, lse, mu, dO, dtO, scale=0.0, flags=0, out=None, workspace=None,
                     stream=None):
    """Backward: returns (dQ, dK, dV, dtQ, dtK, dtV).  `workspace` is a uint8 CUDA tensor of at least
    tvm_attn_jvp_workspace_bytes(...) bytes; one is allocated with torch when not given.
    dO or dtO may be None (a zero cotangent; dtO=None is the "detach JVP" setting).  With dtO=None the entries
    dtQ, dtK, dtV of `out` may be None too; tensors given there come back zero."""
    r = (_native or _load_native()).bwd(Q, K, V, tQ, tK, tV, O, tO, lse, mu, dO, dtO, scale, flags, out, workspace,
                                        None if stream is None else stream.cuda_stream, False)
    if r.__class__ is int:
        _raise("tvm_attn_jvp_bwd", r)
    return r


def tvm_attn_jvp_bwd_noalloc(Q, K, V, tQ, tK, tV, O, tO, lse, mu, dO, dtO, out, scale=0.0, flags=0, stream=None):
    """Backward for callers that cannot allocate: same result as tvm_attn_jvp_bwd, scratch inside the library.

    `out` must hold the six preallocated gradient tensors (dQ, dK, dV, dtQ, dtK, dtV): this wrapper, like the
    C entry point behind it, allocates nothing.  B*H*N may not exceed NOALLOC_MAX_ROWS.  Calls that may overlap
    on the GPU race on the shared scratch; the first call on a device should come before any stream capture."""
    r = (_native or _load_native()).bwd(Q, K, V, tQ, tK, tV, O, tO, lse, mu, dO, dtO, scale, flags, out, None,
                                        None if stream is None else stream.cuda_stream, True)
    if r.__class__ is int:
        _raise("tvm_attn_jvp_bwd_noalloc", r)
    return r


def tvm_qk_rmsnorm_jvp_fwd(Q, tQ, K, tK, gQ, gK, eps=1e-6, stream=None):
    """RMSNorm QK-normalisation with a tangent: returns (Qn, tQn, Kn, tKn)."""
    r = (_native or _load_native()).norm_fwd(Q, tQ, K, tK, gQ, gK, eps, None if stream is None else stream.cuda_stream)
    if r.__class__ is int:
        _raise("tvm_qk_rmsnorm_jvp_fwd", r)
    return r


def tvm_qk_rmsnorm_jvp_bwd(Q, tQ, K, tK, gQ, gK, dQn, dtQn, dKn, dtKn, eps=1e-6, workspace=None, stream=None):
    """Backward of the normalisation: returns (dQ, dtQ, dK, dtK, dgQ, dgK)."""
    r = (_native or _load_native()).norm_bwd(Q, tQ, K, tK, gQ, gK, dQn, dtQn, dKn, dtKn, eps, workspace,
                                             None if stream is None else stream.cuda_stream)
    if r.__class__ is int:
        _raise("tvm_qk_rmsnorm_jvp_bwd", r)
    return r


def tvm_attn_check_status(stream=None, raise_on_error=True):
    rc = int(load().tvm_attn_check_status(_stream_ptr(stream)))
    if rc != 0 and raise_on_error:
        _raise("tvm_attn_check_status", rc)
    return rc


def tvm_attn_selftest_timeout(limit_ns=1_000_000, stream=None):
    """Enqueues the kernel whose bounded wait runs out on purpose (see include/tvm_attn.h)."""
    rc = int(load().tvm_attn_selftest_timeout(int(limit_ns), _stream_ptr(stream)))
    if rc != 0:
        _raise("tvm_attn_selftest_timeout", rc)


def tvm_attn_launch_count():
    return int(load().tvm_attn_launch_count())


def tvm_attn_version():
    return int(load().tvm_attn_version())


def tvm_attn_set_profiling(enable):
    load().tvm_attn_set_profiling(1 if enable else 0)


def tvm_attn_get_profile():
    """Per-kernel milliseconds of the most recent profiled call, in launch order."""
    buf = (ctypes.c_float * 8)()
    n = int(load().tvm_attn_get_profile(buf, 8))
    if n < 0:
        _raise("tvm_attn_get_profile", n)
    return [float(buf[k]) for k in range(n)]
