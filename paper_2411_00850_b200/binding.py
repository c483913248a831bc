"""Binding of the C-ABI library (include/gwq.h) for torch tensors.

Argument marshalling only: every step of the method runs in the CUDA kernels of
libgwq.so.  PyTorch tensors are used as plain device buffers (data_ptr) and for
the current stream.  The calls a program makes often are marshalled in native
code (csrc/torch_ext.cpp); the library itself is also loaded with ctypes, for
the rarer calls and for programs that want the C functions.  There is no CPU
fallback: a missing library or a missing CUDA device raises.
"""
from __future__ import annotations

import ctypes as C
import importlib.util
import os

import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "libgwq.so")
EXT_PATH = os.path.join(_HERE, "_gwq_torch.so")

GWQ_OK = 0
(GWQ_ERR_INVALID_ARG, GWQ_ERR_UNSUPPORTED, GWQ_ERR_ALLOC, GWQ_ERR_NONFINITE, GWQ_ERR_TIMEOUT,
 GWQ_ERR_CUDA, GWQ_ERR_WORKSPACE) = range(1, 8)
GWQ_F16, GWQ_BF16, GWQ_F32 = 0, 1, 2
STATUS_NAMES = {
    0: "GWQ_OK", 1: "GWQ_ERR_INVALID_ARG", 2: "GWQ_ERR_UNSUPPORTED", 3: "GWQ_ERR_ALLOC",
    4: "GWQ_ERR_NONFINITE", 5: "GWQ_ERR_TIMEOUT", 6: "GWQ_ERR_CUDA", 7: "GWQ_ERR_WORKSPACE",
}
EXPORTS = ("gwq_select_outliers", "gwq_select_outliers_static", "gwq_outliers_rows", "gwq_pack", "gwq_linear", "gwq_linear_ws",
           "gwq_linear_workspace_bytes", "gwq_linear_multi", "gwq_linear_multi_ws", "gwq_linear_multi_workspace_bytes",
           "gwq_gradient_mean", "gwq_quality", "gwq_linear_host", "gwq_linear_host_async", "gwq_device_status", "gwq_set_wait_limit", "gwq_free",
           "gwq_trim_memory", "gwq_status_string")
GWQ_MULTI_MAX = 4


class GwqError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        super().__init__(f"{where}: {STATUS_NAMES.get(status, status)}")


class gwq_outliers(C.Structure):
    _fields_ = [("tag", C.c_uint32), ("N", C.c_int32), ("K", C.c_int32), ("nnz", C.c_int64),
                ("row_ptr", C.c_void_p), ("col_idx", C.c_void_p), ("val", C.c_void_p)]


class gwq_packed(C.Structure):
    _fields_ = [("tag", C.c_uint32), ("N", C.c_int32), ("K", C.c_int32), ("bits", C.c_int32),
                ("group", C.c_int32), ("codes", C.c_void_p), ("scales", C.c_void_p),
                ("zeros", C.c_void_p), ("S", C.POINTER(gwq_outliers)), ("priv", C.c_void_p)]


_lib = None


def load_library(path: str = LIB_PATH) -> C.CDLL:
    """Load libgwq.so and declare the prototypes of include/gwq.h."""
    global _lib
    if _lib is not None:
        return _lib
    if not os.path.exists(path):
        raise RuntimeError(f"{path} is missing: build it with `python -m paper_2411_00850_b200.build` "
                           "(there is no fallback path)")
    lib = C.CDLL(path)
    lib.gwq_select_outliers.restype = C.c_int
    lib.gwq_select_outliers.argtypes = [C.c_void_p, C.c_void_p, C.c_int32, C.c_int32, C.c_double,
                                        C.POINTER(C.POINTER(gwq_outliers)), C.c_void_p]
    lib.gwq_select_outliers_static.restype = C.c_int
    lib.gwq_select_outliers_static.argtypes = [C.c_void_p, C.c_void_p, C.c_int32, C.c_int32, C.c_double,
                                               C.c_void_p, C.c_void_p, C.c_void_p, C.c_int64,
                                               C.POINTER(C.c_int64), C.c_void_p]
    lib.gwq_outliers_rows.restype = C.c_int
    lib.gwq_outliers_rows.argtypes = [C.POINTER(gwq_outliers), C.c_int32, C.c_int32, C.POINTER(C.POINTER(gwq_outliers)),
                                      C.c_void_p]
    lib.gwq_pack.restype = C.c_int
    lib.gwq_pack.argtypes = [C.c_void_p, C.POINTER(gwq_outliers), C.c_int32, C.c_int32, C.c_int32, C.c_int32,
                             C.POINTER(C.POINTER(gwq_packed)), C.c_void_p]
    lib.gwq_linear.restype = C.c_int
    lib.gwq_linear.argtypes = [C.POINTER(gwq_packed), C.c_void_p, C.c_int, C.c_int32, C.c_void_p, C.c_int,
                               C.c_void_p]
    lib.gwq_linear_ws.restype = C.c_int
    lib.gwq_linear_ws.argtypes = [C.POINTER(gwq_packed), C.c_void_p, C.c_int, C.c_int32, C.c_void_p, C.c_int,
                                  C.c_void_p, C.c_size_t, C.c_void_p]
    lib.gwq_linear_workspace_bytes.restype = C.c_size_t
    lib.gwq_linear_workspace_bytes.argtypes = [C.POINTER(gwq_packed), C.c_int, C.c_int32]
    lib.gwq_linear_multi.restype = C.c_int
    lib.gwq_linear_multi.argtypes = [C.POINTER(C.POINTER(gwq_packed)), C.c_int32, C.c_void_p, C.c_int, C.c_int32,
                                     C.POINTER(C.c_void_p), C.c_int, C.c_void_p]
    lib.gwq_linear_multi_ws.restype = C.c_int
    lib.gwq_linear_multi_ws.argtypes = [C.POINTER(C.POINTER(gwq_packed)), C.c_int32, C.c_void_p, C.c_int, C.c_int32,
                                        C.POINTER(C.c_void_p), C.c_int, C.c_void_p, C.c_size_t, C.c_void_p]
    lib.gwq_linear_multi_workspace_bytes.restype = C.c_size_t
    lib.gwq_linear_multi_workspace_bytes.argtypes = [C.POINTER(C.POINTER(gwq_packed)), C.c_int32, C.c_int, C.c_int32]
    lib.gwq_gradient_mean.restype = C.c_int
    lib.gwq_gradient_mean.argtypes = [C.POINTER(C.c_void_p), C.c_int32, C.c_int64, C.c_void_p, C.c_void_p]
    lib.gwq_quality.restype = C.c_int
    lib.gwq_quality.argtypes = [C.c_void_p, C.c_void_p, C.POINTER(gwq_packed), C.POINTER(C.c_double),
                                C.POINTER(C.c_double), C.c_void_p]
    lib.gwq_linear_host.restype = C.c_int
    lib.gwq_linear_host.argtypes = lib.gwq_linear.argtypes
    lib.gwq_linear_host_async.restype = C.c_int
    lib.gwq_linear_host_async.argtypes = lib.gwq_linear.argtypes
    lib.gwq_device_status.restype = C.c_int
    lib.gwq_device_status.argtypes = [C.POINTER(gwq_packed), C.c_void_p]
    lib.gwq_set_wait_limit.restype = C.c_int
    lib.gwq_set_wait_limit.argtypes = [C.POINTER(gwq_packed), C.c_int64]
    lib.gwq_free.restype = None
    lib.gwq_free.argtypes = [C.c_void_p]
    lib.gwq_trim_memory.restype = C.c_int
    lib.gwq_trim_memory.argtypes = [C.c_size_t]
    lib.gwq_status_string.restype = C.c_char_p
    lib.gwq_status_string.argtypes = [C.c_int]
    _lib = lib
    return lib


def _stream_ptr() -> int:
    return torch.cuda.current_stream().cuda_stream


def _dtype_code(t: torch.dtype) -> int:
    if t == torch.float16:
        return GWQ_F16
    if t == torch.bfloat16:
        return GWQ_BF16
    if t == torch.float32:
        return GWQ_F32
    raise TypeError(f"unsupported dtype {t}")


def _check(st: int, where: str):
    if st != GWQ_OK:
        raise GwqError(st, where)


_ext = None


def _load_ext():
    """The native half of this module (csrc/torch_ext.cpp), linked against libgwq.so."""
    global _ext
    if _ext is None:
        load_library()
        if not os.path.exists(EXT_PATH):
            raise RuntimeError(f"{EXT_PATH} is missing: build it with `python -m paper_2411_00850_b200.build`")
        spec = importlib.util.spec_from_file_location("_gwq_torch", EXT_PATH)
        ext = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(ext)
        ext.set_error(GwqError)
        _ext = ext
    return _ext


class _Owned:
    """Owner of a library object: `_addr` its address (0 once freed or given away), `_h` the ctypes pointer to it."""
    _struct = None

    def __init__(self, handle, device):
        self._addr = handle if isinstance(handle, int) else C.cast(handle, C.c_void_p).value or 0
        self.device = device

    @property
    def _h(self):
        return C.cast(self._addr, C.POINTER(self._struct)) if self._addr else None

    def free(self):
        addr, self._addr = self._addr, 0
        if addr:
            load_library().gwq_free(addr)

    def __del__(self):
        try:
            self.free()
        except Exception:
            pass


class Outliers(_Owned):
    """Owner of a gwq_outliers* (CSR of the FP16 outlier matrix S)."""
    _struct = gwq_outliers

    @property
    def N(self): return self._h.contents.N
    @property
    def K(self): return self._h.contents.K
    @property
    def nnz(self): return self._h.contents.nnz

    def arrays(self):
        """(row_ptr int32 [N+1], col_idx int32 [nnz], val int16-bit patterns [nnz]) as tensors."""
        return _load_ext().outlier_arrays(self._addr, self.device.index)


class Packed(_Owned):
    """Owner of a gwq_packed* (codes, scales, zero-points and the outliers)."""
    _struct = gwq_packed

    @property
    def N(self): return self._h.contents.N
    @property
    def K(self): return self._h.contents.K
    @property
    def bits(self): return self._h.contents.bits
    @property
    def group(self): return self._h.contents.group
    @property
    def nnz(self): return self._h.contents.S.contents.nnz

    def arrays(self):
        """dict of tensors copied out of the packed object (for inspection and parity)."""
        return _load_ext().packed_arrays(self._addr, self.device.index)

    def packed_bytes(self) -> int:
        """Bytes of codes + scales + zero-points + CSR as stored by the ABI-visible format."""
        c = self._h.contents
        nnz = c.S.contents.nnz
        return (c.N * (c.K // 32) * c.bits * 4 + c.N * (c.K // c.group) * 3 + (c.N + 1) * 4 + nnz * 6)


def _require_cuda(t: torch.Tensor, name: str):
    if not t.is_cuda:
        raise ValueError(f"{name} must be a CUDA tensor (no CPU path exists)")
    if not t.is_contiguous():
        raise ValueError(f"{name} must be contiguous")


def gwq_select_outliers(W: torch.Tensor, G: torch.Tensor, frac: float) -> Outliers:
    """W fp16 [N,K], G fp32 [N,K] on the GPU -> CSR of the ceil(frac*N*K) largest-|G| weights."""
    return Outliers(_load_ext().select(W, G, frac), W.device)


def gwq_select_outliers_static(W: torch.Tensor, G: torch.Tensor, frac: float, row_ptr: torch.Tensor,
                               col_idx: torch.Tensor, val: torch.Tensor) -> int:
    """Selection into caller-owned device tensors (row_ptr int32 [N+1], col_idx int32 [cap],
    val int16 [cap]) without any device allocation inside the library; returns nnz.
    For processes whose device memory is fully owned by their own pool, or that may not
    take the stall of a cudaMalloc.  Calls must not overlap on one GPU; N <= 32768."""
    lib = load_library()
    for t, name in ((W, "W"), (G, "G"), (row_ptr, "row_ptr"), (col_idx, "col_idx"), (val, "val")):
        _require_cuda(t, name)
    N, K = W.shape
    if row_ptr.dtype != torch.int32 or col_idx.dtype != torch.int32 or val.element_size() != 2:
        raise ValueError("row_ptr / col_idx must be int32 and val 16-bit")
    if row_ptr.numel() < N + 1:
        raise ValueError("row_ptr too short")
    cap = min(col_idx.numel(), val.numel())
    nnz = C.c_int64(0)
    with torch.cuda.device(W.device):
        st = lib.gwq_select_outliers_static(W.data_ptr(), G.data_ptr(), N, K, float(frac), row_ptr.data_ptr(),
                                            col_idx.data_ptr(), val.data_ptr(), cap, C.byref(nnz), _stream_ptr())
    _check(st, "gwq_select_outliers_static")
    return int(nnz.value)


def gwq_outliers_rows(S: Outliers, row0: int, row1: int) -> Outliers:
    """Rows [row0, row1) of S as an outlier matrix of its own (for a layer whose rows are split over ranks)."""
    out = C.POINTER(gwq_outliers)()
    with torch.cuda.device(S.device):
        st = load_library().gwq_outliers_rows(S._h, int(row0), int(row1), C.byref(out), _stream_ptr())
    _check(st, "gwq_outliers_rows")
    return Outliers(out, S.device)


def gwq_pack(W: torch.Tensor, S: Outliers, bits: int, group: int) -> Packed:
    """Quantize the non-outliers of W and pack; S is consumed (owned by the result)."""
    P = Packed(_load_ext().pack(W, S._addr, bits, group), W.device)
    S._addr = 0  # ownership moved
    return P


def gwq_linear(P: Packed, x: torch.Tensor, out_dtype: torch.dtype | None = None,
               out: torch.Tensor | None = None, workspace: torch.Tensor | None = None) -> torch.Tensor:
    """y = x (deq(Wq) + S)^T for x [M,K] fp16/bf16 on the GPU; asynchronous on the current stream.
    Where the product needs scratch memory (gwq_linear_workspace_bytes > 0) it is taken from `workspace`
    (a CUDA uint8 tensor) or, by default, from a new torch tensor: the library itself never allocates here, and calls
    on one layer share nothing."""
    return (_ext or _load_ext()).linear(P._addr, x, out_dtype, out, workspace)


def gwq_linear_multi(Ps, x: torch.Tensor, out_dtype: torch.dtype | None = None, outs=None,
                     workspace: torch.Tensor | None = None):
    """[x (deq(P) + S_P)^T for P in Ps] for layers that read the same x [M,K]: one call, and for M <= 32 one launch."""
    addrs = [P._addr for P in Ps]
    if outs is None:
        return (_ext or _load_ext()).linear_multi(addrs, x, out_dtype, None, workspace)
    (_ext or _load_ext()).linear_multi(addrs, x, out_dtype, list(outs), workspace)
    return outs


def gwq_gradient_mean(Gs, out: torch.Tensor | None = None) -> torch.Tensor:
    """FP32 mean of the gradients of several calibration samples (same shape, on the GPU), added in list order."""
    return _load_ext().gradient_mean(list(Gs), out)


def gwq_quality(W: torch.Tensor, G: torch.Tensor, P: Packed):
    """(||W - W_Q||^2, g^T (W - W_Q)) of the packed layer P against W fp16 [N,K] and G fp32 [N,K] on the GPU."""
    return _load_ext().quality(W, G, P._addr, P.device.index)


def gwq_linear_host(P: Packed, x_host: torch.Tensor, y_host: torch.Tensor) -> torch.Tensor:
    """Same product with HOST tensors (ideally pinned); copies in, computes, copies out, synchronises."""
    return (_ext or _load_ext()).linear_host(P._addr, P.device.index, x_host, y_host, False)


def gwq_linear_host_async(P: Packed, x_host: torch.Tensor, y_host: torch.Tensor) -> torch.Tensor:
    """gwq_linear_host without the synchronisation: y_host is valid after the current stream has been synchronised."""
    return (_ext or _load_ext()).linear_host(P._addr, P.device.index, x_host, y_host, True)


def gwq_device_status(P: Packed) -> int:
    """Status recorded by the kernels of earlier gwq_linear calls on P (0 = ok); synchronises."""
    with torch.cuda.device(P.device):
        return int(load_library().gwq_device_status(P._h, _stream_ptr()))


def gwq_set_wait_limit(P: Packed, cycles: int) -> None:
    """SM cycles a bounded device-side wait may spin before the kernel gives up (negative: the default)."""
    _check(int(load_library().gwq_set_wait_limit(P._h, int(cycles))), "gwq_set_wait_limit")


def gwq_free(obj) -> None:
    obj.free()


def gwq_trim_memory(keep_bytes: int = 0, device=None) -> None:
    """Give memory that the library keeps for its next objects (at most 256 MB a device) back to the system."""
    with torch.cuda.device(device):
        _check(int(load_library().gwq_trim_memory(int(keep_bytes))), "gwq_trim_memory")
