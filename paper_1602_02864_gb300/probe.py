"""ctypes binding of libspmm_probe.so (paper_1602_02864_gb300/diag/spmm_probe.h):
the gather-rate diagnostics the benchmark reports beside the SpMM, and the
eigensolvers' FP64 products by themselves.  They are not part of the library's
interface."""
from __future__ import annotations

import ctypes
import os

from . import spmm as _sp

LIB_PATH = os.path.join(os.path.dirname(os.path.abspath(__file__)), "libspmm_probe.so")
if not os.path.exists(LIB_PATH):
    raise ImportError(f"{LIB_PATH} is not built; run `python -c 'import __graft_entry__ as g; g.build()'`")
_lib = ctypes.CDLL(LIB_PATH)
_P, _i32, _i64 = ctypes.c_void_p, ctypes.c_int32, ctypes.c_int64
_dp = ctypes.POINTER(ctypes.c_double)
_lib.spmm_probe_gather.argtypes = [_i64, _i32, _dp, _dp, _P]
_lib.spmm_probe_gather.restype = ctypes.c_int
_lib.spmm_probe_gather_cols.argtypes = [_P, _i32, _i32, _dp, _dp, _P]
_lib.spmm_probe_gather_cols.restype = ctypes.c_int
_lib.spmm_probe_stream_bytes.argtypes = [_P, ctypes.POINTER(_i64)]
_lib.spmm_probe_stream_bytes.restype = ctypes.c_int
_lib.spmm_probe_ts_tn.argtypes = [_P, _i64, _i32, _P, _i64, _i32, _i64, _P, _P]
_lib.spmm_probe_ts_tn.restype = ctypes.c_int
_lib.spmm_probe_ts_nn.argtypes = [_P, _i64, _i32, _P, _i32, _P, _i64, _i64, ctypes.c_double, ctypes.c_double, _P]
_lib.spmm_probe_ts_nn.restype = ctypes.c_int
_lib.spmm_probe_chol_inv.argtypes = [_P, _i32, _P, _P, _P]
_lib.spmm_probe_chol_inv.restype = ctypes.c_int


def spmm_probe_gather(table_bytes, row_bytes, stream=None):
    """(rows/s, bytes/s) of uniformly random row gathers from a table."""
    r, b = ctypes.c_double(0), ctypes.c_double(0)
    _sp._check(_lib.spmm_probe_gather(int(table_bytes), int(row_bytes), ctypes.byref(r), ctypes.byref(b),
                                      _sp._stream_handle(stream)))
    return r.value, b.value


def spmm_probe_gather_cols(h, transpose, row_bytes, stream=None):
    """(rows/s, bytes/s) of gathering one table row per stored entry of the
    handle's column-index stream."""
    r, b = ctypes.c_double(0), ctypes.c_double(0)
    _sp._check(_lib.spmm_probe_gather_cols(h, int(bool(transpose)), int(row_bytes), ctypes.byref(r),
                                           ctypes.byref(b), _sp._stream_handle(stream)))
    return r.value, b.value


def spmm_probe_stream_bytes(h):
    """Bytes of A that each product of a streaming handle copies (0: resident)."""
    n = _i64(0)
    _sp._check(_lib.spmm_probe_stream_bytes(h, ctypes.byref(n)))
    return n.value


def spmm_probe_ts_tn(A, B, C, stream=None):
    """C = A^T B for float64 CUDA tensors (row-major, any row stride; C contiguous)."""
    _sp._check(_lib.spmm_probe_ts_tn(_sp._ptr(A), A.stride(0), A.shape[1], _sp._ptr(B), B.stride(0), B.shape[1],
                                     A.shape[0], _sp._ptr(C), _sp._stream_handle(stream)))
    return C


def spmm_probe_ts_nn(A, C, Out, alpha, beta, stream=None):
    """Out = beta Out + alpha A C for float64 CUDA tensors (C contiguous)."""
    _sp._check(_lib.spmm_probe_ts_nn(_sp._ptr(A), A.stride(0), A.shape[1], _sp._ptr(C), C.shape[1], _sp._ptr(Out),
                                     Out.stride(0), A.shape[0], float(alpha), float(beta),
                                     _sp._stream_handle(stream)))
    return Out


def spmm_probe_chol_inv(G, Rinv, flag, stream=None):
    """Rinv = R^-1 of G = R^T R (float64 CUDA tensors, b x b); flag: an int32 CUDA tensor."""
    _sp._check(_lib.spmm_probe_chol_inv(_sp._ptr(G), G.shape[0], _sp._ptr(Rinv), _sp._ptr(flag),
                                        _sp._stream_handle(stream)))
    return Rinv
