"""Python binding of include/tq.h.  Argument marshalling only: the calls a program makes again and again go through the
extension module _tqbind (csrc/tq_bind.cpp), set-up and size queries through ctypes."""
from __future__ import annotations

import ctypes
import os

import numpy as np
import torch

TQ_MSE, TQ_PROD = 0, 1
TQ_F32, TQ_BF16 = 0, 1
TQ_ORTHOGONAL, TQ_GAUSSIAN = 0, 1
TQ_LAYOUT_CANONICAL, TQ_LAYOUT_NIBBLE = 0, 1
TQ_OP_QUANTIZE, TQ_OP_SCORE, TQ_OP_TOPK, TQ_OP_WSUM, TQ_OP_DEQUANTIZE = 0, 1, 2, 3, 4
TQ_STATIC_SCRATCH_BYTES = 1 << 20

# TQ_LIB_VARIANT=debug loads libtq_debug.so, the build with device-side index checks (build.py --debug)
_LIB_PATH = os.path.join(os.path.dirname(os.path.abspath(__file__)),
                         "libtq_debug.so" if os.environ.get("TQ_LIB_VARIANT") == "debug" else "libtq.so")
_lib = None
_n = None        # the _tqbind module, bound to the loaded library

c_void_p, c_int, c_int64, c_size_t, c_u64 = ctypes.c_void_p, ctypes.c_int, ctypes.c_int64, ctypes.c_size_t, ctypes.c_uint64
_F = ctypes.POINTER(ctypes.c_float)

_SIGNATURES = {
    "tq_last_error": (ctypes.c_char_p, []),
    "tq_launch_count": (c_u64, []),
    "tq_codebook": (c_int, [c_int, c_int, _F, _F]),
    "tq_rotation": (c_int, [c_int, c_u64, c_int, _F]),
    "tq_idx_row_bytes": (c_size_t, [c_int, c_int]),
    "tq_qjl_row_bytes": (c_size_t, [c_int]),
    "tq_plan_create": (c_int, [c_int, c_int, c_int, _F, _F, _F, ctypes.POINTER(c_void_p)]),
    "tq_plan_destroy": (c_int, [c_void_p]),
    "tq_plan_status": (c_int, [c_void_p]),
    "tq_plan_set_layout": (c_int, [c_void_p, c_int]),
    "tq_plan_layout": (c_int, [c_void_p]),
    "tq_convert_layout": (c_int, [c_void_p, c_int64, c_void_p, c_void_p, c_int, c_int, c_void_p]),
    "tq_workspace_bytes": (c_size_t, [c_void_p, c_int, c_int64, c_int, c_int]),
    "tq_quantize_mse": (c_int, [c_void_p, c_void_p, c_int, c_int64, c_int64, c_void_p, c_void_p, c_void_p, c_size_t, c_void_p]),
    "tq_quantize_prod": (c_int, [c_void_p, c_void_p, c_int, c_int64, c_int64, c_void_p, c_void_p, c_void_p, c_void_p,
                                 c_void_p, c_size_t, c_void_p]),
    "tq_dequantize": (c_int, [c_void_p, c_int64, c_void_p, c_void_p, c_void_p, c_void_p, c_void_p, c_int64, c_void_p]),
    "tq_score": (c_int, [c_void_p, c_void_p, c_int, c_int, c_int64, c_int64, c_void_p, c_void_p, c_void_p, c_void_p,
                         c_void_p, c_int64, c_void_p, c_size_t, c_void_p]),
    "tq_score_static": (c_int, [c_void_p, c_void_p, c_int, c_int, c_int64, c_int64, c_void_p, c_void_p, c_void_p, c_void_p,
                                c_void_p, c_int64, c_void_p]),
    "tq_score_static_max_queries": (c_int, [c_void_p]),
    "tq_query_bytes": (c_size_t, [c_void_p, c_int]),
    "tq_query_prepare": (c_int, [c_void_p, c_void_p, c_int, c_int, c_int64, c_void_p, c_size_t, c_void_p]),
    "tq_score_prepared": (c_int, [c_void_p, c_void_p, c_int, c_int64, c_void_p, c_void_p, c_void_p, c_void_p, c_void_p,
                                  c_int64, c_void_p]),
    "tq_selftest_wait_timeout": (c_int, [c_void_p, ctypes.c_longlong, c_void_p]),
    "tq_entropy_lengths": (c_int, [c_int, c_int, _F, c_void_p]),
    "tq_entropy_workspace_bytes": (c_size_t, [c_int64]),
    "tq_entropy_measure": (c_int, [c_void_p, c_void_p, c_int64, c_void_p, c_void_p, c_void_p, c_size_t, c_void_p]),
    "tq_entropy_pack": (c_int, [c_void_p, c_void_p, c_int64, c_void_p, c_void_p, c_void_p, c_size_t, c_void_p]),
    "tq_entropy_unpack": (c_int, [c_void_p, c_void_p, c_int64, c_void_p, c_void_p, c_void_p, c_void_p]),
    "tq_topk": (c_int, [c_void_p, c_void_p, c_int, c_int, c_int64, c_int64, c_void_p, c_void_p, c_void_p, c_void_p,
                        c_int, c_void_p, c_void_p, c_void_p, c_size_t, c_void_p]),
    "tq_select_topk": (c_int, [c_void_p, c_void_p, c_int, c_int64, c_int64, c_int, c_void_p, c_void_p, c_void_p]),
    "tq_softmax": (c_int, [c_void_p, c_void_p, c_int, c_int64, c_int64, ctypes.c_float, c_void_p, c_int64, c_void_p]),
    "tq_wsum": (c_int, [c_void_p, c_void_p, c_int, c_int64, c_int64, c_void_p, c_void_p, c_void_p, c_void_p,
                        c_void_p, c_int64, c_void_p, c_size_t, c_void_p]),
    "tq_attend_decode_workspace_bytes": (c_size_t, [c_int, c_int, c_int64, c_int]),
    "tq_attend_decode": (c_int, [c_void_p, c_int, c_int, c_int64, c_int64, c_int, c_void_p, c_int, c_int64, ctypes.c_float,
                                 c_void_p, c_int64, c_void_p, c_size_t, c_void_p]),
    "tq_kv_append": (c_int, [c_void_p, c_int, c_int, c_int64, c_int64, c_void_p, c_void_p, c_int, c_int64, c_int64, c_void_p]),
}


class KvGroup(ctypes.Structure):
    """struct tq_kv_group of include/tq.h (one channel group of a compressed KV layer), for programs that call
    lib().tq_attend_decode / tq_kv_append themselves; the functions below take mappings."""
    _fields_ = [(name, c_void_p) for name in ("plan_k", "plan_v", "k_idx", "k_qjl", "k_gamma", "k_norms", "v_idx", "v_norms",
                                              "k_channels", "v_channels")]


class TqError(RuntimeError):
    def __init__(self, code: int, message: str):
        super().__init__(f"tq error {code}: {message}")
        self.code = code


def lib() -> ctypes.CDLL:
    """Loads libtq.so (built in-tree by paper_2504_19874_b200/build.py).  Raises if it is missing."""
    global _lib
    if _lib is None:
        if not os.path.exists(_LIB_PATH):
            raise RuntimeError(f"{_LIB_PATH} is missing: run `python -m paper_2504_19874_b200.build` first "
                               "(there is no fallback path)")
        handle = ctypes.CDLL(_LIB_PATH)
        for name, (res, args) in _SIGNATURES.items():
            fn = getattr(handle, name)
            fn.restype, fn.argtypes = res, args
        _lib = handle
    return _lib


def _native():
    """The marshalling module, bound to the library that lib() loads."""
    global _n
    if _n is None:
        lib()
        try:
            from . import _tqbind
        except ImportError as e:
            raise RuntimeError("_tqbind.so is missing or does not load: run `python -m paper_2504_19874_b200.build` first "
                               f"(there is no fallback path): {e}") from e
        _tqbind.bind(_LIB_PATH)
        _n = _tqbind
    return _n


def _check(code: int):
    if code != 0:
        raise TqError(code, lib().tq_last_error().decode())


def _fptr(a: np.ndarray):
    return a.ctypes.data_as(_F)


def _dev(t):
    """Device pointer of a CUDA tensor (None -> NULL)."""
    if t is None:
        return None
    if not t.is_cuda:
        raise ValueError("expected a CUDA tensor (this library has no CPU path)")
    return t.data_ptr()


def _stream():
    return torch.cuda.current_stream().cuda_stream


def tq_launch_count() -> int:
    return lib().tq_launch_count()


def tq_idx_row_bytes(d: int, bits: int) -> int:
    return lib().tq_idx_row_bytes(d, bits)


def tq_qjl_row_bytes(d: int) -> int:
    return lib().tq_qjl_row_bytes(d)


def tq_codebook(d: int, bits: int):
    """(centroids, boundaries) as float32 numpy arrays."""
    levels = 1 << min(max(bits, 0), 8)        # the library rejects bits outside 0..4
    c = np.zeros(levels, dtype=np.float32)
    t = np.zeros(max(levels - 1, 1), dtype=np.float32)
    _check(lib().tq_codebook(d, bits, _fptr(c), _fptr(t)))
    return c, t[:levels - 1]


def tq_rotation(d: int, seed: int, kind: int = TQ_ORTHOGONAL) -> np.ndarray:
    out = np.zeros((d, d), dtype=np.float32)
    _check(lib().tq_rotation(d, seed, kind, _fptr(out)))
    return out


class Plan:
    """Owner of a tq_plan handle (device copies of Pi, S', codebook for one (d, b, mode))."""

    def __init__(self, d: int, bits: int, mode: int, Pi, S, centroids):
        Pi = np.ascontiguousarray(Pi, dtype=np.float32)
        cent = np.ascontiguousarray(centroids, dtype=np.float32)
        Sp = None if S is None else np.ascontiguousarray(S, dtype=np.float32)
        if Pi.shape != (d, d) or (Sp is not None and Sp.shape != (d, d)):
            raise ValueError("Pi and S must be d x d")
        self.d, self.bits, self.mode = d, bits, mode
        self.mse_bits = bits - 1 if mode == TQ_PROD else bits
        if cent.size != (1 << max(self.mse_bits, 0)):
            raise ValueError("centroids must hold 2^b_m values")
        self.idx_row_bytes = tq_idx_row_bytes(d, self.mse_bits)
        self.qjl_row_bytes = tq_qjl_row_bytes(d)
        h = c_void_p()
        _check(lib().tq_plan_create(d, bits, mode, _fptr(Pi), None if Sp is None else _fptr(Sp), _fptr(cent),
                                    ctypes.byref(h)))
        self.handle = h.value

    def set_layout(self, layout: int) -> None:
        """TQ_LAYOUT_CANONICAL or TQ_LAYOUT_NIBBLE (TQ_PROD with b = 4 only): arrangement of the code rows."""
        _check(lib().tq_plan_set_layout(self.handle, layout))

    @property
    def layout(self) -> int:
        return lib().tq_plan_layout(self.handle)

    def close(self):
        if getattr(self, "handle", None):
            lib().tq_plan_destroy(self.handle)
            self.handle = None

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass


def tq_plan_status(plan: Plan) -> None:
    """Synchronises and raises TqError(6) if a kernel of this plan gave up a bounded wait."""
    _check(lib().tq_plan_status(plan.handle))


def tq_convert_layout(plan: Plan, n: int, idx, qjl, src: int, dst: int) -> None:
    """Rewrites n rows of (idx, qjl) in place from layout `src` into layout `dst`."""
    _check(lib().tq_convert_layout(plan.handle, n, _dev(idx), _dev(qjl), src, dst, _stream()))


def tq_workspace_bytes(plan: Plan, op: int, n: int, nq: int = 0, k: int = 0) -> int:
    return lib().tq_workspace_bytes(plan.handle, op, n, nq, k)


def tq_quantize_mse(plan: Plan, X, idx, norms=None, scratch=None):
    _check((_n or _native()).quantize_mse(plan.handle, X, idx, norms, scratch))


def tq_quantize_prod(plan: Plan, X, idx, qjl, gamma, norms=None, scratch=None):
    _check((_n or _native()).quantize_prod(plan.handle, X, idx, qjl, gamma, norms, scratch))


def tq_dequantize(plan: Plan, n: int, idx, qjl, gamma, norms, Xhat):
    _check((_n or _native()).dequantize(plan.handle, n, idx, qjl, gamma, norms, Xhat))


def tq_score(plan: Plan, Q, n: int, idx, qjl, gamma, norms, scores, workspace):
    _check((_n or _native()).score(plan.handle, Q, n, idx, qjl, gamma, norms, scores, workspace))


def tq_score_static(plan: Plan, Q, n: int, idx, qjl, gamma, norms, scores):
    """tq_score for callers that cannot allocate device memory: the rotated-query workspace is an
    array built into the library (TQ_STATIC_SCRATCH_BYTES), shared by every call on the device."""
    _check((_n or _native()).score_static(plan.handle, Q, n, idx, qjl, gamma, norms, scores))


def tq_score_static_max_queries(plan: Plan) -> int:
    return lib().tq_score_static_max_queries(plan.handle)


def tq_query_bytes(plan: Plan, nq: int) -> int:
    return lib().tq_query_bytes(plan.handle, nq)


def tq_query_prepare(plan: Plan, Q, prepared):
    """Query-side work of tq_score (rotations, scan operand) into `prepared` (>= tq_query_bytes(plan, nq) bytes)."""
    _check((_n or _native()).query_prepare(plan.handle, Q, prepared))


def tq_score_prepared(plan: Plan, prepared, nq: int, n: int, idx, qjl, gamma, norms, scores):
    _check((_n or _native()).score_prepared(plan.handle, prepared, nq, n, idx, qjl, gamma, norms, scores))


def tq_selftest_wait_timeout(plan: Plan, limit_cycles: int = 20000) -> None:
    """Enqueues the library's bounded-wait self test; the next tq_plan_status(plan) must raise TqError(6)."""
    _check(lib().tq_selftest_wait_timeout(plan.handle, limit_cycles, _stream()))


def tq_topk(plan: Plan, Q, n: int, idx, qjl, gamma, norms, k: int, top_scores, top_ids, workspace):
    _check((_n or _native()).topk(plan.handle, Q, n, idx, qjl, gamma, norms, k, top_scores, top_ids, workspace))


def tq_wsum(plan: Plan, W, n: int, idx, qjl, gamma, norms, out, workspace):
    _check((_n or _native()).wsum(plan.handle, W, n, idx, qjl, gamma, norms, out, workspace))


def tq_softmax(s1, s2, scale: float, W):
    _check((_n or _native()).softmax(s1, s2, scale, W))


def tq_attend_decode_workspace_bytes(ngroups: int, heads: int, tokens: int, d: int) -> int:
    return lib().tq_attend_decode_workspace_bytes(ngroups, heads, tokens, d)


def tq_attend_decode(groups, heads: int, tokens: int, q_per_kv: int, Q, scale: float, out, workspace, head_stride=None):
    """groups: sequence of dicts with keys plan_k, plan_v (Plan) and k_idx, k_qjl, k_gamma, k_norms, v_idx,
    v_norms, k_channels, v_channels (CUDA tensors or None); rows of all heads head-major, head_stride rows
    per head (default: tokens)."""
    _check((_n or _native()).attend_decode(groups, heads, tokens, tokens if head_stride is None else head_stride, q_per_kv, Q, scale,
                                           out, workspace))


def tq_kv_append(groups, heads: int, head_stride: int, position: int, K, V):
    """Quantises one new token per KV head (K, V: [heads, head_dim]) into row `position` of every head."""
    _check((_n or _native()).kv_append(groups, heads, head_stride, position, K, V))


def tq_entropy_lengths(d: int, bits: int, centroids) -> np.ndarray:
    """Huffman code lengths of the 2^bits index values for the given codebook (uint8 array)."""
    cent = np.ascontiguousarray(centroids, dtype=np.float32)
    out = np.zeros(1 << bits, dtype=np.uint8)
    _check(lib().tq_entropy_lengths(d, bits, _fptr(cent), out.ctypes.data_as(c_void_p)))
    return out


def tq_entropy_pack(plan: Plan, lengths, n: int, idx):
    """(packed uint8 tensor, row_offsets int64 tensor of n + 1 byte offsets): the entropy-coded index rows."""
    ln = np.ascontiguousarray(lengths, dtype=np.uint8)
    got = (_n or _native()).entropy_pack(plan.handle, ln.ctypes.data, n, idx)
    if not isinstance(got, tuple):
        _check(got)
    return got


def tq_entropy_unpack(plan: Plan, lengths, n: int, packed, offsets, idx_out):
    ln = np.ascontiguousarray(lengths, dtype=np.uint8)
    _check((_n or _native()).entropy_unpack(plan.handle, ln.ctypes.data, n, packed, offsets, idx_out))


def tq_select_topk(cand_scores, cand_ids, k: int, top_scores, top_ids):
    _check((_n or _native()).select_topk(cand_scores, cand_ids, k, top_scores, top_ids))
