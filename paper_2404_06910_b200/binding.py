"""ctypes binding of libsp_b200.so (declared in include/sp.h).

Argument marshalling only: every function forwards raw device pointers and sizes to the
C ABI entry point of the same name.  torch is used for device memory and streams.
There is no fallback: if the CUDA library is missing, importing this module raises.
"""
from __future__ import annotations

import ctypes
import os
from dataclasses import dataclass

import numpy as np
import torch

from . import _marshal

_HERE = os.path.dirname(os.path.abspath(__file__))
# SP_B200_DEBUG_BOUNDS=1 selects the twin built with -DSP_DEBUG_BOUNDS (extra device-side layout checks)
LIB_PATH = os.path.join(_HERE, "libsp_b200_debug.so" if os.environ.get("SP_B200_DEBUG_BOUNDS") == "1" else "libsp_b200.so")

SP_OK = 0
SP_ERR_INVALID_ARG, SP_ERR_UNSUPPORTED, SP_ERR_WORKSPACE, SP_ERR_CUDA, SP_ERR_TIMEOUT, SP_ERR_LAYOUT = 1, 2, 3, 4, 5, 6
SP_F32, SP_BF16 = 0, 1
SP_ROWS_ALL, SP_ROWS_QUERY_ONLY = 0, 1
SP_POS_EQUILIBRIUM, SP_POS_LEFT_ALIGNED = 0, 1
SP_ROPE_HALF_SPLIT, SP_ROPE_INTERLEAVED = 0, 1

EXPORTS = (
    "sp_last_error", "sp_version", "sp_positions", "sp_rope_apply",
    "sp_prefill_workspace_bytes", "sp_superpose_prefill",
    "sp_path_scores_workspace_bytes", "sp_path_scores", "sp_prune_topk",
    "sp_decode_workspace_bytes", "sp_pruned_decode", "sp_check_status",
    "sp_pruned_decode_static_max_bytes", "sp_pruned_decode_static",
    "sp_superpose_prefill_alibi", "sp_pruned_decode_alibi", "sp_rope_apply_pair", "sp_pruned_decode_rope",
    "sp_prefill_rope_workspace_bytes", "sp_superpose_prefill_rope",
)


class SpError(RuntimeError):
    def __init__(self, code: int, message: str):
        super().__init__(f"sp status {code}: {message}")
        self.code = code


class _CLayoutHost(ctypes.Structure):
    _fields_ = [(n, ctypes.c_void_p) for n in ("prompt_path_off", "pre_start", "pre_len", "path_start", "doc_len", "qry_len")]


class _CLayout(ctypes.Structure):
    _fields_ = [
        ("n_prompts", ctypes.c_int32), ("n_paths", ctypes.c_int32),
        ("prompt_path_off", ctypes.c_void_p), ("pre_start", ctypes.c_void_p),
        ("pre_len", ctypes.c_void_p), ("path_start", ctypes.c_void_p),
        ("doc_len", ctypes.c_void_p), ("qry_len", ctypes.c_void_p),
        ("total_tokens", ctypes.c_int64),
        ("max_pre_len", ctypes.c_int32), ("max_path_len", ctypes.c_int32),
        ("host_mirror", ctypes.POINTER(_CLayoutHost)),
    ]


def _load() -> ctypes.CDLL:
    if not os.path.exists(LIB_PATH):
        raise ImportError(
            f"{LIB_PATH} is missing: build it with `python -m paper_2404_06910_b200.build` "
            "(there is no CPU or PyTorch fallback)")
    lib = ctypes.CDLL(LIB_PATH)
    c_int, c_i64, c_f, c_d, vp, sz = (ctypes.c_int, ctypes.c_int64, ctypes.c_float, ctypes.c_double,
                                      ctypes.c_void_p, ctypes.c_size_t)
    lp = ctypes.POINTER(_CLayout)
    lib.sp_last_error.restype = ctypes.c_char_p
    lib.sp_version.restype = ctypes.c_char_p
    lib.sp_positions.argtypes = [c_int, c_int, c_int, c_int, vp, c_int, vp, ctypes.POINTER(c_d), ctypes.POINTER(c_d)]
    lib.sp_rope_apply.argtypes = [vp, vp, c_i64, c_i64, c_int, c_int, c_int, c_d, c_int, c_int, vp]
    lib.sp_rope_apply_pair.argtypes = [vp, c_i64, c_int, vp, c_i64, c_int, vp, c_i64, c_int, c_int, c_d, c_int, c_int, vp]
    lib.sp_prefill_workspace_bytes.argtypes = [c_int] * 7
    lib.sp_prefill_workspace_bytes.restype = sz
    lib.sp_superpose_prefill.argtypes = [vp, vp, vp, lp, c_int, c_int, c_int, c_f, c_int, vp, vp, vp, sz, c_int, vp]
    lib.sp_prefill_rope_workspace_bytes.argtypes = [c_int, c_int, c_int, c_int, c_i64, c_int, c_int, c_int]
    lib.sp_prefill_rope_workspace_bytes.restype = sz
    lib.sp_superpose_prefill_rope.argtypes = [vp, vp, vp, lp, vp, c_d, c_int, c_int, c_int, c_int, c_f, vp, vp, vp, sz,
                                              c_int, vp]
    lib.sp_path_scores_workspace_bytes.argtypes = [c_i64]
    lib.sp_path_scores_workspace_bytes.restype = sz
    lib.sp_path_scores.argtypes = [vp, c_i64, vp, vp, c_i64, c_int, c_int, vp, vp, vp, vp, vp, sz, c_int, vp]
    lib.sp_prune_topk.argtypes = [vp, vp, c_int, c_int, vp, vp, vp]
    lib.sp_decode_workspace_bytes.argtypes = [c_int, c_int, c_int]
    lib.sp_decode_workspace_bytes.restype = sz
    lib.sp_pruned_decode.argtypes = [vp, vp, vp, lp, vp, c_int, vp, vp, vp, c_int, c_i64, c_int, c_int, c_int,
                                     c_f, vp, vp, vp, sz, c_int, vp]
    lib.sp_check_status.argtypes = [vp, vp]
    lib.sp_pruned_decode_static_max_bytes.restype = sz
    lib.sp_pruned_decode_static.argtypes = [vp, vp, vp, lp, vp, c_int, vp, vp, vp, c_int, c_i64, c_int, c_int, c_int,
                                            c_f, vp, vp, c_int, vp]
    lib.sp_superpose_prefill_alibi.argtypes = [vp, vp, vp, lp, vp, vp, c_int, c_int, c_int, c_f, c_int, vp, vp, vp, sz,
                                               c_int, vp]
    lib.sp_pruned_decode_alibi.argtypes = [vp, vp, vp, lp, vp, c_int, vp, vp, vp, c_int, c_i64, vp, vp, vp, vp, c_int,
                                           c_int, c_int, c_f, vp, vp, vp, sz, c_int, vp]
    lib.sp_pruned_decode_rope.argtypes = [vp, vp, vp, lp, vp, c_int, vp, vp, vp, c_int, c_i64, vp, c_d, c_int, c_int,
                                          c_int, c_int, c_f, vp, vp, c_int, vp]
    for name in EXPORTS:
        getattr(lib, name)          # raises AttributeError if a declared symbol is not exported
    return lib


lib = _load()

# The launching entry points go through the native marshalling module: its case number (the order here) and the kind of every
# argument, t / r contiguous / strided tensor or None, a address, i integer, d floating point.
_KINDS = (
    ("sp_rope_apply", "rriiiiidiia"),
    ("sp_rope_apply_pair", "riiriiriiidiia"),
    ("sp_superpose_prefill", "tttaiiidittti" "ia"),
    ("sp_superpose_prefill_alibi", "tttattiiidittti" "ia"),
    ("sp_superpose_prefill_rope", "tttatdiiiidttti" "ia"),
    ("sp_path_scores", "rittiiitttttiia"),
    ("sp_prune_topk", "ttiitta"),
    ("sp_pruned_decode", "tttatitttiiiiidttti" "ia"),
    ("sp_pruned_decode_alibi", "tttatitttiittttiiidttti" "ia"),
    ("sp_pruned_decode_rope", "tttatitttiitdiiiidttia"),
    ("sp_pruned_decode_static", "tttatitttiiiiidttia"),
)
for _i, (_name, _kinds) in enumerate(_KINDS):
    _marshal.bind(_i, ctypes.cast(getattr(lib, _name), ctypes.c_void_p).value, _kinds)
(_ROPE, _ROPE_PAIR, _PREFILL, _PREFILL_ALIBI, _PREFILL_ROPE, _SCORES, _TOPK, _DECODE, _DECODE_ALIBI, _DECODE_ROPE,
 _DECODE_STATIC) = range(len(_KINDS))


def _check(rc: int):
    if rc != SP_OK:
        raise SpError(rc, lib.sp_last_error().decode())


def _call(*args):
    rc = _marshal.call(*args)
    if rc:
        raise SpError(rc, lib.sp_last_error().decode())


_DTYPE_CODES = {torch.float32: SP_F32, torch.bfloat16: SP_BF16}


def dtype_code(t: torch.Tensor) -> int:
    code = _DTYPE_CODES.get(t.dtype)
    if code is None:
        raise TypeError(f"unsupported dtype {t.dtype}")
    return code


def _ptr(t):
    if t is None:
        return None
    assert t.is_contiguous(), "tensors must be contiguous"
    return t.data_ptr()


def _nbytes(t):
    return 0 if t is None else t.nbytes


def _stream(stream=None):
    if stream is not None:
        return stream.cuda_stream
    # the current stream's handle without a Stream object around it (1.5 us of every call)
    return torch._C._cuda_getCurrentRawStream(torch._C._cuda_getDevice())


@dataclass
class DeviceLayout:
    """sp_layout with its index arrays resident on the device."""
    c: _CLayout
    arrays: tuple          # keeps the device tensors alive
    n_prompts: int
    n_paths: int
    total_tokens: int
    max_pre_len: int
    max_path_len: int

    @property
    def prompt_path_off(self):
        return self.arrays[0]

    @staticmethod
    def from_host(lay, device="cuda", mirror: bool = True) -> "DeviceLayout":
        """mirror: also hand the host copies of the index arrays to the library, which then
        validates the whole layout on the host in every call."""
        host = tuple(np.ascontiguousarray(a, dtype=np.int32) for a in (lay.prompt_path_off, lay.pre_start, lay.pre_len,
                                                                       lay.path_start, lay.doc_len, lay.qry_len))
        arrs = tuple(torch.from_numpy(a).to(device) for a in host)
        hm = _CLayoutHost(*[a.ctypes.data for a in host]) if mirror else None
        c = _CLayout(lay.n_prompts, lay.n_paths, *[a.data_ptr() for a in arrs],
                     lay.total_tokens, lay.max_pre_len, lay.max_path_len,
                     ctypes.pointer(hm) if mirror else None)
        return DeviceLayout(c, arrs + host + (hm,), lay.n_prompts, lay.n_paths, lay.total_tokens,
                            lay.max_pre_len, lay.max_path_len)


def sp_version() -> str:
    return lib.sp_version().decode()


def sp_positions(pre_len: int, doc_lens, qry_len: int, scheme: int = SP_POS_EQUILIBRIUM, q_mode: int = 0):
    """Host call.  Returns (pos float32 [P + sum(L) + N*Q], S, next_pos)."""
    L = np.ascontiguousarray(doc_lens, dtype=np.int32)
    pos = np.empty(int(pre_len + L.sum() + len(L) * qry_len), dtype=np.float32)
    S, nxt = ctypes.c_double(), ctypes.c_double()
    _check(lib.sp_positions(scheme, q_mode, pre_len, len(L), L.ctypes.data, qry_len, pos.ctypes.data,
                            ctypes.byref(S), ctypes.byref(nxt)))
    return pos, S.value, nxt.value


def sp_rope_apply(x: torch.Tensor, pos: torch.Tensor, n_heads: int, head_dim: int, *, n_tokens=None,
                  ld_token=None, rot_dim=None, base: float = 10000.0, pairing: int = SP_ROPE_HALF_SPLIT,
                  stream=None):
    """In place on x ([n_tokens, n_heads, head_dim] with token stride ld_token elements)."""
    n = pos.numel() if n_tokens is None else n_tokens
    ld = n_heads * head_dim if ld_token is None else ld_token
    _call(_ROPE, x, pos, n, ld, n_heads, head_dim, head_dim if rot_dim is None else rot_dim, base, pairing,
          dtype_code(x), _stream(stream))


def sp_rope_apply_pair(xq: torch.Tensor, n_heads_q: int, xk: torch.Tensor, n_heads_k: int, pos: torch.Tensor,
                       head_dim: int, *, n_tokens=None, ld_q=None, ld_k=None, rot_dim=None, base: float = 10000.0,
                       pairing: int = SP_ROPE_HALF_SPLIT, stream=None):
    """sp_rope_apply on a step's queries and keys (same positions) in one launch, in place."""
    n = pos.numel() if n_tokens is None else n_tokens
    _call(_ROPE_PAIR, xq, n_heads_q * head_dim if ld_q is None else ld_q, n_heads_q, xk, n_heads_k * head_dim if
          ld_k is None else ld_k, n_heads_k, pos, n, head_dim, head_dim if rot_dim is None else rot_dim, base,
          pairing, dtype_code(xq), _stream(stream))


def sp_prefill_workspace_bytes(lay: DeviceLayout, n_heads: int, head_dim: int, dtype: int) -> int:
    return int(lib.sp_prefill_workspace_bytes(lay.n_prompts, lay.n_paths, lay.max_pre_len, lay.max_path_len,
                                              n_heads, head_dim, dtype))


def sp_superpose_prefill(q, k, v, lay: DeviceLayout, scale: float, out, lse=None, ws=None,
                         rows: int = SP_ROWS_ALL, stream=None):
    T, H, D = q.shape
    Hkv = k.shape[1]
    _call(_PREFILL, q, k, v, ctypes.addressof(lay.c), H, Hkv, D, scale, rows, out, lse, ws, _nbytes(ws),
          dtype_code(q), _stream(stream))


def sp_superpose_prefill_alibi(q, k, v, lay: DeviceLayout, pos, slopes, scale: float, out, lse=None, ws=None,
                               rows: int = SP_ROWS_ALL, stream=None):
    """sp_superpose_prefill with the ALiBi bias -slopes[h] * |pos[q] - pos[k]| (pos fp32 [T], slopes fp32 [H])."""
    T, H, D = q.shape
    Hkv = k.shape[1]
    _call(_PREFILL_ALIBI, q, k, v, ctypes.addressof(lay.c), pos, slopes, H, Hkv, D, scale, rows, out, lse, ws,
          _nbytes(ws), dtype_code(q), _stream(stream))


def sp_prefill_rope_workspace_bytes(lay: DeviceLayout, n_heads: int, head_dim: int, dtype: int) -> int:
    return int(lib.sp_prefill_rope_workspace_bytes(lay.n_prompts, lay.n_paths, lay.max_pre_len, lay.max_path_len,
                                                   lay.total_tokens, n_heads, head_dim, dtype))


def sp_superpose_prefill_rope(q, k, v, lay: DeviceLayout, pos, base: float, pairing: int, scale: float, out, lse=None,
                              ws=None, stream=None):
    """sp_superpose_prefill over all rows with the rotation of the (unrotated) q folded in; k already rotated."""
    T, H, D = q.shape
    Hkv = k.shape[1]
    _call(_PREFILL_ROPE, q, k, v, ctypes.addressof(lay.c), pos, base, pairing, H, Hkv, D, scale, out, lse, ws,
          _nbytes(ws), dtype_code(q), _stream(stream))


def sp_path_scores_workspace_bytes(n_rows: int) -> int:
    return int(lib.sp_path_scores_workspace_bytes(n_rows))


def sp_path_scores(logits, targets, row_off, scores, prior=None, weight=None, row_logp=None, ws=None,
                   stream=None):
    R, V = logits.shape
    _call(_SCORES, logits, logits.stride(0) if R else V, targets, row_off, R, row_off.numel() - 1, V, prior,
          weight, scores, row_logp, ws, _nbytes(ws), dtype_code(logits), _stream(stream))


def sp_prune_topk(scores, prompt_path_off, k: int, kept_idx, kept_post=None, stream=None):
    _call(_TOPK, scores, prompt_path_off, prompt_path_off.numel() - 1, k, kept_idx, kept_post, _stream(stream))


def sp_decode_workspace_bytes(n_prompts: int, n_heads: int, head_dim: int) -> int:
    return int(lib.sp_decode_workspace_bytes(n_prompts, n_heads, head_dim))


def sp_pruned_decode(q, k_cache, v_cache, lay: DeviceLayout, kept_idx, k: int, tail_k, tail_v, tail_len,
                     tail_cap: int, scale: float, out, lse=None, ws=None, max_keys: int = 0, stream=None):
    B, H, D = q.shape
    Hkv = k_cache.shape[1]
    _call(_DECODE, q, k_cache, v_cache, ctypes.addressof(lay.c), kept_idx, k, tail_k, tail_v, tail_len,
          tail_cap, max_keys, H, Hkv, D, scale, out, lse, ws, _nbytes(ws), dtype_code(q), _stream(stream))


def sp_pruned_decode_alibi(q, k_cache, v_cache, lay: DeviceLayout, kept_idx, k: int, tail_k, tail_v, tail_len,
                           tail_cap: int, q_pos, cache_pos, tail_pos, slopes, scale: float, out, lse=None, ws=None,
                           max_keys: int = 0, stream=None):
    """sp_pruned_decode with the ALiBi bias: q_pos fp32 [B], cache_pos fp32 [T], tail_pos fp32 [B, tail_cap],
    slopes fp32 [H]."""
    B, H, D = q.shape
    Hkv = k_cache.shape[1]
    _call(_DECODE_ALIBI, q, k_cache, v_cache, ctypes.addressof(lay.c), kept_idx, k, tail_k, tail_v, tail_len,
          tail_cap, max_keys, q_pos, cache_pos, tail_pos, slopes, H, Hkv, D, scale, out, lse, ws, _nbytes(ws),
          dtype_code(q), _stream(stream))


def sp_pruned_decode_rope(q, k_cache, v_cache, lay: DeviceLayout, kept_idx, k: int, tail_k, tail_v, tail_len,
                          tail_cap: int, q_pos, scale: float, out, lse=None, base: float = 10000.0,
                          pairing: int = SP_ROPE_HALF_SPLIT, max_keys: int = 0, stream=None):
    """One decode step with the rotary embedding folded in: q and the newest tail key row arrive
    unrotated and are rotated at q_pos (fp32 [B]); the key row is written back rotated."""
    B, H, D = q.shape
    Hkv = k_cache.shape[1]
    _call(_DECODE_ROPE, q, k_cache, v_cache, ctypes.addressof(lay.c), kept_idx, k, tail_k, tail_v, tail_len,
          tail_cap, max_keys, q_pos, base, pairing, H, Hkv, D, scale, out, lse, dtype_code(q), _stream(stream))


def sp_pruned_decode_static_max_bytes() -> int:
    return int(lib.sp_pruned_decode_static_max_bytes())


def sp_pruned_decode_static(q, k_cache, v_cache, lay: DeviceLayout, kept_idx, k: int, tail_k, tail_v, tail_len,
                            tail_cap: int, scale: float, out, lse=None, max_keys: int = 0, stream=None):
    """sp_pruned_decode for callers that cannot provide a workspace: the split-KV scratch is a
    fixed array inside the library (see include/sp.h for its limit and sharing rules)."""
    B, H, D = q.shape
    Hkv = k_cache.shape[1]
    _call(_DECODE_STATIC, q, k_cache, v_cache, ctypes.addressof(lay.c), kept_idx, k, tail_k, tail_v, tail_len,
          tail_cap, max_keys, H, Hkv, D, scale, out, lse, dtype_code(q), _stream(stream))


def sp_check_status(ws, stream=None) -> None:
    _check(lib.sp_check_status(_ptr(ws), _stream(stream)))
