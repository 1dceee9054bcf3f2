"""Binding of libtik.so: argument marshalling only.

Every operator takes torch CUDA tensors (device memory and the current
stream come from torch); the extension module built from csrc/tik_bind.cpp
checks dtypes/contiguity, makes outputs and scratch and calls the C entry
point of the same name.  All arithmetic happens in the library's kernels;
there is no fallback, and a missing library raises.
"""
from __future__ import annotations

import ctypes
import importlib.util
import os
from typing import Optional

import torch

from . import build as _build

OK = 0
OP_ATTN_TRAIN_FWD, OP_ATTN_PREFILL, OP_ATTN_DECODE, OP_TOKEN_LOGPROB, OP_ATTN_TRAIN_BWD = 0, 1, 2, 3, 4
DEV_BAD_BLOCK, DEV_BAD_TARGET, DEV_WAIT_EXPIRED, DEV_BAD_POSITION, DEV_BAD_CONTEXT = 1, 2, 4, 8, 16

_lib = None
_native = None


class TikError(RuntimeError):
    pass


def load(build_if_missing: bool = False) -> ctypes.CDLL:
    """Loads libtik.so (optionally building it first).  Raises if it is absent."""
    global _lib
    if _lib is not None:
        return _lib
    path = _build.LIB_PATH
    if build_if_missing:
        _build.build()
    if not os.path.exists(path):
        raise TikError("libtik.so is not built (%s); run `python -m paper_2609_35140_b200.build`. "
                       "There is no fallback path." % path)
    lib = ctypes.CDLL(path)
    c = ctypes
    vp, i32, i64, f32, sz = c.c_void_p, c.c_int, c.c_int64, c.c_float, c.c_size_t
    lib.tik_create.argtypes = [c.POINTER(vp), i32]
    lib.tik_destroy.argtypes = [vp]
    lib.tik_status_str.argtypes = [i32]
    lib.tik_status_str.restype = c.c_char_p
    lib.tik_last_error.argtypes = [vp]
    lib.tik_last_error.restype = c.c_char_p
    lib.tik_contract_id.restype = c.c_char_p
    lib.tik_kernel_launches.restype = c.c_ulonglong
    lib.tik_kernel_launches.argtypes = []
    lib.tik_workspace_bytes.argtypes = [i32, i64, i32, i32, i32, i64, i32, i32]
    lib.tik_workspace_bytes.restype = sz
    lib.tik_device_status.argtypes = [vp, vp, c.POINTER(i32)]
    lib.tik_attn_train_fwd.argtypes = [vp, vp, vp, vp, vp, vp, vp, i32, i64, i32, i32, i32, i32, f32, vp, sz, vp]
    lib.tik_kv_cache_write.argtypes = [vp, vp, vp, vp, vp, vp, vp, vp, i32, i32, i64, i32, i32, i32, i32, vp]
    lib.tik_attn_prefill.argtypes = [vp, vp, vp, vp, vp, vp, vp, vp, vp, i32, i32, i64, i32, i32, i32, i32,
                                     i32, i32, i32, f32, vp, sz, vp]
    lib.tik_attn_prefill_kv.argtypes = [vp, vp, vp, vp, vp, vp, vp, vp, vp, vp, vp, i32, i32, i64, i32, i32, i32, i32,
                                        i32, i32, i32, f32, vp, sz, vp]
    lib.tik_attn_prefill_kv.restype = i32
    lib.tik_attn_decode.argtypes = [vp, vp, vp, vp, vp, vp, vp, vp, i32, i32, i32, i32, i32, i32, i32, i32,
                                    f32, vp, sz, vp]
    lib.tik_qk_norm_rope_kv_write.argtypes = [vp, vp, vp, vp, vp, vp, f32, vp, i32, vp, vp, vp, vp, vp, i32, i32,
                                              i64, i32, i32, i32, i32, i32, vp]
    lib.tik_rmsnorm.argtypes = [vp, vp, vp, vp, vp, f32, i64, i32, vp]
    lib.tik_swiglu.argtypes = [vp, vp, vp, i64, i32, vp]
    lib.tik_linear.argtypes = [vp, vp, vp, vp, i64, i32, i32, vp]
    lib.tik_attn_train_bwd.argtypes = [vp, vp, vp, vp, vp, vp, vp, vp, vp, vp, vp, i32, i64, i32, i32, i32, i32, f32,
                                       vp, sz, vp]
    lib.tik_token_logprob.argtypes = [vp, vp, vp, vp, vp, vp, i64, i32, i32, f32, vp, sz, vp]
    lib.tik_attn_decode_static.argtypes = [vp, vp, vp, vp, vp, vp, vp, i32, i32, i32, i32, i32, i32, i32,
                                           i32, f32, vp, vp]
    lib.tik_attn_decode_static.restype = i32
    for name in ("tik_create", "tik_destroy", "tik_device_status", "tik_attn_train_fwd",
                 "tik_kv_cache_write", "tik_attn_prefill", "tik_attn_decode", "tik_token_logprob",
                 "tik_qk_norm_rope_kv_write", "tik_rmsnorm", "tik_swiglu", "tik_linear",
                 "tik_attn_train_bwd"):
        getattr(lib, name).restype = i32
    _lib = lib
    return lib


def contract_id() -> str:
    return load().tik_contract_id().decode()


def _load_native():
    """The extension module that marshals tensors (csrc/tik_bind.cpp), bound to libtik.so."""
    global _native
    if _native is None:
        load()
        path = _build.BIND_PATH
        if not os.path.exists(path):
            raise TikError("%s is not built; run `python -m paper_2609_35140_b200.build`. There is no fallback path."
                           % os.path.basename(path))
        spec = importlib.util.spec_from_file_location("_tikbind", path)
        module = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(module)
        module.init(TikError)
        _native = module
    return _native


def context(device: Optional[int] = None) -> ctypes.c_void_p:
    """The per-device library context (created on first use)."""
    return ctypes.c_void_p((_native or _load_native()).context_handle(device))


def _check(rc: int, ctx) -> None:
    if rc != OK:
        lib = load()
        raise TikError("%s: %s" % (lib.tik_status_str(rc).decode(), lib.tik_last_error(ctx).decode()))


def _stream():
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


def workspace_bytes(op: int, rows_or_batch: int = 0, Hq: int = 0, Hkv: int = 0, d: int = 0,
                    max_ctx: int = 0, H: int = 0, V: int = 0) -> int:
    return int(load().tik_workspace_bytes(op, rows_or_batch, Hq, Hkv, d, max_ctx, H, V))


def kernel_launches() -> int:
    """Kernels the library has launched in this process so far."""
    return int(load().tik_kernel_launches())


def device_status() -> int:
    """Synchronises the current stream; returns and clears the device flags."""
    ctx = context()
    flags = ctypes.c_int(0)
    _check(load().tik_device_status(ctx, _stream(), ctypes.byref(flags)), ctx)
    return flags.value


def tik_attn_train_fwd(q, k, v, cu_seqlens, max_seqlen: int, softmax_scale: float,
                       o: Optional[torch.Tensor] = None, lse: Optional[torch.Tensor] = None, ws=None):
    """q [tot,Hq,d], k/v [tot,Hkv,d] bf16, cu_seqlens int32 [S+1] (device) -> o [tot,Hq,d].
    ws: scratch tensor, None (allocated here) or False (run without: one CTA per work item)."""
    return (_native or _load_native()).attn_train_fwd(q, k, v, cu_seqlens, max_seqlen, softmax_scale, o, lse, ws)


def tik_attn_train_bwd(q, k, v, o, d_o, lse, cu_seqlens, max_seqlen: int, softmax_scale: float,
                       ws: Optional[torch.Tensor] = None):
    """Backward of tik_attn_train_fwd: returns (dq, dk, dv).  o, lse are the forward's outputs."""
    return (_native or _load_native()).attn_train_bwd(q, k, v, o, d_o, lse, cu_seqlens, max_seqlen, softmax_scale, ws)


def tik_kv_cache_write(k_new, v_new, cu_seqlens_new, ctx_lens, k_cache, v_cache, block_table):
    """Copies new K/V rows into the paged caches [num_pages,Hkv,page,d] in place."""
    (_native or _load_native()).kv_cache_write(k_new, v_new, cu_seqlens_new, ctx_lens, k_cache, v_cache, block_table)


def tik_qk_norm_rope_kv_write(q, k, v, q_weight, k_weight, eps: float, cos_sin, cu_seqlens_new,
                              ctx_lens=None, k_cache=None, v_cache=None, block_table=None):
    """Per-head RMSNorm (weights may be None) and NeoX RoPE of q [n,Hq,d] and k [n,Hkv,d] in place;
    with caches, rotated K and V also go to the pages.  cos_sin fp32 [max_pos,d]."""
    (_native or _load_native()).qk_norm_rope_kv_write(q, k, v, q_weight, k_weight, eps, cos_sin, cu_seqlens_new,
                                                      ctx_lens, k_cache, v_cache, block_table)


def tik_rmsnorm(x, weight, eps: float, residual=None, y: Optional[torch.Tensor] = None):
    """RMSNorm of x [T,H] over H; with residual [T,H], residual <- bf16(x + residual) first and that
    sum is normalised.  Returns y [T,H]."""
    return (_native or _load_native()).rmsnorm(x, weight, eps, residual, y)


def tik_swiglu(gate_up, out: Optional[torch.Tensor] = None):
    """gate_up [T,2I] (gate | up) -> silu(gate) * up, [T,I]."""
    return (_native or _load_native()).swiglu(gate_up, out)


def tik_linear(x, weight, y: Optional[torch.Tensor] = None):
    """x [T,K] @ weight[N,K]^T -> y [T,N] (bf16, fp32 accumulation)."""
    return (_native or _load_native()).linear(x, weight, y)


def tik_attn_prefill(q, cu_seqlens_q, ctx_lens, k_cache, v_cache, block_table, max_q_len: int,
                     max_ctx_len: int, softmax_scale: float, o: Optional[torch.Tensor] = None,
                     lse: Optional[torch.Tensor] = None, ws=None):
    """q [totq,Hq,d] against the paged cache -> o [totq,Hq,d].  ws as for tik_attn_train_fwd."""
    return (_native or _load_native()).attn_prefill(q, cu_seqlens_q, ctx_lens, k_cache, v_cache, block_table,
                                                    max_q_len, max_ctx_len, softmax_scale, o, lse, ws)


def tik_attn_prefill_kv(q, k_new, v_new, cu_seqlens_q, ctx_lens, k_cache, v_cache, block_table, max_q_len: int,
                        max_ctx_len: int, softmax_scale: float, o: Optional[torch.Tensor] = None,
                        lse: Optional[torch.Tensor] = None, ws=None):
    """Cache write of k_new / v_new [totq,Hkv,d] and prefill of q [totq,Hq,d] in one call -> o."""
    return (_native or _load_native()).attn_prefill_kv(q, k_new, v_new, cu_seqlens_q, ctx_lens, k_cache, v_cache,
                                                       block_table, max_q_len, max_ctx_len, softmax_scale, o, lse, ws)


def tik_attn_decode(q, ctx_lens, k_cache, v_cache, block_table, max_ctx_len: int, softmax_scale: float,
                    ws: Optional[torch.Tensor] = None, o: Optional[torch.Tensor] = None,
                    lse: Optional[torch.Tensor] = None):
    """q [B,Hq,d]: one token per sequence against the paged cache -> o [B,Hq,d]."""
    return (_native or _load_native()).attn_decode(q, ctx_lens, k_cache, v_cache, block_table, max_ctx_len,
                                                   softmax_scale, ws, o, lse)


def tik_token_logprob(hidden, lm_head, target_ids, inv_temperature: float = 1.0,
                      ws: Optional[torch.Tensor] = None, logprob: Optional[torch.Tensor] = None,
                      lse: Optional[torch.Tensor] = None):
    """hidden [T,H], lm_head [V,H] bf16, target_ids int32 [T] -> logprob fp32 [T]."""
    return (_native or _load_native()).token_logprob(hidden, lm_head, target_ids, inv_temperature, ws, logprob, lse)


STATIC_SCRATCH_BYTES = 8 << 20


def tik_attn_decode_static(q, ctx_lens, k_cache, v_cache, block_table, max_ctx_len: int,
                           softmax_scale: float, o: torch.Tensor, lse: Optional[torch.Tensor] = None,
                           dev_flags: Optional[torch.Tensor] = None) -> int:
    """Decode attention through the entry point that allocates nothing: no library context,
    no workspace (the scratch is a fixed array inside the library) and, unlike the other
    wrappers, no output tensor is created here either - the caller passes `o`.  For callers
    whose device memory is fully committed or who cannot afford cudaMalloc's synchronisation.
    Returns the raw status code (0 = ok; -3 = the problem exceeds the fixed scratch)."""
    return (_native or _load_native()).attn_decode_static(q, ctx_lens, k_cache, v_cache, block_table, max_ctx_len,
                                                          softmax_scale, o, lse, dev_flags)
