"""SPADE verify step on GB300: Python binding of the C-ABI library libspade.so.

This module only marshals arguments: the native extension (csrc/binding.cpp)
checks dtypes and layouts of torch tensors and passes raw device pointers,
sizes and the current CUDA stream to the library's entry points; helpers that
are not on a verify step's path go through ctypes.  Every step of the verify
path runs in the library's CUDA kernels; there is no Python or CPU fallback,
and a call fails loudly if the library is missing.

Entry points (same names as the C ABI in include/spade.h):
    spade_verify_attention  verify-position attention against the KV cache
    spade_verify_accept     LM head + softmax + accept/reject + residual sampling
    spade_kv_commit         append accepted positions, roll back rejected ones
    spade_verify_qkv_rope   QKV projection + rotary embedding of the verify block, K/V into the cache
"""
from __future__ import annotations

import ctypes
import importlib.util
import os

import torch

from . import _build

__all__ = [
    "SpadeError", "load", "build", "library_path",
    "spade_verify_attention", "spade_verify_accept", "spade_kv_commit", "spade_verify_attention_noalloc",
    "spade_verify_qkv_rope", "spade_qkv_workspace_size", "qkv_workspace", "spade_verify_attention_paged", "spade_kv_commit_paged",
    "spade_verify_qkv_rope_paged",
    "spade_attn_workspace_size", "spade_accept_workspace_size", "spade_accept_launches",
    "spade_accept_stats_layout", "read_accept_stats", "spade_verify_accept_commit",
    "spade_verify_accept_sampling", "spade_verify_accept_commit_paged", "spade_selftest_wait_timeout",
    "attn_workspace", "accept_workspace", "status_tensor", "check_status",
    "DEV_BAD_INDEX", "DEV_CAPACITY", "DEV_TIMEOUT", "DEV_FALLBACK",
]

DEV_BAD_INDEX = 0x1
DEV_CAPACITY = 0x2
DEV_TIMEOUT = 0x4
DEV_FALLBACK = 0x8

_lib = None
_native = None  # the extension module, once loaded


class SpadeError(RuntimeError):
    """A non-OK status returned by the library (message from spade_last_error)."""

    def __init__(self, status, message):
        super().__init__(f"{message} [status {status}]")
        self.status = status


def library_path() -> str:
    return _build.LIB_PATH


def build(force: bool = False) -> str:
    return _build.build(force=force)


_i32 = ctypes.c_int32
_vp = ctypes.c_void_p
_sz = ctypes.c_size_t


def load():
    """Load libspade.so (built in-tree); raises if it has not been built."""
    global _lib
    if _lib is not None:
        return _lib
    path = library_path()
    if not os.path.exists(path):
        raise RuntimeError(f"{path} is missing: build the CUDA library first "
                           "(python -c 'import __graft_entry__ as g; g.build()')")
    lib = ctypes.CDLL(path)
    lib.spade_verify_attention.restype = _i32
    lib.spade_verify_attention.argtypes = [_vp, _vp, _vp, _vp, _vp, _vp, _vp, _vp,
                                           _i32, _i32, _i32, _i32, _i32, _i32, _i32,
                                           _vp, _sz, _vp, _vp]
    lib.spade_verify_attention_noalloc.restype = _i32
    lib.spade_verify_attention_noalloc.argtypes = [_vp] * 8 + [_i32] * 7 + [_vp, _vp]
    lib.spade_attn_workspace_size.restype = _sz
    lib.spade_attn_workspace_size.argtypes = [_i32] * 6
    lib.spade_verify_accept.restype = _i32
    lib.spade_verify_accept.argtypes = [_vp] * 10 + [_i32] * 4 + [_vp, _sz, _vp, _vp]
    lib.spade_verify_accept_commit.restype = _i32
    lib.spade_verify_accept_commit.argtypes = [_vp] * 13 + [_i32] * 7 + [_vp, _sz, _vp, _vp]
    lib.spade_accept_workspace_size.restype = _sz
    lib.spade_accept_workspace_size.argtypes = [_i32] * 4
    lib.spade_verify_accept_temperature.restype = _i32
    lib.spade_verify_accept_temperature.argtypes = [_vp] * 11 + [_i32] * 4 + [_vp, _sz, _vp, _vp]
    lib.spade_verify_accept_sampling.restype = _i32
    lib.spade_verify_accept_sampling.argtypes = [_vp] * 15 + [_i32] * 7 + [_vp, _sz, _vp, _vp]
    lib.spade_accept_stats_layout.restype = _i32
    lib.spade_accept_stats_layout.argtypes = [_i32] * 4 + [_vp, _vp, _vp]
    lib.spade_accept_launches.restype = _i32
    lib.spade_accept_launches.argtypes = [_i32] * 4
    lib.spade_selftest_wait_timeout.restype = _i32
    lib.spade_selftest_wait_timeout.argtypes = [_vp, _i32, _vp]
    lib.spade_verify_qkv_rope.restype = _i32
    lib.spade_verify_qkv_rope.argtypes = [_vp] * 8 + [_i32] * 8 + [ctypes.c_float, _vp, _sz, _vp, _vp]
    lib.spade_qkv_workspace_size.restype = _sz
    lib.spade_qkv_workspace_size.argtypes = [_i32] * 4
    lib.spade_verify_attention_paged.restype = _i32
    lib.spade_verify_attention_paged.argtypes = [_vp] * 9 + [_i32] * 9 + [_vp, _sz, _vp, _vp]
    lib.spade_verify_accept_commit_paged.restype = _i32
    lib.spade_verify_accept_commit_paged.argtypes = [_vp] * 14 + [_i32] * 9 + [_vp, _sz, _vp, _vp]
    lib.spade_kv_commit_paged.restype = _i32
    lib.spade_kv_commit_paged.argtypes = [_vp] * 6 + [_i32] * 6 + [_vp, _vp]
    lib.spade_verify_qkv_rope_paged.restype = _i32
    lib.spade_verify_qkv_rope_paged.argtypes = [_vp] * 9 + [_i32] * 10 + [ctypes.c_float, _vp, _sz, _vp, _vp]
    lib.spade_kv_commit.restype = _i32
    lib.spade_kv_commit.argtypes = [_vp] * 5 + [_i32] * 4 + [_vp, _vp]
    lib.spade_status_string.restype = ctypes.c_char_p
    lib.spade_status_string.argtypes = [_i32]
    lib.spade_last_error.restype = ctypes.c_char_p
    lib.spade_last_error.argtypes = []
    lib.spade_version.restype = ctypes.c_char_p
    lib.spade_version.argtypes = []
    _lib = lib
    return lib


def native():
    """The native extension that checks and passes a call's tensors (built with the library)."""
    global _native
    if _native is None:
        load()
        path = _build.NATIVE_PATH
        if not os.path.exists(path):
            raise RuntimeError(f"{path} is missing: build the CUDA library first "
                               "(python -c 'import __graft_entry__ as g; g.build()')")
        spec = importlib.util.spec_from_file_location("_spade_native", path)
        module = importlib.util.module_from_spec(spec)
        spec.loader.exec_module(module)
        _native = module
    return _native


def _ptr(t):
    return None if t is None else ctypes.c_void_p(t.data_ptr())


def _stream(stream):
    if stream is None:
        stream = torch.cuda.current_stream()
    return ctypes.c_void_p(stream.cuda_stream)


def _check_rc(rc):
    if rc != 0:
        lib = load()
        raise SpadeError(rc, f"{lib.spade_status_string(rc).decode()}: {lib.spade_last_error().decode()}")


def _need(t, name, dtype, ndim=None):
    if t is None:
        raise ValueError(f"{name} is required")
    if t.dtype != dtype:
        raise TypeError(f"{name} must be {dtype}, got {t.dtype}")
    if not t.is_cuda:
        raise ValueError(f"{name} must be a CUDA tensor")
    if not t.is_contiguous():
        raise ValueError(f"{name} must be contiguous")
    if ndim is not None and t.dim() != ndim:
        raise ValueError(f"{name} must have {ndim} dims, got {t.dim()}")


def status_tensor(device="cuda"):
    """A zeroed device int32 status word."""
    return torch.zeros(1, dtype=torch.int32, device=device)


def check_status(status):
    """Reads the device status word (synchronises) and returns its SPADE_DEV_* bits."""
    return int(status.item())


# ---------------------------------------------------------------------------
def spade_attn_workspace_size(B, Hq, Hkv, D, cap, max_k):
    return int(load().spade_attn_workspace_size(B, Hq, Hkv, D, cap, max_k))


def attn_workspace(B, Hq, Hkv, D, cap, max_k, device="cuda"):
    """A zeroed workspace for spade_verify_attention (zeroed once; calls keep it zeroed)."""
    n = spade_attn_workspace_size(B, Hq, Hkv, D, cap, max_k)
    if n == 0:
        raise SpadeError(-1, "spade_attn_workspace_size returned 0: " + load().spade_last_error().decode())
    return torch.zeros(n, dtype=torch.uint8, device=device)


def spade_verify_attention(q, k_cache, v_cache, ctx_lens, n_draft, cu_q, out, lse=None, *,
                           max_k, workspace, status, stream=None):
    """out[cu_q[b]+i, h] = softmax(q K^T / sqrt(D)) V over keys [0, ctx_b + i] (KV head h // G)."""
    rc = (_native or native()).attention(
        q, k_cache, v_cache, ctx_lens, n_draft, cu_q, out, lse, max_k, workspace, status, stream)
    if rc:
        _check_rc(rc)
    return out


def spade_verify_attention_noalloc(q, k_cache, v_cache, ctx_lens, n_draft, cu_q, out, lse=None, *,
                                   max_k, status, stream=None):
    """spade_verify_attention for callers that cannot allocate: scratch in a static device array.

    Calls that overlap on the GPU share that array and race; the first call on
    a device resolves the array's address and should precede any stream capture.
    An ``lse`` that is given must be a contiguous float32 CUDA tensor.
    """
    rc = (_native or native()).attention_noalloc(
        q, k_cache, v_cache, ctx_lens, n_draft, cu_q, out, lse, max_k, status, stream)
    if rc:
        _check_rc(rc)
    return out


# ---------------------------------------------------------------------------
def spade_accept_workspace_size(B, R, H, V):
    return int(load().spade_accept_workspace_size(B, R, H, V))


def spade_selftest_wait_timeout(status, limit_us, stream=None):
    """One bounded wait that nothing completes: SPADE_DEV_TIMEOUT lands in `status` after limit_us."""
    _need(status, "status", torch.int32, 1)
    _check_rc(load().spade_selftest_wait_timeout(_ptr(status), int(limit_us), _stream(stream)))


def spade_accept_stats_layout(B, R, H, V):
    """Byte offsets of the merged row statistics and the draft logits in an accept workspace.

    Returns (row_stats_offset, draft_logit_offset, replica_stride); see include/spade.h.
    """
    a, b, c = ctypes.c_size_t(0), ctypes.c_size_t(0), ctypes.c_int32(0)
    _check_rc(load().spade_accept_stats_layout(B, R, H, V, ctypes.byref(a), ctypes.byref(b), ctypes.byref(c)))
    return int(a.value), int(b.value), int(c.value)


def read_accept_stats(workspace, B, R, H, V):
    """Row statistics a completed accept call left in `workspace` (reads device memory).

    Returns dict of torch CPU tensors: max [R] f32, sumexp [R] f32, argmax [R] i32,
    accept_bit [R] i32, draft_logit [R] f32 (rows with a draft only are meaningful).
    """
    off_s, off_d, _ = spade_accept_stats_layout(B, R, H, V)
    st = workspace[off_s:off_s + 16 * R].view(torch.float32).view(R, 4).cpu()
    ld = workspace[off_d:off_d + 4 * R].view(torch.float32).cpu()
    return dict(max=st[:, 0].clone(), sumexp=st[:, 1].clone(), argmax=st[:, 2].clone().view(torch.int32),
                accept_bit=st[:, 3].clone().view(torch.int32), draft_logit=ld.clone())


def spade_accept_launches(B, R, H, V):
    """Kernel launches of one accept call: 1, or 2 (statistics, then decisions and draws)."""
    return int(load().spade_accept_launches(B, R, H, V))


def accept_workspace(B, R, H, V, device="cuda"):
    """A zeroed workspace for spade_verify_accept (zeroed once; calls keep it usable)."""
    n = spade_accept_workspace_size(B, R, H, V)
    if n == 0:
        raise SpadeError(-1, "spade_accept_workspace_size returned 0: " + load().spade_last_error().decode())
    return torch.zeros(n, dtype=torch.uint8, device=device)


def spade_verify_accept(hidden, w_lm, draft_tokens, draft_probs, uniforms, mode, cu_q, n_draft,
                        accepted_len, next_token, *, workspace, status, stream=None, temperature=None):
    """Greedy / rejection-sampling verification of every sequence (see include/spade.h); with
    ``temperature`` ([B] float32) the verifier's p is softmax(logits / T)."""
    rc = (_native or native()).accept(
        hidden, w_lm, draft_tokens, draft_probs, uniforms, mode, cu_q, n_draft,
        accepted_len, next_token, temperature, workspace, status, stream)
    if rc:
        _check_rc(rc)
    return accepted_len, next_token


def spade_verify_accept_commit(hidden, w_lm, draft_tokens, draft_probs, uniforms, mode, cu_q, n_draft,
                               accepted_len, next_token, k_cache, v_cache, ctx_lens, *, workspace,
                               status, stream=None):
    """spade_verify_accept followed by spade_kv_commit in one launch (see include/spade.h)."""
    rc = (_native or native()).accept_commit(
        hidden, w_lm, draft_tokens, draft_probs, uniforms, mode, cu_q, n_draft,
        accepted_len, next_token, k_cache, v_cache, ctx_lens, workspace, status, stream)
    if rc:
        _check_rc(rc)
    return accepted_len, next_token


def spade_verify_accept_sampling(hidden, w_lm, draft_tokens, draft_probs, uniforms, mode, cu_q, n_draft,
                                 accepted_len, next_token, *, workspace, status, temperature=None, top_p=None,
                                 k_cache=None, v_cache=None, ctx_lens=None, stream=None):
    """spade_verify_accept with per-sequence ``temperature`` and ``top_p`` ([B] float32, either
    may be None) and, with k_cache / v_cache / ctx_lens given, the fused KV commit
    (see include/spade.h)."""
    rc = (_native or native()).accept_sampling(
        hidden, w_lm, draft_tokens, draft_probs, uniforms, mode, cu_q, n_draft,
        accepted_len, next_token, temperature, top_p, k_cache, v_cache, ctx_lens, workspace, status,
        stream)
    if rc:
        _check_rc(rc)
    return accepted_len, next_token


def spade_verify_accept_commit_paged(hidden, w_lm, draft_tokens, draft_probs, uniforms, mode, cu_q, n_draft,
                                     accepted_len, next_token, k_pool, v_pool, block_table, ctx_lens, *,
                                     workspace, status, stream=None):
    """spade_verify_accept_commit on paged caches: pools [num_pages, Hkv, page_size, D] and a
    block table [B, max_pages] (see include/spade.h)."""
    rc = (_native or native()).accept_commit_paged(
        hidden, w_lm, draft_tokens, draft_probs, uniforms, mode, cu_q, n_draft,
        accepted_len, next_token, k_pool, v_pool, block_table, ctx_lens, workspace, status, stream)
    if rc:
        _check_rc(rc)
    return accepted_len, next_token


# ---------------------------------------------------------------------------
def spade_qkv_workspace_size(R, Hq, Hkv, D):
    return int(load().spade_qkv_workspace_size(R, Hq, Hkv, D))


def qkv_workspace(R, Hq, Hkv, D, device="cuda"):
    """A zeroed workspace for spade_verify_qkv_rope (zeroed once; calls keep its counters zeroed)."""
    n = spade_qkv_workspace_size(R, Hq, Hkv, D)
    if n == 0:
        raise SpadeError(-1, "spade_qkv_workspace_size returned 0: " + load().spade_last_error().decode())
    return torch.zeros(n, dtype=torch.uint8, device=device)


def spade_verify_qkv_rope(x, w_qkv, ctx_lens, n_draft, cu_q, q_out, k_cache, v_cache, *, Hq, Hkv,
                          rope_theta, max_k, workspace, status, stream=None):
    """q, k, v of the verify block (rotary embedding at ctx + i); K/V into cache slots ctx .. ctx + k."""
    rc = (_native or native()).qkv(
        x, w_qkv, ctx_lens, n_draft, cu_q, q_out, k_cache, v_cache, Hq, Hkv, rope_theta, max_k, workspace, status,
        stream)
    if rc:
        _check_rc(rc)
    return q_out


# ---------------------------------------------------------------------------
# Paged KV cache: pools [num_pages, Hkv, page_size, D], block_table [B, max_pages].
def spade_verify_attention_paged(q, k_pool, v_pool, block_table, ctx_lens, n_draft, cu_q, out, lse=None, *,
                                 max_k, workspace, status, stream=None):
    """spade_verify_attention on a paged cache (see include/spade.h)."""
    rc = (_native or native()).attention_paged(
        q, k_pool, v_pool, block_table, ctx_lens, n_draft, cu_q, out, lse, max_k, workspace, status, stream)
    if rc:
        _check_rc(rc)
    return out


def spade_kv_commit_paged(k_pool, v_pool, block_table, ctx_lens, accepted_len, n_draft, *, status, stream=None):
    """spade_kv_commit on a paged cache (see include/spade.h)."""
    rc = (_native or native()).commit_paged(
        k_pool, v_pool, block_table, ctx_lens, accepted_len, n_draft, status, stream)
    if rc:
        _check_rc(rc)


def spade_verify_qkv_rope_paged(x, w_qkv, block_table, ctx_lens, n_draft, cu_q, q_out, k_pool, v_pool, *, Hq,
                                rope_theta, max_k, workspace, status, stream=None):
    """spade_verify_qkv_rope writing the block's K/V into a paged cache (see include/spade.h)."""
    rc = (_native or native()).qkv_paged(
        x, w_qkv, block_table, ctx_lens, n_draft, cu_q, q_out, k_pool, v_pool, Hq, rope_theta, max_k, workspace,
        status, stream)
    if rc:
        _check_rc(rc)
    return q_out


# ---------------------------------------------------------------------------
def spade_kv_commit(k_cache, v_cache, ctx_lens, accepted_len, n_draft, *, status, stream=None):
    """ctx_lens += accepted_len + 1; rejected draft slots of the caches are cleared."""
    rc = (_native or native()).commit(k_cache, v_cache, ctx_lens, accepted_len, n_draft, status, stream)
    if rc:
        _check_rc(rc)