"""Thin Python binding of the C ABI (include/refadapt.h), same names.

Only argument marshalling happens here (natively, csrc/binding.cpp, for the
calls of a step): torch tensors supply device memory and streams; every step
of the computation runs in librefadapt.so's kernels.
Tensors are [B, H, n, d] bf16 CUDA views with a contiguous last axis (any
other strides, 16-byte aligned).
"""
import ctypes

import torch

from . import _lib
from ._lib import RaSeg, check

__all__ = ["seg", "refadapt_joint_attn", "refadapt_mass_partial_len", "refadapt_q_delta",
           "refadapt_q_delta_workspace_size", "refadapt_q_delta_noalloc", "refadapt_state_size", "refadapt_state_init",
           "refadapt_gate", "refadapt_ref_cache_update", "refadapt_set_wait_budget_ns",
           "refadapt_check_error", "refadapt_version", "refadapt_last_launch", "refadapt_selftest_wait_timeout", "q_delta_workspace", "new_state",
           "alloc_mass_partial", "refadapt_rope_table", "rope_table", "refadapt_ln_modulate", "refadapt_gemm"]


def _ptr(t):
    return None if t is None else ctypes.c_void_p(t.data_ptr())


def _stream(stream):
    if stream is None:
        stream = torch.cuda.current_stream()
    if isinstance(stream, torch.cuda.Stream):
        return ctypes.c_void_p(stream.cuda_stream)
    return ctypes.c_void_p(int(stream))


def _handle(stream):
    """A stream argument for the native calls: None (the current stream) or the raw handle."""
    if stream is None:
        return None
    return stream.cuda_stream if isinstance(stream, torch.cuda.Stream) else int(stream)


def seg(t, n=None) -> RaSeg:
    """ra_seg of a [B, H, n, d] bf16 CUDA tensor (None -> empty/absent segment)."""
    if t is None:
        return RaSeg(None, 0, 0, 0, int(n or 0), 0)
    if t.dim() != 4 or t.dtype != torch.bfloat16 or not t.is_cuda or (t.shape[3] > 1 and t.stride(3) != 1):
        raise ValueError("expected a [B, H, n, d] bf16 CUDA tensor with contiguous last axis, got %s %s %s"
                         % (tuple(t.shape), t.dtype, t.device))
    ptr = t.data_ptr() if t.numel() > 0 else 0
    return RaSeg(ptr or None, t.stride(0), t.stride(1), t.stride(2), t.shape[2], 0)


def refadapt_mass_partial_len(n_text, n_tgt) -> int:
    return int(_lib.load().refadapt_mass_partial_len(int(n_text), int(n_tgt)))


def alloc_mass_partial(B, H, n_text, n_tgt, device="cuda"):
    return torch.zeros((B, H, refadapt_mass_partial_len(n_text, n_tgt)), dtype=torch.float32, device=device)


def refadapt_joint_attn(q, k, v, o, mass_partial, mode=None, softmax_scale=0.0, ref_logit_bias=None,
                        mass_rows=0, err_word=None, mass_row_stride=0, ref_fresh=None, a_b=None, step=0,
                        stream=None):
    """q, k, v, o: sequences (text, ref, tgt) of [B, H, n, d] tensors; q[1] / o[1] may be None.
    ref_fresh: optional (q, k, v) of this step's reference rows for the fused
    cache update (q may be None when q[1] is); a_b, step: the stamp it writes."""
    if ref_fresh is None and a_b is not None:
        raise ValueError("refadapt_joint_attn: a_b is written only with ref_fresh")
    return check("refadapt_joint_attn", _lib.native().joint_attn(
        q, k, v, o, mass_partial, mode, float(softmax_scale), ref_logit_bias, int(mass_rows), err_word,
        int(mass_row_stride), ref_fresh, a_b, int(step), _handle(stream)))


def refadapt_q_delta_workspace_size(B, H) -> int:
    return int(_lib.load().refadapt_q_delta_workspace_size(int(B), int(H)))


def q_delta_workspace(B, H, device="cuda"):
    """A zero-filled workspace for refadapt_q_delta (reusable across calls)."""
    return torch.zeros(refadapt_q_delta_workspace_size(B, H), dtype=torch.uint8, device=device)


def refadapt_q_delta(q_cur, q_prev, d_out, workspace, eps=1e-6, stream=None):
    return check("refadapt_q_delta", _lib.native().q_delta(q_cur, q_prev, d_out, workspace, float(eps),
                                                           _handle(stream)))


def refadapt_q_delta_noalloc(q_cur, q_prev, d_out, eps=1e-6, stream=None):
    """refadapt_q_delta without a workspace (static scratch inside the library;
    B * H <= RA_Q_DELTA_NOALLOC_MAX_BH; calls must not overlap on the GPU)."""
    lib = _lib.load()
    B, H, _, d = q_cur.shape
    sc, sp = seg(q_cur), seg(q_prev)
    return check("refadapt_q_delta_noalloc", lib.refadapt_q_delta_noalloc(
        ctypes.byref(sc), ctypes.byref(sp), B, H, d, float(eps), _ptr(d_out), _stream(stream)))


def refadapt_state_size(B) -> int:
    return int(_lib.load().refadapt_state_size(int(B)))


def refadapt_state_init(state, B, stream=None):
    return check("refadapt_state_init", _lib.load().refadapt_state_init(_ptr(state), int(B), _stream(stream)))


def new_state(B, device="cuda", stream=None):
    st = torch.empty(refadapt_state_size(B), dtype=torch.uint8, device=device)
    refadapt_state_init(st, B, stream)
    return st


def refadapt_gate(t, b, state, mode_out, theta, delta_max, B, H, q_delta=None, mass_partial_prev=None,
                  mass_row_count=0, forced_boundary=-1, gbar_out=None, m_out=None, cue=0, stream=None):
    return check("refadapt_gate", _lib.native().gate(
        int(t), int(b), state, mode_out, float(theta), int(delta_max), int(B), int(H), q_delta, mass_partial_prev,
        int(mass_row_count), int(forced_boundary), gbar_out, m_out, int(cue), _handle(stream)))


def refadapt_q_delta_gate(q_cur, q_prev, d_out, workspace, t, b, state, mode_out, theta, delta_max,
                          mass_partial_prev, mass_row_count, eps=1e-6, forced_boundary=-1, gbar_out=None,
                          m_out=None, cue=0, stream=None):
    """refadapt_q_delta then refadapt_gate on its D (t >= 1), in one launch
    when the Q change takes its cluster path."""
    return check("refadapt_q_delta_gate", _lib.native().q_delta_gate(
        q_cur, q_prev, d_out, workspace, float(eps), _handle(stream), int(t), int(b), state, mode_out, float(theta),
        int(delta_max), mass_partial_prev, int(mass_row_count), int(forced_boundary), gbar_out, m_out, int(cue)))


def refadapt_ref_cache_update(k_src, v_src, k_cache, v_cache, mode, t, a_b=None, x_src=None, x_cache=None,
                              stream=None):
    lib = _lib.load()
    B, H, _, d = k_src.shape
    ks, vs, kc, vc = seg(k_src), seg(v_src), seg(k_cache), seg(v_cache)
    if x_src is not None:
        xs, xc = seg(x_src), seg(x_cache)
        xp, xcp = ctypes.byref(xs), ctypes.byref(xc)
        x_heads, x_width = x_src.shape[1], x_src.shape[3]
    else:
        xp = xcp = None
        x_heads = x_width = 0
    return check("refadapt_ref_cache_update", lib.refadapt_ref_cache_update(
        ctypes.byref(ks), ctypes.byref(vs), ctypes.byref(kc), ctypes.byref(vc), B, H, d, xp, xcp,
        x_heads, x_width, _ptr(mode), int(t), _ptr(a_b), _stream(stream)))


def refadapt_set_wait_budget_ns(ns):
    _lib.load().refadapt_set_wait_budget_ns(int(ns))


def refadapt_check_error(err_word, stream=None):
    return check("refadapt_check_error", _lib.load().refadapt_check_error(_ptr(err_word), _stream(stream)))


def refadapt_selftest_wait_timeout(err_word, budget_ns, stream=None):
    return check("refadapt_selftest_wait_timeout",
                 _lib.load().refadapt_selftest_wait_timeout(_ptr(err_word), int(budget_ns), _stream(stream)))


def refadapt_last_launch() -> str:
    return _lib.load().refadapt_last_launch().decode()


def refadapt_version() -> int:
    return int(_lib.load().refadapt_version())


# --------------------------------------------------------------------------- DiT block around the attention
def refadapt_rope_table(table, n_pos, d, base=10000.0, stream=None):
    return check("refadapt_rope_table", _lib.load().refadapt_rope_table(
        _ptr(table), int(n_pos), int(d), float(base), _stream(stream)))


def rope_table(n_pos, d, base=10000.0, device="cuda", stream=None):
    """[n_pos, d/2, 2] fp32 (cos, sin) table built by refadapt_rope_table."""
    t = torch.empty((int(n_pos), int(d) // 2, 2), dtype=torch.float32, device=device)
    refadapt_rope_table(t, n_pos, d, base, stream)
    return t


def refadapt_ln_modulate(segs, C, eps=1e-6, mode=None, stream=None):
    """segs: up to three dicts with h, x ([B, rows, C] bf16), shift, scale
    ([B, C] fp32) and optional gated (bool)."""
    return check("refadapt_ln_modulate",
                 _lib.native().ln_modulate(segs, int(C), float(eps), mode, _handle(stream)))


def refadapt_gemm(segs, N, K, epilogue, mode=None, rope=None, H=0, d=0, norm_eps=1e-6, err_word=None,
                  tile_mode=0, stream=None):
    """segs: up to three dicts with a ([B, rows, K] bf16), w ([N, K] bf16),
    optional bias ([N] fp32), gated; plus per epilogue out ([B, rows, N]),
    resid and gate ([B, N] fp32) for RESID, or q, k, v ([B, H, rows, d]),
    q_norm, k_norm ([d] fp32) and pos_offset for QKV."""
    return check("refadapt_gemm", _lib.native().gemm(
        segs, int(N), int(K), int(epilogue), mode, rope, int(H), int(d), float(norm_eps), err_word, int(tile_mode),
        _handle(stream)))
