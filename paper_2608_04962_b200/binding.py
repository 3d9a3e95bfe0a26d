"""Thin Python binding of the C-ABI library ``libspecroll.so``.

Argument marshalling only: every function checks dtype / device / contiguity of torch
tensors, allocates outputs and the workspace with torch, and passes raw pointers to the
entry point of the same name (``_native``, csrc/native.cpp, does that; this module holds the
signatures and the calls that only ask the host).  No step of the method runs in Python.  The
library is loaded on first use and loading fails loudly when it has not been built: there is no
fallback.
"""
from __future__ import annotations

import ctypes as C
import os
from typing import Dict, Optional

import numpy as np
import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
# SPECROLL_LIB selects another build of the same library (the debug build with index checks, libspecroll_check.so)
LIB_PATH = os.environ.get("SPECROLL_LIB") or os.path.join(_HERE, "libspecroll.so")
_lib = None
_native = None      # csrc/native.cpp, attached to the loaded library

EXPORTS = ("specroll_version", "specroll_strerror", "specroll_node_budget", "specroll_check_status", "specroll_check_inject",
           "specroll_propose_workspace_bytes", "specroll_propose", "specroll_workspace_status",
           "specroll_tree_draw",
           "specroll_tree_attn_workspace_bytes", "specroll_tree_attn", "specroll_tree_attn_launches",
           "specroll_tree_attn_paged_workspace_bytes", "specroll_tree_attn_paged",
           "specroll_commit_path", "specroll_commit_path_layers", "specroll_gather_hidden",
           "specroll_verify_workspace_bytes", "specroll_verify", "specroll_verify_static",
           "specroll_verify_nucleus_workspace_bytes", "specroll_verify_nucleus",
           "specroll_reflex_feedback_workspace_bytes", "specroll_reflex_feedback", "specroll_reflex_feedback_ex",
           "specroll_reflex_sketch", "specroll_reflex_gate",
           "specroll_target_head_stats_workspace_bytes", "specroll_target_head_stats", "specroll_target_head_rows",
           "specroll_verify_want_ids", "specroll_verify_walk_sparse", "specroll_verify_terminal_rows",
           "specroll_target_head_tile_mass_bytes", "specroll_target_head_stats_tiles", "specroll_verify_hidden")


PROPOSE_LEGACY_MMA = 1
REFLEX_PRE_HEAD = 2
ATTN_LEGACY_MMA = 1
ATTN_REUSE_PLAN = 2
ATTN_CACHE_SETTLED = 4
ATTN_NO_PDL = 8
VERIFY_LAZY_STATS = 1
FEEDBACK_SEVERITY = 1
PAGE_TOKENS = 128


class SpecrollError(RuntimeError):
    pass


class ProposeDesc(C.Structure):
    _fields_ = [("B", C.c_int32), ("N", C.c_int32), ("K", C.c_int32), ("k", C.c_int32),
                ("d", C.c_int32), ("V", C.c_int32), ("temperature", C.c_float),
                ("ln_eps", C.c_float), ("rms_eps", C.c_float), ("clip_c", C.c_float),
                ("flags", C.c_int32)]


class AttnDesc(C.Structure):
    _fields_ = [("B", C.c_int32), ("N", C.c_int32), ("Hq", C.c_int32), ("Hkv", C.c_int32),
                ("D", C.c_int32), ("scale", C.c_float), ("flags", C.c_int32)]


class VerifyDesc(C.Structure):
    _fields_ = [("B", C.c_int32), ("N", C.c_int32), ("K", C.c_int32), ("k", C.c_int32),
                ("V", C.c_int32), ("temperature", C.c_float), ("flags", C.c_int32)]


class FeedbackDesc(C.Structure):
    _fields_ = [("R", C.c_int32), ("k", C.c_int32), ("k_support", C.c_int32), ("d", C.c_int32), ("V", C.c_int32),
                ("temperature", C.c_float), ("eps", C.c_float), ("flags", C.c_int32), ("severity_min", C.c_float)]


class GateDesc(C.Structure):
    _fields_ = [("R", C.c_int32), ("S", C.c_int32), ("d", C.c_int32), ("rank", C.c_int32), ("H", C.c_int32),
                ("z_delta", C.c_float), ("mem_eps", C.c_float), ("flags", C.c_int32)]


def lib():
    """The loaded library.  Raises if it is missing: the CUDA path is the only path."""
    global _lib
    if _lib is None:
        if not os.path.exists(LIB_PATH):
            raise SpecrollError(
                f"{LIB_PATH} is missing: build it with `python -m paper_2608_04962_b200.build` "
                "(there is no CPU or PyTorch fallback)")
        l = C.CDLL(LIB_PATH)
        l.specroll_version.restype = C.c_int
        l.specroll_strerror.restype = C.c_char_p
        l.specroll_strerror.argtypes = [C.c_int]
        l.specroll_node_budget.restype = C.c_int32
        l.specroll_node_budget.argtypes = [C.c_int32] * 4
        for n in ("specroll_propose_workspace_bytes", "specroll_verify_workspace_bytes",
                  "specroll_tree_attn_workspace_bytes", "specroll_tree_attn_paged_workspace_bytes",
                  "specroll_verify_nucleus_workspace_bytes", "specroll_reflex_feedback_workspace_bytes",
                  "specroll_target_head_stats_workspace_bytes"):
            getattr(l, n).restype = C.c_size_t
        for n in ("specroll_propose", "specroll_workspace_status", "specroll_tree_draw", "specroll_tree_attn",
                  "specroll_verify", "specroll_verify_static", "specroll_tree_attn_paged", "specroll_commit_path",
                  "specroll_commit_path_layers", "specroll_gather_hidden", "specroll_verify_nucleus",
                  "specroll_tree_attn_launches", "specroll_reflex_feedback"):
            getattr(l, n).restype = C.c_int
        try:
            from . import _native as n
        except ImportError as e:
            raise SpecrollError(
                f"the binding's native part is missing or does not load ({e}): build it with "
                "`python -m paper_2608_04962_b200.build`") from e
        n.attach(SpecrollError, _host_i32, {name: C.cast(getattr(l, name), C.c_void_p).value for name in EXPORTS})
        n.set_alloc(None if _empty is torch.empty else _alloc_for_native)
        global _native
        _native, _lib = n, l
    return _lib


def _n():
    """The native part, with the library loaded."""
    if _native is None:
        lib()
    return _native


def _check(rc: int, what: str):
    if rc != 0:
        raise SpecrollError(f"{what}: {lib().specroll_strerror(rc).decode()} (code {rc})")


def _host_i32(a, name: str) -> np.ndarray:
    a = np.ascontiguousarray(np.asarray(a), dtype=np.int32)
    if a.ndim != 1:
        raise SpecrollError(f"{name} must be one-dimensional")
    return a


def _stream() -> C.c_void_p:
    return C.c_void_p(torch.cuda.current_stream().cuda_stream)


# Every device tensor this module allocates (outputs and workspaces) comes from this function.  The tests swap in
# an allocator that surrounds each tensor with guard bytes and checks them afterwards (set_allocator); by default
# it is torch.empty.
_empty = torch.empty


_DTYPES = {0: torch.uint8, 3: torch.int32, 6: torch.float32, 15: torch.bfloat16}   # by at::ScalarType


def _alloc_for_native(shape, dtype_code, device_index):
    return _empty(shape, dtype=_DTYPES[dtype_code],
                  device=torch.device("cuda", device_index) if device_index >= 0 else torch.device("cpu"))


def set_allocator(fn=None):
    """Replaces the allocator of outputs and workspaces (signature of torch.empty); None restores torch.empty."""
    global _empty
    _empty = torch.empty if fn is None else fn
    if _native is not None:
        _native.set_alloc(None if fn is None else _alloc_for_native)


def alloc(*size, **kw) -> torch.Tensor:
    """torch.empty through the current allocator (for callers that keep outputs and workspaces of their own)."""
    return _empty(*size, **kw)


def version() -> int:
    return int(lib().specroll_version())


def check_status(reset: bool = True):
    """specroll_check_status after a device synchronisation: (code, detail).  code is -1 for a normal build, 0 when
    the debug build's index checks found nothing, else SPECROLL_EINDEX with detail = the sequence it was found in."""
    torch.cuda.synchronize()
    detail = C.c_int32(0)
    rc = int(lib().specroll_check_status(C.byref(detail), C.c_int32(1 if reset else 0)))
    return rc, int(detail.value)


def workspace_status(workspace: torch.Tensor) -> int:
    """specroll_workspace_status: 0, or the error code a kernel left in this workspace (synchronises)."""
    return int(lib().specroll_workspace_status(C.c_void_p(workspace.data_ptr()), _stream()))


def node_budget(C_hw: int, B_active: int, N_min: int = 1, N_max: int = 10) -> int:
    return int(lib().specroll_node_budget(C_hw, B_active, N_min, N_max))


# ----------------------------------------------------------------------------------- propose


def propose_workspace_bytes(B, N, K, k, d, V, temperature=1.0, ln_eps=1e-5, rms_eps=1e-6,
                            clip_c=0.0, flags=0) -> int:
    desc = ProposeDesc(B, N, K, k, d, V, temperature, ln_eps, rms_eps, clip_c, flags)
    return int(lib().specroll_propose_workspace_bytes(C.byref(desc)))


def propose(h, anchor, A, bias, W, m, alpha, parent, u_draw, k, temperature=1.0, ln_eps=1e-5,
            rms_eps=1e-6, clip_c=0.0, ln_gamma=None, ln_beta=None, workspace=None,
            out: Optional[Dict[str, torch.Tensor]] = None, flags: int = 0,
            check_status: bool = False) -> Dict[str, torch.Tensor]:
    """specroll_propose.  Device tensors in, dict of device tensors out.
    ``check_status`` also calls specroll_workspace_status (synchronises the stream)."""
    out, workspace = _n().propose(h, anchor, A, bias, W, m, alpha, parent, u_draw, k, temperature, ln_eps, rms_eps, clip_c,
                                  ln_gamma, ln_beta, workspace, out, flags)
    if check_status:
        _check(workspace_status(workspace), "specroll_workspace_status")
    return out


def tree_draw(parent, anchor, cand_id, cand_logit, u_draw, temperature=1.0) -> Dict[str, torch.Tensor]:
    """specroll_tree_draw."""
    return _n().tree_draw(parent, anchor, cand_id, cand_logit, u_draw, temperature)


# ----------------------------------------------------------------------------------- attention


def tree_attn_workspace_bytes(B, N, Hq, Hkv, D, kv_indptr_host, scale=None) -> int:
    ip = _host_i32(kv_indptr_host, "kv_indptr_host")
    desc = AttnDesc(B, N, Hq, Hkv, D, scale if scale is not None else 1.0 / float(np.sqrt(D)), 0)
    return int(lib().specroll_tree_attn_workspace_bytes(C.byref(desc), ip.ctypes.data_as(C.c_void_p)))


def tree_attn_launches(B, N, Hq, Hkv, D, kv_indptr_host, flags: int = 0) -> int:
    """Kernels one tree_attn call enqueues for these lengths (the plan decides whether a merge kernel runs)."""
    ip = _host_i32(kv_indptr_host, "kv_indptr_host")
    desc = AttnDesc(B, N, Hq, Hkv, D, 1.0 / float(np.sqrt(D)), flags)
    return int(lib().specroll_tree_attn_launches(C.byref(desc), ip.ctypes.data_as(C.c_void_p)))


def tree_attn(Q, Kc, Vc, kv_indptr_dev, kv_indptr_host, Kt, Vt, parent, scale=None, want_lse=False,
              workspace=None, out=None, lse=None, flags: int = 0, check_status: bool = False):
    """specroll_tree_attn.  Returns O (and lse when asked).
    ``check_status`` also calls specroll_workspace_status (synchronises the stream)."""
    out, lse, workspace = _n().tree_attn(Q, Kc, Vc, kv_indptr_dev, kv_indptr_host, Kt, Vt, parent, scale, want_lse, workspace,
                                         out, lse, flags)
    if check_status:
        _check(workspace_status(workspace), "specroll_workspace_status")
    return (out, lse) if want_lse else out


def tree_attn_paged_workspace_bytes(B, N, Hq, Hkv, D, kv_len_host, scale=None) -> int:
    kl = _host_i32(kv_len_host, "kv_len_host")
    desc = AttnDesc(B, N, Hq, Hkv, D, scale if scale is not None else 1.0 / float(np.sqrt(D)), 0)
    return int(lib().specroll_tree_attn_paged_workspace_bytes(C.byref(desc), kl.ctypes.data_as(C.c_void_p)))


def tree_attn_paged(Q, Kp, Vp, page_table, page_indptr, kv_len_dev, kv_len_host, Kt, Vt, parent, scale=None,
                    want_lse=False, workspace=None, out=None, lse=None, flags: int = 0, check_status: bool = False):
    """specroll_tree_attn_paged.  Kp, Vp: [n_pages, 128, Hkv, D]; page_table, page_indptr, kv_len_dev: device
    int32; kv_len_host: host copy of the lengths.  Returns O (and lse when asked)."""
    out, lse, workspace = _n().tree_attn_paged(Q, Kp, Vp, page_table, page_indptr, kv_len_dev, kv_len_host, Kt, Vt, parent,
                                               scale, want_lse, workspace, out, lse, flags)
    if check_status:
        _check(workspace_status(workspace), "specroll_workspace_status")
    return (out, lse) if want_lse else out


def commit_path(Kt, Vt, path_node, n_acc, Kp, Vp, page_table, page_indptr, kv_len, kv_len_out=None, status=None):
    """specroll_commit_path: appends the committed path's tree rows to one layer's paged cache (in place)."""
    _n().commit_path(Kt, Vt, path_node, n_acc, Kp, Vp, page_table, page_indptr, kv_len, kv_len_out, status)


def commit_path_layers(Kt, Vt, path_node, n_acc, Kp, Vp, page_table, page_indptr, kv_len, kv_len_out=None,
                       status=None):
    """specroll_commit_path_layers: Kt, Vt, Kp, Vp are lists with one tensor per layer."""
    _n().commit_path_layers(Kt, Vt, path_node, n_acc, Kp, Vp, page_table, page_indptr, kv_len, kv_len_out, status)


def gather_hidden(hidden, term_node, out=None):
    """specroll_gather_hidden: hidden[B,N,d] bf16, term_node[B] -> h_next[B,d]."""
    return _n().gather_hidden(hidden, term_node, out)


# ----------------------------------------------------------------------------------- verify


def verify_workspace_bytes(B, N, K, k, V, temperature=1.0) -> int:
    desc = VerifyDesc(B, N, K, k, V, temperature, 0)
    return int(lib().specroll_verify_workspace_bytes(C.byref(desc)))


def verify_nucleus_workspace_bytes(B, N, K, k, V, temperature=1.0) -> int:
    desc = VerifyDesc(B, N, K, k, V, temperature, 0)
    return int(lib().specroll_verify_nucleus_workspace_bytes(C.byref(desc)))


def verify(logits, parent, tree_tok, tree_cand, cand_id, cand_logit, u_acc, u_fin, temperature=1.0,
           workspace=None, out: Optional[Dict[str, torch.Tensor]] = None, flags: int = 0) -> Dict[str, torch.Tensor]:
    """specroll_verify.  Device tensors in, dict of device tensors out."""
    return _n().verify(logits, parent, tree_tok, tree_cand, cand_id, cand_logit, u_acc, u_fin, temperature, workspace, out,
                       flags)


def verify_fused(hidden, W, parent, tree_tok, tree_cand, cand_id, cand_logit, u_acc, u_fin, temperature=1.0):
    """Exact verification from the target's final hidden states, without the logits tensor: the projection with
    fused row statistics and tile masses over all (sequence, node) rows (specroll_target_head_stats_tiles), then the walk
    on the target logits of the candidate tokens and the terminal draw from the one vocabulary tile that holds its
    token (specroll_verify_hidden).
    hidden [B, N, d] bf16, W [V, d] bf16; the other arguments as for ``verify``.  Returns the same dict."""
    return _n().verify_fused(hidden, W, parent, tree_tok, tree_cand, cand_id, cand_logit, u_acc, u_fin, temperature)


def verify_nucleus(logits, parent, tree_tok, tree_cand, cand_id, cand_logit, u_acc, u_fin, top_p, temperature=1.0,
                   workspace=None, out: Optional[Dict[str, torch.Tensor]] = None,
                   flags: int = 0) -> Dict[str, torch.Tensor]:
    """specroll_verify_nucleus: verification against nucleus-truncated target distributions.
    The returned dict also holds nucleus_thr and nucleus_sum [B,N]."""
    return _n().verify_nucleus(logits, parent, tree_tok, tree_cand, cand_id, cand_logit, u_acc, u_fin, top_p, temperature,
                               workspace, out, flags)


def reflex_feedback_workspace_bytes(R, k, k_support, d, V, temperature=1.0, eps=1e-6) -> int:
    desc = FeedbackDesc(R, k, k_support, d, V, temperature, eps, 0, 0.0)
    return int(lib().specroll_reflex_feedback_workspace_bytes(C.byref(desc)))


def reflex_feedback(logits, rec_row, row_max, row_sum, cand_id, cand_logit, y_star, W, rho, rec_mem, m, k_support,
                    temperature=1.0, eps=1e-6, workspace=None, severity_min=None, want_e=False):
    """specroll_reflex_feedback(_ex): verifier feedback of R matured records, memory ``m`` updated in place.
    logits [rows, V] bf16 (any leading shape), row_max/row_sum [rows]; returns d_dist, d_cov, tv, severity [R]
    (and e [R, d] with ``want_e``).  With ``severity_min`` the update is weighted by the severity and
    observations below it are discarded."""
    return _n().reflex_feedback(logits, rec_row, row_max, row_sum, cand_id, cand_logit, y_star, W, rho, rec_mem, m, k_support,
                                temperature, eps, workspace, severity_min, want_e)


def reflex_sketch(X, Pi, rows=None):
    """specroll_reflex_sketch: normalised random-projection sketches [R, rank] of the rows of X [*, d] fp32
    (``rows`` [R] i32 selects them; all rows in order when None) under the projection Pi [rank, d] fp32."""
    return _n().reflex_sketch(X, Pi, rows)


def reflex_gate(s, xi, slot, keep, n, mean, M2, n_fb, m, horizon, n_align_min, n_fb_min, alpha_lo, alpha_hi,
                z_delta=0.60, mem_eps=1e-12):
    """specroll_reflex_gate: alignments of R matured records into the slots' online moments (n, mean, M2, n_fb
    updated in place), then the reliability score and the correction ratio of every slot.  Returns a [R],
    rel [S], alpha [S]."""
    return _n().reflex_gate(s, xi, slot, keep, n, mean, M2, n_fb, m, horizon, n_align_min, n_fb_min, alpha_lo, alpha_hi,
                            z_delta, mem_eps)


def target_head_stats(H, W, want_id=None, temperature=1.0, workspace=None):
    """specroll_target_head_stats: row_max, row_sum [R] and want_logit [R, kw] (bf16) of l = bf16(H W^T) without
    storing l.  H [R, d] bf16, W [V, d] bf16, want_id [R, kw] i32 or None."""
    return _n().target_head_stats(H, W, want_id, temperature, workspace)


def target_head_rows(H, W, out=None):
    """specroll_target_head_rows: logits [R, V] bf16 = bf16(H W^T)."""
    return _n().target_head_rows(H, W, out)


def verify_static(logits, parent, tree_tok, tree_cand, cand_id, cand_logit, u_acc, u_fin, temperature=1.0,
                  out: Dict[str, torch.Tensor] = None) -> Dict[str, torch.Tensor]:
    """specroll_verify_static: verification for hosts that cannot allocate a workspace.

    The scratch is a fixed array inside the library, so this wrapper passes none.  The output
    tensors must be supplied by a caller that truly cannot allocate (``out``); when ``out`` is
    omitted they are created here with torch for convenience, which is the only allocation on
    this path and is the caller's, not the library's.  Raises SpecrollError with the library's
    message when B or B*k exceed the entry point's fixed limits.
    """
    return _n().verify_static(logits, parent, tree_tok, tree_cand, cand_id, cand_logit, u_acc, u_fin, temperature, out)


# ----------------------------------------------------------------------------------- helpers


def bf16_tensor(bits: np.ndarray, device="cuda") -> torch.Tensor:
    """uint16 bf16 bit patterns (host numpy) -> bf16 tensor on the device."""
    t = torch.from_numpy(np.ascontiguousarray(bits).view(np.int16))
    return t.view(torch.bfloat16).to(device)


def bf16_bits(t: torch.Tensor) -> np.ndarray:
    """bf16 tensor -> uint16 bit patterns on the host."""
    return t.detach().contiguous().view(torch.int16).cpu().numpy().view(np.uint16)
