"""Binding of ``librocs.so`` (declared in ``include/rocs.h``).

Argument marshalling only: torch supplies device memory and streams, every step of the
computation runs inside the library's CUDA kernels.  There is no CPU or eager fallback: if the
library is missing or a call fails, an exception is raised.  The calls of a scoring loop go through
the extension ``_native`` (``csrc/binding.cpp``), the rest through ctypes.

Functions mirror the C entry points (``rocs_`` prefix dropped): :func:`plan_create`,
:func:`ikbo_linear`, :func:`linear`, :func:`dca_attention`, :func:`glm_interaction`.
bf16 tensors are ``torch.bfloat16``, fp32 tensors ``torch.float32``.
"""
from __future__ import annotations

import ctypes
import os
from typing import Optional

import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "librocs.so")
_lib = None
_ext = None

OK = 0
BF16, F32 = 0, 1
ACT_NONE, ACT_RELU = 0, 1
PATH_AUTO, PATH_GENERAL = 0, 1
NORM_LAYER, NORM_RMS = 0, 1

EXPORTS = [
    "rocs_status_string", "rocs_padded_ld", "rocs_set_path", "rocs_plan_create", "rocs_plan_destroy",
    "rocs_ikbo_linear_workspace", "rocs_ikbo_linear", "rocs_linear", "rocs_dca_attention_workspace",
    "rocs_dca_attention", "rocs_glm_interaction_workspace", "rocs_glm_interaction",
    "rocs_glm_fm_projection_workspace", "rocs_glm_fm_projection", "rocs_group_norm",
    "rocs_last_device_status", "rocs_ikbo_linear_static", "rocs_ikbo_linear_static_max_z_elems",
    "rocs_ikbo_linear_static_max_candidates", "rocs_ikbo_linear_stats_workspace", "rocs_ikbo_linear_stats",
    "rocs_weight_row_sums", "rocs_linear_normed",
]


class RocsError(RuntimeError):
    def __init__(self, code: int, where: str):
        self.code = code
        super().__init__(f"{where}: {status_string(code)} ({code})")


def lib() -> ctypes.CDLL:
    """Loads librocs.so on first use; raises if it has not been built."""
    global _lib
    if _lib is None:
        if not os.path.exists(LIB_PATH):
            raise RuntimeError(
                f"{LIB_PATH} is missing: build it with `python -m paper_2607_27744_b200.build` "
                "(there is no fallback path)")
        L = ctypes.CDLL(LIB_PATH)
        vp, i32, i64, f32, sz = ctypes.c_void_p, ctypes.c_int32, ctypes.c_int64, ctypes.c_float, ctypes.c_size_t
        L.rocs_status_string.restype = ctypes.c_char_p
        L.rocs_status_string.argtypes = [ctypes.c_int]
        L.rocs_padded_ld.restype = i64
        L.rocs_padded_ld.argtypes = [i64, ctypes.c_int]
        L.rocs_set_path.argtypes = [ctypes.c_int]
        L.rocs_plan_create.argtypes = [ctypes.POINTER(vp), i32, i64, vp, vp, vp]
        L.rocs_plan_destroy.argtypes = [vp]
        L.rocs_ikbo_linear_workspace.restype = sz
        L.rocs_ikbo_linear_workspace.argtypes = [vp, i32]
        L.rocs_ikbo_linear.argtypes = [vp, ctypes.c_int, i32, i32, i32, vp, i64, vp, i64, vp, i64, vp, i64,
                                       vp, ctypes.c_int, vp, i64, vp, sz, vp]
        L.rocs_linear.argtypes = [ctypes.c_int, i64, i32, i32, vp, i64, vp, i64, vp, ctypes.c_int, vp, i64, vp]
        L.rocs_dca_attention_workspace.restype = sz
        L.rocs_dca_attention_workspace.argtypes = [vp, i32, i32, i32]
        L.rocs_dca_attention.argtypes = [vp, ctypes.c_int, i32, i32, i32, f32, vp, vp, vp, i64, vp, vp, vp, sz, vp]
        L.rocs_glm_interaction_workspace.restype = sz
        L.rocs_glm_interaction_workspace.argtypes = [vp, i32, i32, i32]
        L.rocs_glm_interaction.argtypes = [vp, ctypes.c_int, i32, i32, i32, vp, vp, vp, i32, i32, vp, vp, vp, vp,
                                           vp, sz, vp]
        L.rocs_glm_fm_projection_workspace.restype = sz
        L.rocs_glm_fm_projection_workspace.argtypes = [vp, i32, i32]
        L.rocs_glm_fm_projection.argtypes = [vp, ctypes.c_int, i32, i32, i32, i32, vp, vp, vp, vp, vp, vp, sz, vp]
        L.rocs_group_norm.argtypes = [ctypes.c_int, ctypes.c_int, i64, i32, vp, i64, vp, vp, f32, vp, i64, vp]
        L.rocs_last_device_status.argtypes = [ctypes.POINTER(ctypes.c_uint32)]
        L.rocs_ikbo_linear_stats_workspace.restype = sz
        L.rocs_ikbo_linear_stats_workspace.argtypes = [vp, i32]
        L.rocs_ikbo_linear_stats.argtypes = [vp, ctypes.c_int, i32, i32, i32, vp, i64, vp, i64, vp, i64, vp, i64,
                                             vp, ctypes.c_int, vp, i64, vp, vp, sz, vp]
        L.rocs_weight_row_sums.argtypes = [ctypes.c_int, i32, i32, vp, i64, vp, vp]
        L.rocs_linear_normed.argtypes = [ctypes.c_int, ctypes.c_int, i64, i32, i32, vp, i64, vp, f32, vp, i64, vp, vp,
                                         ctypes.c_int, vp, i64, vp]
        L.rocs_ikbo_linear_static_max_z_elems.restype = sz
        L.rocs_ikbo_linear_static_max_candidates.restype = sz
        L.rocs_ikbo_linear_static.argtypes = [ctypes.c_int, i32, i64, vp, i32, i32, i32, vp, i64, vp, i64, vp, i64,
                                              vp, i64, vp, ctypes.c_int, vp, i64, vp]
        _lib = L
    return _lib


def status_string(code: int) -> str:
    return lib().rocs_status_string(code).decode()


def _check(code: int, where: str):
    if code != OK:
        raise RocsError(code, where)


def padded_ld(n: int, dtype: int) -> int:
    return int(lib().rocs_padded_ld(n, dtype))


def set_path(path: int):
    _check(lib().rocs_set_path(path), "rocs_set_path")


def last_device_status() -> int:
    """Synchronises, then raises RocsError if a bounded device-side wait expired."""
    detail = ctypes.c_uint32(0)
    code = lib().rocs_last_device_status(ctypes.byref(detail))
    if code != OK:
        raise RocsError(code, f"device status word 0x{detail.value:08x}")
    return detail.value


def _native():
    """Loads the extension on first use; raises if it (or the library it calls) has not been built."""
    global _ext
    lib()
    try:
        from . import _native as ext
    except ImportError as e:
        raise RuntimeError(f"the extension _native is missing or broken ({e}): build it with "
                           "`python -m paper_2607_27744_b200.build` (there is no fallback path)") from e
    ext.set_error_type(RocsError)
    _ext = ext
    return ext


class Plan:
    """Owns a ``rocs_plan_t`` (Section 4.1: the request-candidate map in segment form)."""

    def __init__(self, cand_offsets: torch.Tensor, cand_offsets_host=None):
        self.handle = None
        self.cand_offsets = cand_offsets
        host = cand_offsets_host
        if host is None:
            host = cand_offsets.cpu()
        elif not (isinstance(host, torch.Tensor) and host.dtype is torch.int32 and host.is_contiguous()):
            host = torch.as_tensor(host, dtype=torch.int32).contiguous()
        self._host = host
        self.handle, self.R, self.N = (_ext or _native()).plan_create(cand_offsets, host)

    def close(self):
        handle, self.handle = self.handle, None
        if handle:
            _ext.plan_destroy(handle)

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass


def plan_create(cand_offsets: torch.Tensor, cand_offsets_host=None) -> Plan:
    return Plan(cand_offsets, cand_offsets_host)


def ikbo_linear_workspace(plan: Plan, d_out: int) -> int:
    return int(lib().rocs_ikbo_linear_workspace(plan.handle, d_out))


def ikbo_linear(plan: Plan, XR: Optional[torch.Tensor], XC: torch.Tensor, W_CR: Optional[torch.Tensor],
                W_CC: torch.Tensor, bias: Optional[torch.Tensor] = None, relu: bool = False,
                out: Optional[torch.Tensor] = None, workspace: Optional[torch.Tensor] = None) -> torch.Tensor:
    """Y_i = act(Z[m_i] + X^C_i W_CC^T), Z = X^R W_CR^T + bias (Eq. 14).  W_CR / W_CC may be column
    slices of one [d_out, d_req + d_cand] weight."""
    return (_ext or _native()).ikbo_linear(plan.handle, plan.R, plan.N, XR, XC, W_CR, W_CC, bias, relu, out, workspace)


def ikbo_linear_stats(plan: Plan, XR: torch.Tensor, XC: torch.Tensor, W_CR: torch.Tensor, W_CC: torch.Tensor,
                      bias: Optional[torch.Tensor] = None, relu: bool = False, out: Optional[torch.Tensor] = None,
                      row_stats: Optional[torch.Tensor] = None, workspace: Optional[torch.Tensor] = None):
    """ikbo_linear that also leaves each output row's (sum, sum of squares) for a normalisation folded
    into the next layer (Eq. 7).  Returns (Y, row_stats [N, 2] fp32)."""
    return (_ext or _native()).ikbo_linear_stats(plan.handle, plan.R, plan.N, XR, XC, W_CR, W_CC, bias, relu, out, row_stats,
                                                 workspace)


def weight_row_sums(W: torch.Tensor, out: Optional[torch.Tensor] = None) -> torch.Tensor:
    """wbar[n] = sum_k W[n, k] in fp32: the W 1 term of a LayerNorm folded into the layer."""
    return (_ext or _native()).weight_row_sums(W, out)


def linear_normed(X: torch.Tensor, row_stats: torch.Tensor, W: torch.Tensor, wbar: Optional[torch.Tensor] = None,
                  bias: Optional[torch.Tensor] = None, eps: float = 1e-5, kind: int = NORM_LAYER, relu: bool = False,
                  out: Optional[torch.Tensor] = None) -> torch.Tensor:
    """Y = act(norm(X) W^T + bias) with the normalisation applied to the layer's accumulators (Eq. 7
    folded into the epilogue); gamma and beta are folded into W and bias by the caller."""
    return (_ext or _native()).linear_normed(X, row_stats, W, wbar, bias, eps, kind, relu, out)


def linear(X: torch.Tensor, W: torch.Tensor, bias: Optional[torch.Tensor] = None, relu: bool = False,
           out: Optional[torch.Tensor] = None) -> torch.Tensor:
    """Y = act(X W^T + bias), the one-group case of Eq. 4."""
    return (_ext or _native()).linear(X, W, bias, relu, out)


def dca_attention(plan: Plan, Q: torch.Tensor, K: torch.Tensor, V: torch.Tensor, seq_offsets: torch.Tensor,
                  scale: float = 0.0, out: Optional[torch.Tensor] = None) -> torch.Tensor:
    """Candidate-side cross attention over the request's shared K/V (Eq. 13).
    Q [N, n_q, H, dh]; K, V [T, H, dh]; seq_offsets int32 [R+1] on the device."""
    return (_ext or _native()).dca_attention(plan.handle, plan.R, plan.N, Q, K, V, seq_offsets, scale, out)


def glm_interaction_workspace(plan: Plan, n_r: int, n_c: int, n_co: int) -> int:
    return int(lib().rocs_glm_interaction_workspace(plan.handle, n_r, n_c, n_co))


def glm_interaction(plan: Plan, XR: torch.Tensor, XC: torch.Tensor, W: Optional[torch.Tensor] = None,
                    n_ro: int = 0, n_co: int = 0, want_raw: bool = True, want_request_side: bool = True,
                    workspace: Optional[torch.Tensor] = None, outs: Optional[dict] = None) -> dict:
    """GLM factorization machine (Eq. 9-10) with optional row-axis compression (Eq. 5-6).
    Returns a dict with the tensors that were requested among YR, YC, OR, OC."""
    R, n_r, _ = XR.shape
    N, n_c, _ = XC.shape
    n = n_r + n_c
    outs = dict(outs) if outs else {}

    def fill(key, *shape):
        if key not in outs:
            outs[key] = torch.empty(shape, dtype=XC.dtype, device=XC.device)

    if want_raw:
        if want_request_side:
            fill("YR", R, n_r, n)
        fill("YC", N, n_c, n)
    if W is not None:
        if want_request_side:
            fill("OR", R, n_ro, n)
        fill("OC", N, n_co, n)
    (_ext or _native()).glm_interaction(plan.handle, plan.R, plan.N, XR, XC, W, n_ro, n_co, outs.get("YR"), outs.get("YC"),
                                        outs.get("OR"), outs.get("OC"), workspace)
    return outs


def glm_fm_projection_workspace(plan: Plan, d: int, k: int) -> int:
    return int(lib().rocs_glm_fm_projection_workspace(plan.handle, d, k))


def glm_fm_projection(plan: Plan, XR: torch.Tensor, XC: torch.Tensor, P: torch.Tensor,
                      want_request_side: bool = True, workspace: Optional[torch.Tensor] = None,
                      outs: Optional[dict] = None) -> dict:
    """GLM factorization machine (Eq. 9-10) projected to k columns, F = G P with P [n_r + n_c, k].
    Returns a dict with FC [N, n_c, k] and, if requested, FR [R, n_r, k]."""
    k = P.shape[1]
    outs = dict(outs) if outs else {}
    if want_request_side and "FR" not in outs:
        outs["FR"] = torch.empty((XR.shape[0], XR.shape[1], k), dtype=XC.dtype, device=XC.device)
    if "FC" not in outs:
        outs["FC"] = torch.empty((XC.shape[0], XC.shape[1], k), dtype=XC.dtype, device=XC.device)
    (_ext or _native()).glm_fm_projection(plan.handle, plan.R, plan.N, XR, XC, P, outs.get("FR"), outs.get("FC"), workspace)
    return outs


def group_norm(X: torch.Tensor, gamma: Optional[torch.Tensor] = None, beta: Optional[torch.Tensor] = None,
               eps: float = 1e-5, kind: int = NORM_LAYER, out: Optional[torch.Tensor] = None) -> torch.Tensor:
    """Group-local LayerNorm / RMSNorm (Eq. 7) of one group's tensor X [M, d], row by row."""
    return (_ext or _native()).group_norm(X, gamma, beta, eps, kind, out)


def ikbo_linear_static(cand_offsets: torch.Tensor, XR: torch.Tensor, XC: torch.Tensor, W_CR: torch.Tensor,
                       W_CC: torch.Tensor, out: torch.Tensor, bias: Optional[torch.Tensor] = None,
                       relu: bool = False) -> torch.Tensor:
    """The split linear layer through ``rocs_ikbo_linear_static``: no plan, no workspace, and the call
    allocates nothing -- for hosts that cannot call cudaMalloc while scoring.  The caller passes the
    output tensor; scratch lives in a fixed array inside the library (limits: R * d_out <= 1 Mi,
    N <= 256 Ki; calls share the array, so do not let two of them overlap on the GPU)."""
    return (_ext or _native()).ikbo_linear_static(cand_offsets, XR, XC, W_CR, W_CC, out, bias, relu)
