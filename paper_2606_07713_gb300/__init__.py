"""DNF attention forward for GB300 (sm_103a).

O = softmax(scale * Q K^T) V with a max-subtracted softmax, computed without any
score, probability or transposed-K array in device memory (the Denotational
Normal Form of Mullin & Hains, "Attention at the Theoretical Minimum").

The computation runs in libmoa_attn.so (hand-written CUDA: a tcgen05/TMEM/TMA
kernel for bf16 and a CUDA-core kernel for fp32).  This package is its thin
Python binding: PyTorch supplies device memory and the current stream, nothing
else.  There is no CPU fallback.
"""
from __future__ import annotations

import math

from ._lib import (MOA_BF16, MOA_FP32, MoaError, check, lib, moa_attn_dnf_bytes,  # noqa: F401
                   moa_attn_flops, moa_attn_fwd, moa_attn_fwd_staged, moa_attn_version,
                   moa_get_device_status, moa_last_error, moa_selftest_wait_timeout,
                   moa_attn_fwd_splitkv, moa_attn_splitkv_workspace_bytes, moa_attn_fwd_lse,
                   moa_attn_bwd, moa_attn_bwd_workspace_bytes, moa_qkv_proj,
                   moa_attn_split_plan, MOA_SPLITS_AUTO, moa_attn_bwd_fused,
                   moa_attn_bwd_fused_workspace_bytes, moa_attn_bwd_fused_plan)

__all__ = ["attn_fwd", "attn_fwd_staged", "get_device_status", "attn_flops", "dnf_bytes",
           "MOA_FP32", "MOA_BF16", "MoaError", "moa_attn_fwd", "moa_attn_fwd_staged",
           "moa_last_error", "moa_get_device_status", "moa_attn_flops", "moa_attn_dnf_bytes",
           "moa_attn_version", "moa_selftest_wait_timeout", "attn_fwd_splitkv",
           "moa_attn_fwd_splitkv", "moa_attn_splitkv_workspace_bytes", "attn_fwd_lse",
           "moa_attn_fwd_lse", "attn_bwd", "moa_attn_bwd", "moa_attn_bwd_workspace_bytes",
           "qkv_proj", "moa_qkv_proj", "moa_attn_split_plan", "MOA_SPLITS_AUTO",
           "moa_attn_bwd_fused", "moa_attn_bwd_fused_workspace_bytes", "moa_attn_bwd_fused_plan"]


_torch = None  # the torch module, bound by the first call (the package imports without torch)


def _bind_torch():
    global _torch
    import torch
    _torch = torch
    return torch


def _dtype_code(t) -> int:
    torch = _torch or _bind_torch()
    dt = t.dtype
    if dt is torch.bfloat16:
        return MOA_BF16
    if dt is torch.float32:
        return MOA_FP32
    raise TypeError(f"unsupported dtype {dt}; use torch.bfloat16 or torch.float32")


def _dims(q, k, v):
    qs, ks, vs = q.shape, k.shape, v.shape
    if len(qs) != 4 or len(ks) != 4 or len(vs) != 4:
        raise ValueError("q, k, v must be [B, H, N, d]")
    B, H, Nq, dk = qs
    kb, kh, Nk, kd = ks
    vb, vh, vn, dv = vs
    if kb != B or kh != H or vb != B or vh != H:
        raise ValueError(f"batch/head mismatch: {tuple(qs)} {tuple(ks)} {tuple(vs)}")
    if kd != dk or vn != Nk:
        raise ValueError(f"shape mismatch: {tuple(qs)} {tuple(ks)} {tuple(vs)}")
    return B, H, Nq, Nk, dk, dv


def _call(fn, device, stream, *args) -> None:
    """fn(*args, stream) on `device` (stream None: torch's current one); raises on a non-OK status.
    A small call is bound by this host path: the raw stream handle and the current-device test take
    0.3 us where a Stream object and a device guard took 3.6 us."""
    torch = _torch or _bind_torch()
    index = device.index
    s = torch._C._cuda_getCurrentRawStream(index) if stream is None else stream.cuda_stream
    if torch._C._cuda_getDevice() == index:
        status = fn(*args, s)
    else:
        with torch.cuda.device(device):
            status = fn(*args, s)
    if status != 0:
        check(status)


def attn_fwd(q, k, v, scale: float | None = None, out=None, stream=None):
    """O = softmax(scale * q k^T) v for CUDA tensors [B, H, N, d] (bf16 or fp32).

    scale defaults to 1/sqrt(d_k).  Runs asynchronously on `stream` (default:
    torch's current stream of q's device) and returns `out` (allocated if None).
    """
    for t in (q, k, v):
        if not t.is_cuda:
            raise ValueError("attn_fwd needs CUDA tensors")
        if not t.is_contiguous():
            raise ValueError("attn_fwd needs contiguous tensors")
    if not (q.dtype == k.dtype == v.dtype):
        raise TypeError("q, k, v must share one dtype")
    code = _dtype_code(q)
    B, H, Nq, Nk, dk, dv = _dims(q, k, v)
    if scale is None:
        scale = 1.0 / math.sqrt(dk)
    device = q.device
    if out is None:
        out = _torch.empty((B, H, Nq, dv), dtype=q.dtype, device=device)
    elif out.shape != (B, H, Nq, dv) or out.dtype != q.dtype or not out.is_contiguous():
        raise ValueError("out has the wrong shape, dtype or layout")
    _call(lib().moa_attn_fwd, device, stream, q.data_ptr(), k.data_ptr(), v.data_ptr(),
          out.data_ptr(), B, H, Nq, Nk, dk, dv, float(scale), code)
    return out


def attn_fwd_lse(q, k, v, scale: float | None = None, out=None, lse=None, stream=None):
    """(O, LSE): attn_fwd's output and the float32 [B, H, N_q] natural-log log-sum-exp of each
    row's scaled scores, ln sum_k exp(scale <q_i, k_k>)."""
    for t in (q, k, v):
        if not t.is_cuda or not t.is_contiguous():
            raise ValueError("attn_fwd_lse needs contiguous CUDA tensors")
    if not (q.dtype == k.dtype == v.dtype):
        raise TypeError("q, k, v must share one dtype")
    code = _dtype_code(q)
    B, H, Nq, Nk, dk, dv = _dims(q, k, v)
    if scale is None:
        scale = 1.0 / math.sqrt(dk)
    device = q.device
    if out is None:
        out = _torch.empty((B, H, Nq, dv), dtype=q.dtype, device=device)
    elif out.shape != (B, H, Nq, dv) or out.dtype != q.dtype or not out.is_contiguous():
        raise ValueError("out has the wrong shape, dtype or layout")
    if lse is None:
        lse = _torch.empty((B, H, Nq), dtype=_torch.float32, device=device)
    elif lse.shape != (B, H, Nq) or lse.dtype != _torch.float32 or not lse.is_contiguous():
        raise ValueError("lse must be a contiguous float32 [B, H, N_q] tensor")
    _call(lib().moa_attn_fwd_lse, device, stream, q.data_ptr(), k.data_ptr(), v.data_ptr(),
          out.data_ptr(), lse.data_ptr(), B, H, Nq, Nk, dk, dv, float(scale), code)
    return out, lse


def attn_bwd(q, k, v, o, lse, do, scale: float | None = None, workspace=None, stream=None,
             fused: bool = False):
    """(dQ, dK, dV) for O = softmax(scale q k^T) v given dO = dL/dO, from the forward's o and lse
    (attn_fwd_lse).  CUDA tensors [B, H, N, d]; lse float32 [B, H, N_q].  fused=True runs
    moa_attn_bwd_fused (bf16, d_k = d_v = 64; the key blocks' dQ tiles are added in fp32 by TMA
    reductions, in a run-dependent order)."""
    for t in (q, k, v, o, do, lse):
        if not t.is_cuda or not t.is_contiguous():
            raise ValueError("attn_bwd needs contiguous CUDA tensors")
    if not (q.dtype == k.dtype == v.dtype == o.dtype == do.dtype):
        raise TypeError("q, k, v, o, do must share one dtype")
    code = _dtype_code(q)
    B, H, Nq, Nk, dk, dv = _dims(q, k, v)
    if tuple(o.shape) != (B, H, Nq, dv) or tuple(do.shape) != (B, H, Nq, dv):
        raise ValueError("o and do must be [B, H, N_q, d_v]")
    if tuple(lse.shape) != (B, H, Nq) or lse.dtype != _torch.float32:
        raise ValueError("lse must be float32 [B, H, N_q]")
    if scale is None:
        scale = 1.0 / math.sqrt(dk)
    dq = _torch.empty_like(q)
    dkk = _torch.empty_like(k)
    dvv = _torch.empty_like(v)
    L = lib()
    wsb = L.moa_attn_bwd_fused_workspace_bytes if fused else L.moa_attn_bwd_workspace_bytes
    fn = L.moa_attn_bwd_fused if fused else L.moa_attn_bwd
    device = q.device
    if workspace is None:
        need = wsb(B, H, Nq, Nk, dk, dv, code)
        workspace = _torch.empty(max(need, 16), dtype=_torch.uint8, device=device)
    _call(fn, device, stream, q.data_ptr(), k.data_ptr(), v.data_ptr(), o.data_ptr(), do.data_ptr(),
          lse.data_ptr(), dq.data_ptr(), dkk.data_ptr(), dvv.data_ptr(), B, H, Nq, Nk, dk, dv,
          float(scale), code, workspace.data_ptr(), workspace.numel())
    return dq, dkk, dvv


def qkv_proj(x, w, H: int, d_k: int, d_v: int, out=None, stream=None):
    """(Q, K, V) = (X W_Q, X W_K, X W_V) in head-major layout [B, H, N, d] from x [B, N, d_model]
    and w [d_model, 2*H*d_k + H*d_v] (W_Q | W_K | W_V), bf16 CUDA tensors."""
    for t in (x, w):
        if not t.is_cuda or not t.is_contiguous():
            raise ValueError("qkv_proj needs contiguous CUDA tensors")
    if x.dim() != 3 or w.dim() != 2:
        raise ValueError("x must be [B, N, d_model] and w [d_model, 2*H*d_k + H*d_v]")
    if x.dtype != w.dtype:
        raise TypeError("x and w must share one dtype")
    code = _dtype_code(x)
    B, N, d = x.shape
    if tuple(w.shape) != (d, 2 * H * d_k + H * d_v):
        raise ValueError(f"w must be {(d, 2 * H * d_k + H * d_v)}, got {tuple(w.shape)}")
    device, dtype = x.device, x.dtype
    if out is None:
        out = (_torch.empty((B, H, N, d_k), dtype=dtype, device=device),
               _torch.empty((B, H, N, d_k), dtype=dtype, device=device),
               _torch.empty((B, H, N, d_v), dtype=dtype, device=device))
    q, k, v = out
    _call(lib().moa_qkv_proj, device, stream, x.data_ptr(), w.data_ptr(), q.data_ptr(),
          k.data_ptr(), v.data_ptr(), B, N, d, H, d_k, d_v, code)
    return q, k, v


def attn_fwd_splitkv(q, k, v, num_splits: int = MOA_SPLITS_AUTO, scale: float | None = None,
                     out=None, workspace=None, stream=None):
    """attn_fwd with the key axis split into up to num_splits ranges merged at the end.  With
    MOA_SPLITS_AUTO (0) the library chooses from q's device: when the 256-row query blocks leave
    SMs idle, every block's key axis is split so that the CTAs fill the SMs (if its cost model
    predicts a saving); otherwise nothing is split and the result is attn_fwd's.  The workspace
    (a CUDA uint8 tensor of at least moa_attn_splitkv_workspace_bytes(...) bytes) is allocated
    here when not given."""
    for t in (q, k, v):
        if not t.is_cuda or not t.is_contiguous():
            raise ValueError("attn_fwd_splitkv needs contiguous CUDA tensors")
    if not (q.dtype == k.dtype == v.dtype):
        raise TypeError("q, k, v must share one dtype")
    code = _dtype_code(q)
    B, H, Nq, Nk, dk, dv = _dims(q, k, v)
    if scale is None:
        scale = 1.0 / math.sqrt(dk)
    device = q.device
    if out is None:
        out = _torch.empty((B, H, Nq, dv), dtype=q.dtype, device=device)
    L, splits = lib(), int(num_splits)
    if workspace is None:
        if _torch._C._cuda_getDevice() == device.index:
            need = L.moa_attn_splitkv_workspace_bytes(B, H, Nq, Nk, dk, dv, code, splits)
        else:  # MOA_SPLITS_AUTO reads the current device
            with _torch.cuda.device(device):
                need = L.moa_attn_splitkv_workspace_bytes(B, H, Nq, Nk, dk, dv, code, splits)
        workspace = _torch.empty(max(need, 16), dtype=_torch.uint8, device=device)
    _call(L.moa_attn_fwd_splitkv, device, stream, q.data_ptr(), k.data_ptr(), v.data_ptr(),
          out.data_ptr(), B, H, Nq, Nk, dk, dv, float(scale), code, splits, workspace.data_ptr(),
          workspace.numel())
    return out


def attn_fwd_staged(hq, hk, hv, ho, dq, dk_, dv_, do, scale: float | None = None, stream=None):
    """Host tensors in, host tensor out: copies hq/hk/hv to the device buffers dq/dk_/dv_,
    runs the kernel into do and copies it back into ho, all on one stream.  The result is in
    ho after the stream is synchronised."""
    code = _dtype_code(dq)
    B, H, Nq, Nk, dk, dv = _dims(dq, dk_, dv_)
    for h, d in ((hq, dq), (hk, dk_), (hv, dv_), (ho, do)):
        if h.is_cuda or not d.is_cuda or h.shape != d.shape or h.dtype != d.dtype:
            raise ValueError("staged call needs matching host and device tensors")
        if not (h.is_contiguous() and d.is_contiguous()):
            raise ValueError("staged call needs contiguous tensors")
    if scale is None:
        scale = 1.0 / math.sqrt(dk)
    _call(lib().moa_attn_fwd_staged, dq.device, stream, hq.data_ptr(), hk.data_ptr(), hv.data_ptr(),
          ho.data_ptr(), dq.data_ptr(), dk_.data_ptr(), dv_.data_ptr(), do.data_ptr(), B, H, Nq, Nk,
          dk, dv, float(scale), code)
    return ho


def get_device_status(stream=None) -> int:
    """Synchronises the stream and returns/clears the kernels' timeout status word."""
    import torch
    s = stream if stream is not None else torch.cuda.current_stream()
    return moa_get_device_status(s.cuda_stream)


def attn_flops(B, H, N_q, N_k, d_k, d_v) -> float:
    return moa_attn_flops(B, H, N_q, N_k, d_k, d_v)


def dnf_bytes(B, H, N_q, N_k, d_k, d_v, dtype: int) -> float:
    return moa_attn_dnf_bytes(B, H, N_q, N_k, d_k, d_v, dtype)
