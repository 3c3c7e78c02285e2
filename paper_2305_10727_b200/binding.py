"""Thin Python binding of libgpusq.so: argument marshalling only.

Every function has the name of the C entry point it calls (without the
``gpusq_`` prefix), takes CUDA ``torch`` tensors, allocates the outputs with
torch when the caller does not pass them, enqueues on torch's current stream
and returns without synchronising.  All arithmetic runs in the CUDA kernels.
A missing library or a non-zero status raises; there is no fallback.  The
functions that run per inference or per weight do their checks, allocations
and the call in ``_gpusq_torch.so`` (csrc/torch_binding.cpp); the rest goes
through ctypes.
"""
from __future__ import annotations

import ctypes
import os
from typing import Optional

import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "libgpusq.so")

ACT_NONE, ACT_GELU = 0, 1
OUT_F16, OUT_I8, OUT_I32 = 0, 1, 2
SCALE_COMPUTE, SCALE_GIVEN = 0, 1

EXPORTS = (
    "gpusq_status_string", "gpusq_prune24", "gpusq_quant_weight", "gpusq_compress24",
    "gpusq_decompress24", "gpusq_packed_bytes", "gpusq_pack24", "gpusq_quant_act_workspace",
    "gpusq_quant_act", "gpusq_quant_act_static", "gpusq_patch_quant", "gpusq_spgemm_i8", "gpusq_gemm_i8_dense", "gpusq_set_block_tokens", "gpusq_set_tile_mix", "gpusq_set_tile_runs", "gpusq_tile_plan", "gpusq_set_quant_act_wait", "gpusq_set_quant_act_late", "gpusq_quant_act_shares_taken", "gpusq_set_gemm_wait", "gpusq_set_max_clusters",
    "gpusq_spgemm_i8_absmax", "gpusq_quant_act_absmax",
    "gpusq_prune48", "gpusq_quant_weight4", "gpusq_compress48", "gpusq_expand48", "gpusq_quant_act4",
    "gpusq_compress24_f16", "gpusq_packed_bytes_f16", "gpusq_pack24_f16", "gpusq_spgemm_f16",
)

_lib = None
_raw_stream, _current_device = torch._C._cuda_getCurrentRawStream, torch._C._cuda_getDevice


class GpusqError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        super().__init__("%s failed: %s" % (where, status_string(status)))


def load() -> ctypes.CDLL:
    """Load libgpusq.so (built in-tree by ``build.py``); raises if it is missing."""
    global _lib
    if _lib is not None:
        return _lib
    if not os.path.exists(LIB_PATH):
        raise RuntimeError(
            "libgpusq.so not found at %s: build it with `python -m paper_2305_10727_b200.build` "
            "(there is no CPU fallback)" % LIB_PATH)
    lib = ctypes.CDLL(LIB_PATH)
    vp, i32, i64, sz = ctypes.c_void_p, ctypes.c_int, ctypes.c_int64, ctypes.c_size_t
    lib.gpusq_status_string.argtypes = [i32]
    lib.gpusq_status_string.restype = ctypes.c_char_p
    lib.gpusq_prune24.argtypes = [vp, vp, vp, i32, i32, vp]
    lib.gpusq_quant_weight.argtypes = [vp, vp, vp, i32, i32, vp]
    lib.gpusq_compress24.argtypes = [vp, vp, vp, i32, i32, vp]
    lib.gpusq_decompress24.argtypes = [vp, vp, vp, i32, i32, vp]
    lib.gpusq_packed_bytes.argtypes = [i32, i32]
    lib.gpusq_packed_bytes.restype = sz
    lib.gpusq_pack24.argtypes = [vp, vp, vp, i32, i32, vp]
    lib.gpusq_quant_act_workspace.argtypes = [i64, i32]
    lib.gpusq_quant_act_workspace.restype = sz
    lib.gpusq_quant_act.argtypes = [vp, vp, vp, i32, i64, i32, vp, sz, vp]
    lib.gpusq_quant_act_static.argtypes = [vp, vp, vp, i32, i64, i32, vp]
    lib.gpusq_patch_quant.argtypes = [vp, vp, vp, i32, i32, i32, i32, i32, i32, i32, vp, sz, vp]
    gemm_args = [vp, vp, vp, vp, vp, i32, i32, vp, vp, i64, i32, i32, vp, vp]
    lib.gpusq_spgemm_i8.argtypes = gemm_args
    lib.gpusq_gemm_i8_dense.argtypes = gemm_args
    lib.gpusq_spgemm_i8_absmax.argtypes = [vp, vp, vp, vp, vp, i32, vp, vp, i64, i32, i32, vp, vp]
    lib.gpusq_quant_act_absmax.argtypes = [vp, vp, vp, vp, i64, i32, vp]
    lib.gpusq_prune48.argtypes = [vp, vp, vp, i32, i32, vp]
    lib.gpusq_quant_weight4.argtypes = [vp, vp, vp, i32, i32, vp]
    lib.gpusq_compress48.argtypes = [vp, vp, vp, i32, i32, vp]
    lib.gpusq_expand48.argtypes = [vp, vp, vp, vp, i32, i32, vp]
    lib.gpusq_quant_act4.argtypes = [vp, vp, vp, i32, i64, i32, vp, sz, vp]
    lib.gpusq_set_block_tokens.argtypes = [i32]
    lib.gpusq_set_tile_mix.argtypes = [i32, i32]
    lib.gpusq_set_tile_runs.argtypes = [i32, i32, i32]
    lib.gpusq_tile_plan.argtypes = [i64, i32, i32, i32, i32, i32, vp]
    lib.gpusq_set_quant_act_wait.argtypes = [ctypes.c_ulonglong, i32]
    lib.gpusq_set_quant_act_late.argtypes = [i32, i32, ctypes.c_uint]
    lib.gpusq_quant_act_shares_taken.argtypes = [vp]
    lib.gpusq_set_gemm_wait.argtypes = [ctypes.c_uint, i32]
    lib.gpusq_set_max_clusters.argtypes = [i32]
    lib.gpusq_compress24_f16.argtypes = [vp, vp, vp, i32, i32, vp]
    lib.gpusq_packed_bytes_f16.argtypes = [i32, i32]
    lib.gpusq_packed_bytes_f16.restype = sz
    lib.gpusq_pack24_f16.argtypes = [vp, vp, vp, i32, i32, vp]
    lib.gpusq_spgemm_f16.argtypes = [vp, vp, vp, i32, i32, vp, i64, i32, i32, vp, vp]
    for name in EXPORTS:
        if name not in ("gpusq_status_string", "gpusq_packed_bytes", "gpusq_packed_bytes_f16",
                        "gpusq_quant_act_workspace"):
            getattr(lib, name).restype = i32
    _lib = lib
    return lib


_native = None


def _n():
    """The native part of this binding; raises if it or libgpusq.so is missing, or built for another torch or Python."""
    global _native
    if _native is None:
        load()
        from . import _gpusq_torch, build
        if _gpusq_torch.built_for != build.built_for():
            raise RuntimeError("_gpusq_torch.so was built for %s, this is %s: build it with `python -m paper_2305_10727_b200.build`"
                               % (_gpusq_torch.built_for, build.built_for()))
        _gpusq_torch.set_errors(GpusqError, torch.OutOfMemoryError)
        _native = _gpusq_torch
    return _native


def status_string(status: int) -> str:
    return load().gpusq_status_string(int(status)).decode()


def _check(status: int, where: str) -> None:
    if status != 0:
        raise GpusqError(status, where)


# For the calls that go through ctypes.  Addresses are passed as plain integers (the argument types convert
# them) and the stream is asked for as its handle: a pointer object per argument and a Stream object per
# call cost 5 us.
def _ptr(t: Optional[torch.Tensor]):
    return None if t is None else t.data_ptr()


def _stream() -> int:
    return _raw_stream(_current_device())


def _dev(t: torch.Tensor, dtype, what: str) -> torch.Tensor:
    if not t.is_cuda or t.dtype != dtype or not t.is_contiguous():
        raise ValueError("%s must be a contiguous CUDA tensor of dtype %s" % (what, dtype))
    return t


def prune24(W: torch.Tensor, Wp: Optional[torch.Tensor] = None, mask: Optional[torch.Tensor] = None,
            want_mask: bool = False):
    return _n().prune24(W, Wp, mask, bool(want_mask))


def quant_weight(Wp: torch.Tensor, Wq: Optional[torch.Tensor] = None, w_scale: Optional[torch.Tensor] = None):
    return _n().quant_weight(Wp, Wq, w_scale)


def compress24(Wq: torch.Tensor, vals: Optional[torch.Tensor] = None, meta: Optional[torch.Tensor] = None):
    return _n().compress24(Wq, vals, meta)


def decompress24(vals: torch.Tensor, meta: torch.Tensor, Wq: Optional[torch.Tensor] = None):
    _dev(vals, torch.int8, "vals")
    _dev(meta, torch.uint8, "meta")
    N, K = vals.shape[0], vals.shape[1] * 2
    if Wq is None:
        Wq = torch.empty((N, K), dtype=torch.int8, device=vals.device)
    _check(load().gpusq_decompress24(_ptr(vals), _ptr(meta), _ptr(Wq), N, K, _stream()), "gpusq_decompress24")
    return Wq


def packed_bytes(N: int, K: int) -> int:
    return int(load().gpusq_packed_bytes(N, K))


def pack24(vals: torch.Tensor, meta: torch.Tensor, Wpacked: Optional[torch.Tensor] = None):
    return _n().pack24(vals, meta, Wpacked)


def quant_act_workspace(M: int, K: int) -> int:
    return int(load().gpusq_quant_act_workspace(M, K))


def quant_act(X: torch.Tensor, Xq: Optional[torch.Tensor] = None, x_scale: Optional[torch.Tensor] = None,
              scale_mode: int = SCALE_COMPUTE, workspace: Optional[torch.Tensor] = None):
    return _n().quant_act(X, Xq, x_scale, scale_mode, workspace)


QUANT_ACT_STATUS_OFFSET = 8196       # GPUSQ_QUANT_ACT_STATUS_OFFSET of gpusq.h


def quant_act_status(workspace: torch.Tensor) -> int:
    """The status word gpusq_quant_act keeps in its workspace (0, or 7 = a bounded wait expired).  Synchronises."""
    word = workspace.view(torch.uint8)[QUANT_ACT_STATUS_OFFSET:QUANT_ACT_STATUS_OFFSET + 4].view(torch.int32)
    return int(word.cpu().item())


def set_quant_act_wait(limit_ns: int, withhold_last_cta: bool = False) -> None:
    """Test hook (gpusq_testing.h): bound of the one-launch kernel's waits; optionally plant an arrival that never comes."""
    _check(load().gpusq_set_quant_act_wait(int(limit_ns), 1 if withhold_last_cta else 0), "gpusq_set_quant_act_wait")


def set_quant_act_late(first: int, count: int, ns: int) -> None:
    """Test hook (gpusq_testing.h): CTAs [first, first + count) of the one-launch kernel start ns nanoseconds late."""
    _check(load().gpusq_set_quant_act_late(int(first), int(count), int(ns)), "gpusq_set_quant_act_late")


def quant_act_shares_taken() -> int:
    """Test hook (gpusq_testing.h): shares of the one-launch kernel taken over so far.  Synchronises."""
    n = ctypes.c_uint(0)
    _check(load().gpusq_quant_act_shares_taken(ctypes.byref(n)), "gpusq_quant_act_shares_taken")
    return n.value


def set_gemm_wait(limit_us: int, withhold_loads: bool = False) -> None:
    """Test hook (gpusq_testing.h): bound of the GEMM kernels' waits; optionally plant loads that never come."""
    _check(load().gpusq_set_gemm_wait(int(limit_us), 1 if withhold_loads else 0), "gpusq_set_gemm_wait")


def quant_act_static(X: torch.Tensor, Xq: Optional[torch.Tensor] = None, x_scale: Optional[torch.Tensor] = None,
                     scale_mode: int = SCALE_COMPUTE):
    """gpusq_quant_act_static: no workspace argument; the library's own fixed scratch is used."""
    _dev(X, torch.float16, "X")
    M, K = X.shape
    if Xq is None:
        Xq = torch.empty((M, K), dtype=torch.int8, device=X.device)
    if x_scale is None:
        if scale_mode == SCALE_GIVEN:
            raise ValueError("scale_mode GIVEN needs x_scale")
        x_scale = torch.empty((1,), dtype=torch.float32, device=X.device)
    _check(load().gpusq_quant_act_static(_ptr(X), _ptr(Xq), _ptr(x_scale), scale_mode, M, K, _stream()),
           "gpusq_quant_act_static")
    return Xq, x_scale


def patch_quant(img: torch.Tensor, P: int, Kp: Optional[int] = None, Xq: Optional[torch.Tensor] = None,
                x_scale: Optional[torch.Tensor] = None, scale_mode: int = SCALE_COMPUTE,
                workspace: Optional[torch.Tensor] = None):
    """gpusq_patch_quant: img f16 [B, C, H, W] -> (Xq i8 [B*(H/P)*(W/P), Kp], x_scale)."""
    _dev(img, torch.float16, "img")
    B, C, H, W = img.shape
    if Kp is None:
        Kp = (C * P * P + 15) // 16 * 16
    tokens = B * (H // P) * (W // P)
    if Xq is None:
        Xq = torch.empty((tokens, Kp), dtype=torch.int8, device=img.device)
    if x_scale is None:
        if scale_mode == SCALE_GIVEN:
            raise ValueError("scale_mode GIVEN needs x_scale")
        x_scale = torch.empty((1,), dtype=torch.float32, device=img.device)
    if workspace is None and scale_mode == SCALE_COMPUTE:
        workspace = torch.zeros((quant_act_workspace(tokens, Kp),), dtype=torch.uint8, device=img.device)
    ws_bytes = 0 if workspace is None else workspace.numel() * workspace.element_size()
    _check(load().gpusq_patch_quant(_ptr(img), _ptr(Xq), _ptr(x_scale), scale_mode, B, C, H, W, P, Kp,
                                    _ptr(workspace), ws_bytes, _stream()), "gpusq_patch_quant")
    return Xq, x_scale


def flatten_conv_weight(W4: torch.Tensor, Kp: Optional[int] = None) -> torch.Tensor:
    """Conv weight [D, C, P, P] -> [D, Kp] f32 row-major, zero columns beyond C*P*P (a copy, no arithmetic)."""
    D = W4.shape[0]
    K = W4[0].numel()
    if Kp is None:
        Kp = (K + 15) // 16 * 16
    Wf = torch.zeros((D, Kp), dtype=torch.float32, device=W4.device)
    Wf[:, :K] = W4.reshape(D, K)
    return Wf


def spgemm_i8(Xq: torch.Tensor, Wpacked: torch.Tensor, N: int, w_scale=None, x_scale=None, bias=None,
              act: int = ACT_NONE, out_type: int = OUT_F16, out_scale=None, Y=None, status_buf=None):
    return _n().spgemm_i8(Xq, Wpacked, N, w_scale, x_scale, bias, act, out_type, out_scale, Y, status_buf)


def spgemm_i8_absmax(Xq: torch.Tensor, Wpacked: torch.Tensor, N: int, w_scale, x_scale, bias=None,
                     act: int = ACT_NONE, Y=None, y_absmax=None, status_buf=None):
    """gpusq_spgemm_i8_absmax: FP16 output plus max |Y| merged into y_absmax (float32[1], zeroed here if not given)."""
    if y_absmax is None:
        y_absmax = torch.zeros((1,), dtype=torch.float32, device=Xq.device)
    return _n().spgemm_i8_absmax(Xq, Wpacked, N, w_scale, x_scale, bias, act, Y, y_absmax, status_buf)


def quant_act_absmax(X: torch.Tensor, absmax: torch.Tensor, Xq: Optional[torch.Tensor] = None,
                     x_scale: Optional[torch.Tensor] = None):
    """gpusq_quant_act_absmax: one-pass quantisation with the scale derived from a known max |X|."""
    return _n().quant_act_absmax(X, absmax, Xq, x_scale)


def gemm_i8_dense(Xq: torch.Tensor, Wq: torch.Tensor, w_scale=None, x_scale=None, bias=None,
                  act: int = ACT_NONE, out_type: int = OUT_F16, out_scale=None, Y=None, status_buf=None):
    _dev(Wq, torch.int8, "Wq")
    return _n().gemm_i8_dense(Xq, Wq, Wq.shape[0], w_scale, x_scale, bias, act, out_type, out_scale, Y, status_buf)


def set_block_tokens(block_t: int) -> None:
    """Test hook (gpusq_testing.h): force the GEMM tile height; 0 = automatic."""
    _check(load().gpusq_set_block_tokens(block_t), "gpusq_set_block_tokens")


def set_tile_runs(block_t: int, n_big: int, run_tiles: int) -> None:
    """Test hook (gpusq_testing.h): as set_tile_mix, in token runs of run_tiles tiles with resident weights."""
    _check(load().gpusq_set_tile_runs(int(block_t), int(n_big), int(run_tiles)), "gpusq_set_tile_runs")


def tile_plan(M: int, N: int, K: int, half: bool = False, out_type: int = OUT_F16, clusters: int = 74):
    """Test hook (gpusq_testing.h): (tokens per tile, runs of that height, runs, tiles per run) of a 2:4 launch; needs no GPU."""
    plan = (ctypes.c_int * 4)()
    _check(load().gpusq_tile_plan(int(M), int(N), int(K), int(half), int(out_type), int(clusters), plan), "gpusq_tile_plan")
    return tuple(plan)


def set_max_clusters(clusters: int) -> None:
    """Measurement hook (gpusq_testing.h): the GEMM launches use at most that many CTA pairs (0 = all)."""
    _check(load().gpusq_set_max_clusters(int(clusters)), "gpusq_set_max_clusters")


def set_tile_mix(block_t: int, n_big: int) -> None:
    """Test hook (gpusq_testing.h): n_big token tiles of block_t tokens, the rest 32 tokens lower."""
    _check(load().gpusq_set_tile_mix(block_t, n_big), "gpusq_set_tile_mix")


# ---- FP16 2:4 sparse model ----
OUT_F32 = 2


def compress24_f16(Wp: torch.Tensor):
    return _n().compress24_f16(Wp)


def packed_bytes_f16(N: int, K: int) -> int:
    return int(load().gpusq_packed_bytes_f16(N, K))


def pack24_f16(vals: torch.Tensor, meta: torch.Tensor, Wpacked: Optional[torch.Tensor] = None):
    return _n().pack24_f16(vals, meta, Wpacked)


def spgemm_f16(X: torch.Tensor, Wpacked: torch.Tensor, N: int, bias=None, act: int = ACT_NONE,
               out_type: int = OUT_F16, Y=None, status_buf=None):
    return _n().spgemm_f16(X, Wpacked, N, bias, act, out_type, Y, status_buf)


# ---- INT4 model (pair-wise 4:8 sparsity) ----

def prune48(W: torch.Tensor, want_mask: bool = False):
    return _n().prune48(W, bool(want_mask))


def quant_weight4(Wp: torch.Tensor):
    return _n().quant_weight4(Wp, None, None)


def compress48(Wq: torch.Tensor):
    return _n().compress48(Wq)


def expand48(vals4: torch.Tensor, meta4: torch.Tensor):
    """(vals4, meta4) of the 4-bit format -> (vals, meta) of the 2:4 INT8 format, columns regrouped."""
    return _n().expand48(vals4, meta4)


def quant_act4(X: torch.Tensor, Xq: Optional[torch.Tensor] = None, x_scale: Optional[torch.Tensor] = None,
               scale_mode: int = SCALE_COMPUTE, workspace: Optional[torch.Tensor] = None):
    """gpusq_quant_act4: 4-bit activation codes (INT8 containers) in the regrouped column order."""
    return _n().quant_act4(X, Xq, x_scale, scale_mode, workspace)