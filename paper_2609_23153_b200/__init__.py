"""Python binding of the sparkattn C-ABI library (``libsparkattn.so``).

Argument marshalling only, for the per-layer calls in native code
(``_sparkattn.so``, ``csrc/binding.cpp``), for the others through ctypes: every
step of the path (block selection, FP8 quantisation, block-sparse attention)
runs in the CUDA kernels behind the ``extern "C"`` entry points declared in
``include/sparkattn.h``.  PyTorch is used for device memory and streams.  There
is no CPU fallback: if the shared library is missing or cannot be loaded, every call raises.
"""
from __future__ import annotations

import ctypes
import os
from typing import Optional, Tuple

import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "libsparkattn.so")
VERSION = 1

OK = 0
E_INVALID_ARG = -1
E_UNSUPPORTED_SHAPE = -2
E_MISALIGNED = -3
E_WORKSPACE_TOO_SMALL = -4
E_CUDA = -5
E_DEVICE_TIMEOUT = -6
E_BAD_INDEX = -7
E_NO_DEVICE = -8

BF16 = 0
FP8_E4M3 = 1

EXPORTS = (
    "sparkattn_version", "sparkattn_status_string", "sparkattn_workspace_bytes", "sparkattn_select",
    "sparkattn_quant_fp8", "sparkattn_quant_fp8_per_token", "sparkattn_fwd", "sparkattn_read_status", "sparkattn_arena_bytes",
    "sparkattn_attention_host", "sparkattn_select_noalloc", "sparkattn_select_noalloc_max_bytes",
    "sparkattn_select_noalloc_status", "sparkattn_comp_workspace_bytes", "sparkattn_comp_state",
    "sparkattn_comp_apply", "sparkattn_select_window", "sparkattn_fwd_window", "sparkattn_brick_count",
    "sparkattn_brick_layout", "sparkattn_gather_tokens", "sparkattn_select_padded", "sparkattn_fwd_padded",
    "sparkattn_quant_fp8_pooled", "sparkattn_select_pooled", "sparkattn_fwd_gated_workspace_bytes", "sparkattn_fwd_gated",
)


class Shape(ctypes.Structure):
    """Mirror of ``sparkattn_shape_t``."""
    _fields_ = [
        ("struct_size", ctypes.c_uint32), ("version", ctypes.c_uint32),
        ("B", ctypes.c_int32), ("H", ctypes.c_int32), ("N", ctypes.c_int32), ("d", ctypes.c_int32),
        ("block", ctypes.c_int32), ("reserved", ctypes.c_int32),
        ("stride_b", ctypes.c_int64), ("stride_h", ctypes.c_int64), ("stride_n", ctypes.c_int64),
        ("softmax_scale", ctypes.c_float), ("pad", ctypes.c_uint32),
    ]


_SHAPE_BYTES = ctypes.sizeof(Shape)


class SparkAttnError(RuntimeError):
    def __init__(self, status: int, where: str):
        self.status = status
        super().__init__(f"{where}: {status_string(status)} ({status})")


# What the native marshalling of the per-layer calls (csrc/binding.cpp) calls, in its order.
_BOUND = ("workspace_bytes", "select", "select_window", "select_padded", "select_pooled", "quant_fp8", "quant_fp8_pooled",
          "quant_fp8_per_token", "fwd", "fwd_window", "fwd_padded", "gather_tokens", "comp_workspace_bytes", "comp_state", "comp_apply",
          "fwd_gated_workspace_bytes", "fwd_gated")
_NO_WORKSPACE = 1        # the library does not serve the shape: the workspace query returned 0

_lib = None
_native = None


def lib() -> ctypes.CDLL:
    """Loads the shared library (once).  Raises if it has not been built."""
    global _lib, _native
    if _lib is None:
        if not os.path.exists(LIB_PATH):
            raise ImportError(
                f"{LIB_PATH} is missing: build it with `python -m paper_2609_23153_b200.build` "
                "(there is no fallback path)")
        L = ctypes.CDLL(LIB_PATH)
        vp, i32, sz = ctypes.c_void_p, ctypes.c_int32, ctypes.c_size_t
        sp = ctypes.POINTER(Shape)
        L.sparkattn_version.restype = ctypes.c_int
        L.sparkattn_status_string.restype = ctypes.c_char_p
        L.sparkattn_status_string.argtypes = [ctypes.c_int]
        L.sparkattn_workspace_bytes.restype = sz
        L.sparkattn_workspace_bytes.argtypes = [sp, i32, i32]
        L.sparkattn_select.restype = ctypes.c_int
        L.sparkattn_select.argtypes = [sp, vp, vp, i32, vp, vp, vp, sz, vp]
        L.sparkattn_quant_fp8.restype = ctypes.c_int
        L.sparkattn_quant_fp8.argtypes = [sp, vp, vp, vp, ctypes.c_uint32, vp]
        L.sparkattn_quant_fp8_pooled.restype = ctypes.c_int
        L.sparkattn_quant_fp8_pooled.argtypes = [sp, vp, vp, vp, i32, vp, sz, vp]
        L.sparkattn_select_pooled.restype = ctypes.c_int
        L.sparkattn_select_pooled.argtypes = [sp, i32, vp, vp, vp, sz, vp]
        L.sparkattn_quant_fp8_per_token.restype = ctypes.c_int
        L.sparkattn_quant_fp8_per_token.argtypes = [sp, vp, vp, vp, vp]
        L.sparkattn_fwd.restype = ctypes.c_int
        L.sparkattn_fwd.argtypes = [sp, i32, vp, vp, vp, vp, vp, vp, vp, vp, i32, vp, vp, vp, sz, vp]
        L.sparkattn_read_status.restype = ctypes.c_int
        L.sparkattn_read_status.argtypes = [vp, vp]
        L.sparkattn_brick_count.restype = ctypes.c_int64
        L.sparkattn_brick_count.argtypes = [vp, vp]
        L.sparkattn_brick_layout.restype = ctypes.c_int
        L.sparkattn_brick_layout.argtypes = [vp, vp, i32, vp, vp, vp, vp]
        L.sparkattn_gather_tokens.restype = ctypes.c_int
        L.sparkattn_gather_tokens.argtypes = [sp, vp, sp, vp, vp, vp, sz, vp]
        L.sparkattn_select_padded.restype = ctypes.c_int
        L.sparkattn_select_padded.argtypes = [sp, vp, vp, i32, vp, vp, vp, vp, sz, vp]
        L.sparkattn_fwd_padded.restype = ctypes.c_int
        L.sparkattn_fwd_padded.argtypes = [sp, i32, vp, vp, vp, vp, vp, vp, vp, vp, i32, vp, vp, vp, vp, sz, vp]
        L.sparkattn_arena_bytes.restype = sz
        L.sparkattn_arena_bytes.argtypes = [sp, i32, i32]
        L.sparkattn_attention_host.restype = ctypes.c_int
        L.sparkattn_attention_host.argtypes = [sp, i32, vp, vp, vp, i32, vp, vp, vp, sz, vp]
        L.sparkattn_select_noalloc.restype = ctypes.c_int
        L.sparkattn_select_noalloc.argtypes = [sp, vp, vp, i32, vp, vp, vp]
        L.sparkattn_select_noalloc_max_bytes.restype = sz
        L.sparkattn_select_noalloc_status.restype = ctypes.c_int
        L.sparkattn_select_noalloc_status.argtypes = [vp]
        L.sparkattn_select_window.restype = ctypes.c_int
        L.sparkattn_select_window.argtypes = [sp, vp, vp, i32, i32, i32, vp, vp, vp, sz, vp]
        L.sparkattn_fwd_window.restype = ctypes.c_int
        L.sparkattn_fwd_window.argtypes = [sp, i32, vp, vp, vp, vp, vp, vp, vp, vp, i32, i32, i32, vp, vp, vp, sz, vp]
        L.sparkattn_comp_workspace_bytes.restype = sz
        L.sparkattn_comp_workspace_bytes.argtypes = [sp, vp]
        L.sparkattn_comp_state.restype = ctypes.c_int
        L.sparkattn_comp_state.argtypes = [sp, vp, vp, vp, i32, vp, vp, vp, vp, vp, sz, vp]
        L.sparkattn_comp_apply.restype = ctypes.c_int
        L.sparkattn_comp_apply.argtypes = [sp, vp, vp, i32, vp, vp, vp, vp, vp, vp, vp, ctypes.c_float, vp, sz, vp]
        L.sparkattn_fwd_gated_workspace_bytes.restype = sz
        L.sparkattn_fwd_gated_workspace_bytes.argtypes = [sp, i32, vp]
        L.sparkattn_fwd_gated.restype = ctypes.c_int
        L.sparkattn_fwd_gated.argtypes = [sp, vp, vp, vp, vp, vp, i32, vp, i32, vp, vp, vp, vp, vp, ctypes.c_float, vp,
                                          vp, vp, sz, vp]
        from . import _sparkattn
        _sparkattn.bind(*(ctypes.cast(getattr(L, "sparkattn_" + name), vp).value for name in _BOUND))
        _native = _sparkattn
        _lib = L
    return _lib


def _calls():
    if _lib is None:
        lib()
    return _native


def status_string(status: int) -> str:
    return lib().sparkattn_status_string(int(status)).decode()


def _check(rc: int, where: str) -> None:
    if rc != OK:
        if rc == _NO_WORKSPACE:
            raise SparkAttnError(E_UNSUPPORTED_SHAPE, "sparkattn_workspace_bytes")
        raise SparkAttnError(rc, where)


# The current stream's handle alone: building a torch.cuda.Stream object around it takes 3.4 us, a seventh of a small
# call.  The name is not part of torch's public interface: where it is missing the public way is taken.
_raw_stream = getattr(torch._C, "_cuda_getCurrentRawStream", None)


def _stream_ptr(stream: Optional[torch.cuda.Stream]) -> int:
    if stream is None and _raw_stream is not None:
        return _raw_stream(torch.cuda.current_device())
    return (torch.cuda.current_stream() if stream is None else stream).cuda_stream


def _ptr(t: Optional[torch.Tensor]) -> Optional[int]:
    return None if t is None else t.data_ptr()


def make_shape(x: torch.Tensor, block: int, softmax_scale: float = 0.0) -> Shape:
    """Shape descriptor for a [B, H, N, d] tensor (d contiguous, arbitrary outer strides)."""
    stride = x.stride()
    if len(stride) != 4 or stride[3] != 1:
        raise ValueError("expected a [B, H, N, d] tensor with a contiguous last dimension")
    B, H, N, d = x.shape
    return Shape(_SHAPE_BYTES, VERSION, B, H, N, d, block, 0, stride[0], stride[1], stride[2], float(softmax_scale), 0)


def _same_layout(ref: torch.Tensor, *others: torch.Tensor) -> None:
    for o in others:
        if o.shape != ref.shape or o.stride() != ref.stride():
            raise ValueError("tensors of one call must share shape and strides")


def workspace_bytes(shape: Shape, which: int, topk_or_kmax: int) -> int:
    return int(lib().sparkattn_workspace_bytes(ctypes.byref(shape), which, topk_or_kmax))


def alloc_workspace(shape: Shape, which: int, topk_or_kmax: int, device) -> torch.Tensor:
    n = workspace_bytes(shape, which, topk_or_kmax)
    if n == 0:
        raise SparkAttnError(E_UNSUPPORTED_SHAPE, "sparkattn_workspace_bytes")
    return torch.empty(n, dtype=torch.uint8, device=device)


def read_status(workspace: torch.Tensor, stream: Optional[torch.cuda.Stream] = None) -> int:
    return int(lib().sparkattn_read_status(_ptr(workspace), _stream_ptr(stream)))


def select(q: torch.Tensor, k: torch.Tensor, block: int, topk: int, *,
           kept_idx: Optional[torch.Tensor] = None, kept_cnt: Optional[torch.Tensor] = None,
           workspace: Optional[torch.Tensor] = None, stream: Optional[torch.cuda.Stream] = None,
           frame_tokens: int = 0, window: int = 0, block_valid: Optional[torch.Tensor] = None,
           ) -> Tuple[torch.Tensor, torch.Tensor]:
    """``sparkattn_select`` (``sparkattn_select_window`` when ``frame_tokens`` > 0, ``sparkattn_select_padded``
    with ``block_valid``, device int32 [nb]): q, k bf16 [B,H,N,d] on the device -> (kept_idx int32
    [B,H,nb,topk] ascending, kept_cnt int32 [B,H,nb])."""
    if block_valid is not None and frame_tokens > 0:
        raise ValueError("block_valid and a causal window cannot be combined")
    rc, kept_idx, kept_cnt = _calls().select(q, k, block, topk, kept_idx, kept_cnt, workspace,
                                             None if stream is None else stream.cuda_stream, frame_tokens, window, block_valid)
    if rc != OK:
        _check(rc, "sparkattn_select_padded" if block_valid is not None else
               "sparkattn_select_window" if frame_tokens > 0 else "sparkattn_select")
    return kept_idx, kept_cnt


def select_noalloc(q: torch.Tensor, k: torch.Tensor, block: int, topk: int, kept_idx: torch.Tensor,
                   kept_cnt: Optional[torch.Tensor], stream: Optional[torch.cuda.Stream] = None) -> None:
    """``sparkattn_select_noalloc``: same selection as :func:`select`, for callers that
    must not allocate device memory at call time.  The caller passes the output
    buffers; the scratch is a fixed 32 MiB array inside the library, shared by all
    calls on the device (do not overlap calls; make the first call on a device
    before any stream capture)."""
    _same_layout(q, k)
    shape = make_shape(q, block)
    rc = lib().sparkattn_select_noalloc(ctypes.byref(shape), _ptr(q), _ptr(k), topk, _ptr(kept_idx), _ptr(kept_cnt),
                                        _stream_ptr(stream))
    _check(rc, "sparkattn_select_noalloc")


def quant_fp8(x: torch.Tensor, block: int, *, codes: Optional[torch.Tensor] = None,
              scales: Optional[torch.Tensor] = None, stream: Optional[torch.cuda.Stream] = None,
              ) -> Tuple[torch.Tensor, torch.Tensor]:
    """``sparkattn_quant_fp8``: x bf16 [B,H,N,d] -> (codes uint8, same strides; scales fp32 [B,H,nb])."""
    rc, codes, scales = _calls().quant_fp8(x, block, codes, scales, None if stream is None else stream.cuda_stream)
    _check(rc, "sparkattn_quant_fp8")
    return codes, scales


def quant_fp8_pooled(x: torch.Tensor, block: int, key_side: bool, select_workspace: torch.Tensor, *,
                     codes: Optional[torch.Tensor] = None, scales: Optional[torch.Tensor] = None,
                     stream: Optional[torch.cuda.Stream] = None) -> Tuple[torch.Tensor, torch.Tensor]:
    """``sparkattn_quant_fp8_pooled``: :func:`quant_fp8` that also leaves the pooled block means of ``x`` (the query
    tensor, or the key tensor with ``key_side``) in ``select_workspace`` for :func:`select_pooled`."""
    rc, codes, scales = _calls().quant_fp8_pooled(x, block, key_side, select_workspace, codes, scales,
                                                  None if stream is None else stream.cuda_stream)
    _check(rc, "sparkattn_quant_fp8_pooled")
    return codes, scales


def select_pooled(ref: torch.Tensor, block: int, topk: int, workspace: torch.Tensor, *,
                  kept_idx: Optional[torch.Tensor] = None, kept_cnt: Optional[torch.Tensor] = None,
                  stream: Optional[torch.cuda.Stream] = None) -> Tuple[torch.Tensor, torch.Tensor]:
    """``sparkattn_select_pooled``: scores + top-k on the pooled means two :func:`quant_fp8_pooled` calls left in
    ``workspace``; ``ref`` is any [B,H,N,d] tensor of the problem (for the shape)."""
    rc, kept_idx, kept_cnt = _calls().select_pooled(ref, block, topk, workspace, kept_idx, kept_cnt,
                                                    None if stream is None else stream.cuda_stream)
    _check(rc, "sparkattn_select_pooled")
    return kept_idx, kept_cnt


def quant_fp8_per_token(x: torch.Tensor, *, codes: Optional[torch.Tensor] = None,
                        scales: Optional[torch.Tensor] = None, stream: Optional[torch.cuda.Stream] = None,
                        ) -> Tuple[torch.Tensor, torch.Tensor]:
    """``sparkattn_quant_fp8_per_token``: x bf16 [B,H,N,d] -> (codes uint8, same strides; scales fp32 [B,H,N])."""
    rc, codes, scales = _calls().quant_fp8_per_token(x, codes, scales, None if stream is None else stream.cuda_stream)
    _check(rc, "sparkattn_quant_fp8_per_token")
    return codes, scales


def fwd(q: torch.Tensor, k: torch.Tensor, v: torch.Tensor, kept_idx: torch.Tensor,
        kept_cnt: Optional[torch.Tensor], block: int, *,
        scales: Optional[Tuple[torch.Tensor, torch.Tensor, torch.Tensor]] = None,
        softmax_scale: float = 0.0, out: Optional[torch.Tensor] = None, return_lse: bool = False,
        workspace: Optional[torch.Tensor] = None, stream: Optional[torch.cuda.Stream] = None,
        check_status: bool = False, frame_tokens: int = 0, window: int = 0,
        block_valid: Optional[torch.Tensor] = None):
    """``sparkattn_fwd`` (``sparkattn_fwd_window`` when ``frame_tokens`` > 0, ``sparkattn_fwd_padded`` with
    ``block_valid``, device int32 [nb]).  bf16 q,k,v, or uint8
    E4M3 codes with ``scales=(q_scale, k_scale, v_scale)``.  Returns out bf16 [B,H,N,d] (and lse
    fp32 [B,H,N])."""
    if block_valid is not None and frame_tokens > 0:
        raise ValueError("block_valid and a causal window cannot be combined")
    sq, sk, sv = scales if scales is not None else (None, None, None)
    rc, out, lse, workspace = _calls().fwd(q, k, v, kept_idx, kept_cnt, block, BF16 if scales is None else FP8_E4M3, sq, sk, sv,
                                           softmax_scale, out, return_lse, workspace,
                                           None if stream is None else stream.cuda_stream, frame_tokens, window, block_valid)
    _check(rc, "sparkattn_fwd")
    if check_status:
        _check(read_status(workspace, stream), "sparkattn_fwd (device status)")
    return (out, lse) if return_lse else out


def brick_layout(grid, brick, block: int, device="cuda:0", stream: Optional[torch.cuda.Stream] = None):
    """``sparkattn_brick_layout``: (gather int32 [bricks * block] with -1 for padding, block_valid int32 [bricks],
    scatter int32 [N]) for a (T, Hg, Wg) grid cut into (bt, bh, bw) bricks, one block per brick."""
    g = (ctypes.c_int32 * 3)(*[int(v) for v in grid])
    b = (ctypes.c_int32 * 3)(*[int(v) for v in brick])
    bricks = int(lib().sparkattn_brick_count(ctypes.cast(g, ctypes.c_void_p), ctypes.cast(b, ctypes.c_void_p)))
    if bricks == 0:
        raise SparkAttnError(E_INVALID_ARG, "sparkattn_brick_count")
    n = int(grid[0]) * int(grid[1]) * int(grid[2])
    gather = torch.empty(bricks * block, dtype=torch.int32, device=device)
    valid = torch.empty(bricks, dtype=torch.int32, device=device)
    scatter = torch.empty(n, dtype=torch.int32, device=device)
    rc = lib().sparkattn_brick_layout(ctypes.cast(g, ctypes.c_void_p), ctypes.cast(b, ctypes.c_void_p), block, _ptr(gather),
                                      _ptr(valid), _ptr(scatter), _stream_ptr(stream))
    _check(rc, "sparkattn_brick_layout")
    return gather, valid, scatter


def gather_tokens(x: torch.Tensor, index: torch.Tensor, *, out: Optional[torch.Tensor] = None,
                  workspace: Optional[torch.Tensor] = None, stream: Optional[torch.cuda.Stream] = None,
                  check_status: bool = False) -> torch.Tensor:
    """``sparkattn_gather_tokens``: out[b,h,i,:] = x[b,h,index[i],:] (zero row for index -1); x bf16 [B,H,N,d],
    index int32 [N_out] on the device, out bf16 [B,H,N_out,d]."""
    rc, out, workspace = _calls().gather_tokens(x, index, out, workspace, None if stream is None else stream.cuda_stream)
    _check(rc, "sparkattn_gather_tokens")
    if check_status:
        _check(read_status(workspace, stream), "sparkattn_gather_tokens (device status)")
    return out


def arena_bytes(shape: Shape, dtype: int, topk: int) -> int:
    return int(lib().sparkattn_arena_bytes(ctypes.byref(shape), dtype, topk))


def attention_host(q: torch.Tensor, k: torch.Tensor, v: torch.Tensor, block: int, topk: int, *,
                   dtype: int = BF16, out: Optional[torch.Tensor] = None,
                   kept_idx: Optional[torch.Tensor] = None, arena: Optional[torch.Tensor] = None,
                   device="cuda:0", stream: Optional[torch.cuda.Stream] = None) -> torch.Tensor:
    """``sparkattn_attention_host``: q, k, v contiguous bf16 HOST tensors (pinned for
    speed); runs copy-in, select, (quant,) fwd, copy-out and returns the host output."""
    for t in (q, k, v):
        if t.device.type != "cpu" or not t.is_contiguous() or t.dtype != torch.bfloat16:
            raise ValueError("attention_host expects contiguous bf16 CPU tensors")
    shape = make_shape(q, block)
    if out is None:
        out = torch.empty_like(q).pin_memory()
    if arena is None:
        arena = torch.empty(arena_bytes(shape, dtype, topk), dtype=torch.uint8, device=device)
    rc = lib().sparkattn_attention_host(ctypes.byref(shape), dtype, _ptr(q), _ptr(k), _ptr(v), topk, _ptr(out),
                                        _ptr(kept_idx), _ptr(arena), arena.numel(), _stream_ptr(stream))
    _check(rc, "sparkattn_attention_host")
    return out


def comp_workspace_bytes(shape: Shape, grid) -> int:
    g = (ctypes.c_int32 * 3)(*[int(x) for x in grid])
    return int(lib().sparkattn_comp_workspace_bytes(ctypes.byref(shape), g))


def comp_state(k: torch.Tensor, v: torch.Tensor, pk: torch.Tensor, grid, axis: torch.Tensor, freq: torch.Tensor, *,
               state: Optional[torch.Tensor] = None, workspace: Optional[torch.Tensor] = None,
               stream: Optional[torch.cuda.Stream] = None, check_status: bool = False) -> torch.Tensor:
    """``sparkattn_comp_state``: k, v bf16 [B,H,N,d]; pk bf16 [H,r,d]; grid (T,Hg,Wg); axis/freq the
    rotary tables (rank/2 entries, any device).  Returns the state fp32 [B,H,r,d]."""
    T, Hg, Wg = grid
    rc, state, workspace = _calls().comp_state(k, v, pk, int(T), int(Hg), int(Wg), axis, freq, state, workspace,
                                               None if stream is None else stream.cuda_stream)
    _check(rc, "sparkattn_comp_state")
    if check_status:
        _check(read_status(workspace, stream), "sparkattn_comp_state (device status)")
    return state


def comp_apply(q: torch.Tensor, pq: torch.Tensor, state: torch.Tensor, gate: torch.Tensor, o_sparse: torch.Tensor,
               grid, axis: torch.Tensor, freq: torch.Tensor, *, eps: float = 1e-6,
               out: Optional[torch.Tensor] = None, workspace: Optional[torch.Tensor] = None,
               stream: Optional[torch.cuda.Stream] = None, check_status: bool = False) -> torch.Tensor:
    """``sparkattn_comp_apply``: q, o_sparse bf16 [B,H,N,d]; pq bf16 [H,r,d]; state fp32 [B,H,r,d];
    gate fp32 [B,H,N].  Returns the fused output bf16 [B,H,N,d]."""
    T, Hg, Wg = grid
    rc, out, workspace = _calls().comp_apply(q, pq, state, gate, o_sparse, int(T), int(Hg), int(Wg), axis, freq, eps, out, workspace,
                                             None if stream is None else stream.cuda_stream)
    _check(rc, "sparkattn_comp_apply")
    if check_status:
        _check(read_status(workspace, stream), "sparkattn_comp_apply (device status)")
    return out


def fwd_gated_workspace_bytes(shape: Shape, kmax: int, grid) -> int:
    g = (ctypes.c_int32 * 3)(*[int(x) for x in grid])
    return int(lib().sparkattn_fwd_gated_workspace_bytes(ctypes.byref(shape), kmax, g))


def fwd_gated(q: torch.Tensor, k: torch.Tensor, v: torch.Tensor, kept_idx: torch.Tensor,
              kept_cnt: Optional[torch.Tensor], pq: torch.Tensor, state: torch.Tensor, gate: torch.Tensor,
              grid, axis: torch.Tensor, freq: torch.Tensor, *, eps: float = 1e-6, softmax_scale: float = 0.0,
              out: Optional[torch.Tensor] = None, return_lse: bool = False, workspace: Optional[torch.Tensor] = None,
              stream: Optional[torch.cuda.Stream] = None, check_status: bool = False):
    """``sparkattn_fwd_gated``: the bf16 forward over 128-token blocks whose epilogue adds the gated
    compensation term.  Arguments as in ``fwd`` and ``comp_apply``; returns the module output bf16
    [B,H,N,d] (and the lse of the sparse branch, fp32 [B,H,N])."""
    T, Hg, Wg = grid
    rc, out, lse, workspace = _calls().fwd_gated(q, k, v, kept_idx, kept_cnt, pq, state, gate, int(T), int(Hg), int(Wg), axis, freq,
                                                 eps, softmax_scale, out, return_lse, workspace,
                                                 None if stream is None else stream.cuda_stream)
    _check(rc, "sparkattn_fwd_gated")
    if check_status:
        _check(read_status(workspace, stream), "sparkattn_fwd_gated (device status)")
    return (out, lse) if return_lse else out
