"""Binding of the C-ABI CUDA library (``libmixdq.so``).

Argument marshalling only: torch tensors supply device memory and the current stream,
every step of the path runs in the library's kernels.  There is no CPU fallback: if the
shared library is missing the first call raises.

The layer calls and the tensor helpers that a program runs per step (``NATIVE``) are functions of the extension module
``_mixdq_native`` (``csrc/bind.cpp``), loaded at the first use of one of them; their signatures stand in their
docstrings.  Sizes, plans and the parity hooks go through ctypes.
"""
from __future__ import annotations

import ctypes as C
import os
from typing import Optional

import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "libmixdq.so")

LAYOUT_CANONICAL = 0
LAYOUT_DEVICE = 1
TOKENS_PER_PROMPT = 77

_i64, _int, _vp, _sz = C.c_int64, C.c_int, C.c_void_p, C.c_size_t

_SIGNATURES = {
    "mixdq_version": (C.c_int, []),
    "mixdq_strerror": (C.c_char_p, [_int]),
    "mixdq_kernel_launches": (C.c_ulonglong, []),
    "mixdq_int8_tile_plan": (_int, [_i64, _i64, _i64, _int, C.POINTER(_int), C.POINTER(_int), C.POINTER(_int)]),
    "mixdq_int8_chan_tile": (_int, [_i64, _i64, _i64, _int, C.POINTER(_int), C.POINTER(_int)]),
    "mixdq_linear_fused_quant_tile": (_int, [_i64, _i64, _i64, _int]),
    "mixdq_int8_layer_plan": (_int, [_i64, _i64, _i64, _int, _int, C.POINTER(_int), C.POINTER(_int), C.POINTER(_int)]),
    "mixdq_packed_bytes": (_int, [_i64, _i64, _int, _int, C.POINTER(_sz)]),
    "mixdq_weight_minmax_params": (_int, [_vp, _i64, _i64, _int, _int, _vp, _vp, _vp]),
    "mixdq_pack_weights": (_int, [_vp, _i64, _i64, _int, _vp, _vp, _int, _vp, _vp]),
    "mixdq_unpack_weights": (_int, [_vp, _i64, _i64, _int, _int, _int, _vp, _vp]),
    "mixdq_act_absmax": (_int, [_vp, _i64, _i64, _i64, _int, _vp, _vp]),
    "mixdq_act_scale_from_absmax": (_int, [_vp, _vp, _vp]),
    "mixdq_act_scale": (_int, [_vp, _i64, _i64, _i64, _int, _vp, _vp]),
    "mixdq_act_asym_params": (_int, [_vp, _i64, _i64, _i64, _vp, _vp, _vp]),
    "mixdq_act_minmax": (_int, [_vp, _i64, _i64, _i64, _vp, _vp]),
    "mixdq_act_asym_params_from_minmax": (_int, [_vp, _vp, _vp, _vp]),
    "mixdq_weight_code_sums": (_int, [_vp, _i64, _i64, _int, _vp, _vp]),
    "mixdq_linear_a8_asym": (_int, [_vp, _i64, _i64, _i64, _vp, _i64, _int, _vp, _vp, _vp, _vp, _vp, _vp, _vp,
                                    _sz, _vp, _vp]),
    "mixdq_linear_a8_asym_acc_i32": (_int, [_vp, _i64, _i64, _i64, _vp, _i64, _int, _vp, _vp, _vp, _vp, _vp,
                                            _sz, _vp, _vp]),
    "mixdq_conv3x3_a8_asym": (_int, [_vp, _i64, _i64, _i64, _i64, _vp, _i64, _int, _int, _vp, _vp, _vp, _vp, _vp,
                                     _vp, _vp, _sz, _vp, _vp]),
    "mixdq_conv3x3_a8_asym_acc_i32": (_int, [_vp, _i64, _i64, _i64, _i64, _vp, _i64, _int, _int, _vp, _vp, _vp,
                                             _vp, _vp, _sz, _vp, _vp]),
    "mixdq_quantize_acts": (_int, [_vp, _i64, _i64, _i64, _vp, _vp, _vp]),
    "mixdq_linear_q8": (_int, [_vp, _i64, _i64, _vp, _i64, _int, _vp, _vp, _vp, _vp, _vp, _vp]),
    "mixdq_conv3x3_q8": (_int, [_vp, _i64, _i64, _i64, _i64, _vp, _i64, _int, _int, _vp, _vp, _vp, _vp, _vp, _vp]),
    "mixdq_linear_a8_fused_quant": (_int, [_vp, _i64, _i64, _i64, _vp, _i64, _int, _vp, _vp, _vp, _vp, _i64, _int, _vp, _vp]),
    "mixdq_selftest_abandoned_wait": (_int, [_vp, _i64, _i64, _vp, _i64, _int, _vp, _vp, _vp, _int, _vp, _vp]),
    "mixdq_selftest_abandoned_chan_wait": (_int, [_vp, _i64, _i64, _vp, _vp, _i64, _vp, _i64, _int, _vp, _vp, _int, _vp, _vp, _int, _vp, _vp]),
    "mixdq_linear_q8_acc_i32": (_int, [_vp, _i64, _i64, _vp, _i64, _int, _vp, _vp, _vp]),
    "mixdq_split_workspace_bytes": (_int, [_i64, _i64, _i64, _i64, _i64, C.POINTER(_sz)]),
    "mixdq_linear_a8_split": (_int, [_vp, _i64, _i64, _i64, _i64, _vp, _vp, _i64, _int, _vp, _vp, _vp, _vp, _vp, _vp,
                                     _sz, _vp, _vp]),
    "mixdq_linear_a8_split_acc_i32": (_int, [_vp, _i64, _i64, _i64, _i64, _vp, _vp, _i64, _int, _vp, _vp, _vp, _vp,
                                             _vp, _sz, _vp, _vp]),
    "mixdq_conv3x3_a8_split": (_int, [_vp, _i64, _i64, _i64, _i64, _i64, _vp, _vp, _i64, _int, _int, _vp, _vp, _vp,
                                      _vp, _vp, _vp, _sz, _vp, _vp]),
    "mixdq_conv3x3_a8_split_acc_i32": (_int, [_vp, _i64, _i64, _i64, _i64, _i64, _vp, _vp, _i64, _int, _int, _vp, _vp,
                                              _vp, _vp, _vp, _sz, _vp, _vp]),
    "mixdq_workspace_bytes": (_int, [_i64, _i64, _i64, _int, _int, C.POINTER(_sz)]),
    "mixdq_conv3x3_workspace_bytes": (_int, [_i64, _i64, _i64, _i64, _i64, _int, _int, _int, C.POINTER(_sz)]),
    "mixdq_linear": (_int, [_vp, _i64, _i64, _i64, _vp, _i64, _int, _vp, _vp, _int, _vp, _vp, _vp, _vp, _sz,
                            _vp, _vp]),
    "mixdq_linear_acc_i32": (_int, [_vp, _i64, _i64, _i64, _vp, _i64, _int, _vp, _vp, _vp, _sz, _vp, _vp]),
    "mixdq_conv3x3": (_int, [_vp, _i64, _i64, _i64, _i64, _vp, _i64, _int, _int, _vp, _vp, _int, _vp, _vp, _vp,
                             _vp, _sz, _vp, _vp]),
    "mixdq_conv3x3_acc_i32": (_int, [_vp, _i64, _i64, _i64, _i64, _vp, _i64, _int, _int, _vp, _vp, _vp, _sz,
                                     _vp, _vp]),
    "mixdq_conv1x1": (_int, [_vp, _i64, _i64, _i64, _i64, _vp, _i64, _int, _vp, _vp, _int, _vp, _vp, _vp, _vp,
                             _sz, _vp, _vp]),
    "mixdq_crossattn_kv": (_int, [_vp, _i64, _i64, _vp, _i64, _int, _vp, _vp, _vp, _vp, _vp, _sz, _vp, _vp]),
    "mixdq_crossattn_kv_acc_i32": (_int, [_vp, _i64, _i64, _vp, _i64, _int, _vp, _vp, _vp, _sz, _vp, _vp]),
    "mixdq_probe_mma_loop": (_int, [_int, _int, C.POINTER(C.c_double), _vp, _vp]),
    "mixdq_static_scratch_bytes": (_sz, []),
    "mixdq_linear_a8_static_scratch": (_int, [_vp, _i64, _i64, _i64, _vp, _i64, _int, _vp, _vp, _vp, _vp, _vp,
                                              _vp]),
}

EXPORTS = tuple(_SIGNATURES)

# Functions of the extension module, defined here at their first use.
NATIVE = (
    "weight_minmax_params", "pack_weights", "weight_code_sums", "act_absmax", "act_scale_from_absmax", "act_scale",
    "act_minmax", "act_asym_params", "linear", "linear_a8_asym", "quantize_acts", "linear_q8", "linear_a8_fused_quant",
    "linear_a8_static_scratch", "linear_a8_split", "crossattn_kv", "conv3x3", "conv3x3_a8_asym", "conv3x3_q8",
    "conv3x3_a8_split", "conv1x1",
)

_lib = None


class MixdqError(RuntimeError):
    pass


def lib():
    """Load the shared library (once).  Raises if it has not been built."""
    global _lib
    if _lib is None:
        if not os.path.exists(LIB_PATH):
            raise MixdqError(f"{LIB_PATH} is missing: build it with python -m paper_2405_17873_b200.build")
        L = C.CDLL(LIB_PATH)
        for name, (res, args) in _SIGNATURES.items():
            fn = getattr(L, name)
            fn.restype = res
            fn.argtypes = args
        _lib = L
    return _lib


def __getattr__(name: str):
    if name not in NATIVE:
        raise AttributeError(f"module {__name__!r} has no attribute {name!r}")
    lib()  # the extension links against it: the same copy serves both
    try:
        from . import _mixdq_native as native
    except ImportError as e:
        raise MixdqError(f"_mixdq_native is missing or does not load ({e}): build it with "
                         "python -m paper_2405_17873_b200.build") from e
    native._set_error_class(MixdqError)
    globals().update((n, getattr(native, n)) for n in NATIVE)
    return globals()[name]


def _chk(rc: int, what: str):
    if rc != 0:
        raise MixdqError(f"{what}: {lib().mixdq_strerror(rc).decode()} ({rc})")


def _ptr(t: Optional[torch.Tensor]):
    if t is None:
        return None
    assert t.is_cuda and t.is_contiguous(), "device-resident contiguous tensors only"
    return C.c_void_p(t.data_ptr())


def _stream():
    return C.c_void_p(torch.cuda.current_stream().cuda_stream)


def version() -> int:
    return lib().mixdq_version()


def kernel_launches() -> int:
    return int(lib().mixdq_kernel_launches())


def int8_tile_plan(M: int, N: int, k_blocks: int, w_bits: int, with_splits: bool = False):
    """(tile_rows, tile_cols[, reduction_splits]) of the int8 tensor-core GEMM for this shape on the current device."""
    r, c, sp = _int(0), _int(0), _int(0)
    _chk(lib().mixdq_int8_tile_plan(M, N, k_blocks, w_bits, C.byref(r), C.byref(c), C.byref(sp)), "mixdq_int8_tile_plan")
    return (r.value, c.value, sp.value) if with_splits else (r.value, c.value)


def int8_chan_tile(M: int, N: int, k_blocks: int, w_bits: int):
    """(channels, tokens) of the channel-major tile that runs this shape ahead of int8_tile_plan's, (0, 0) for none."""
    c, t = _int(0), _int(0)
    _chk(lib().mixdq_int8_chan_tile(M, N, k_blocks, w_bits, C.byref(c), C.byref(t)), "mixdq_int8_chan_tile")
    return c.value, t.value


def linear_fused_quant_tile(M: int, N: int, K: int, w_bits: int) -> int:
    """Tile width of the one-kernel (fused quantization) form for this linear layer, 0 when it runs as two kernels."""
    r = lib().mixdq_linear_fused_quant_tile(M, N, K, w_bits)
    if r < 0:
        _chk(r, "mixdq_linear_fused_quant_tile")
    return r


LAYER_KINDS = ("linear", "codes", "kv", "split")
LAYER_FORMS = ("single", "pair", "chan", "chan_many", "fused", "branches")


def int8_layer_plan(M: int, N: int, k_blocks: int, w_bits: int, kind: str = "linear"):
    """(form, tile_tokens, tile_channels, reduction_splits): the kernel that runs this int8 layer (mixdq_int8_layer_plan)."""
    t, c, sp = _int(0), _int(0), _int(0)
    form = lib().mixdq_int8_layer_plan(M, N, k_blocks, w_bits, LAYER_KINDS.index(kind), C.byref(t), C.byref(c), C.byref(sp))
    if form < 0:
        _chk(form, "mixdq_int8_layer_plan")
    return LAYER_FORMS[form], t.value, c.value, sp.value


def packed_bytes(N: int, K: int, bits: int, layout: int = LAYOUT_DEVICE) -> int:
    out = _sz(0)
    _chk(lib().mixdq_packed_bytes(N, K, bits, layout, C.byref(out)), "mixdq_packed_bytes")
    return out.value


def workspace_bytes(rows: int, N: int, K: int, w_bits: int, act_bits: int) -> int:
    out = _sz(0)
    _chk(lib().mixdq_workspace_bytes(rows, N, K, w_bits, act_bits, C.byref(out)), "mixdq_workspace_bytes")
    return out.value


def conv3x3_workspace_bytes(B: int, H: int, W: int, Cin: int, Cout: int, stride: int, w_bits: int,
                            act_bits: int) -> int:
    out = _sz(0)
    _chk(lib().mixdq_conv3x3_workspace_bytes(B, H, W, Cin, Cout, stride, w_bits, act_bits, C.byref(out)),
         "mixdq_conv3x3_workspace_bytes")
    return out.value


def new_workspace(nbytes: int, device="cuda") -> Optional[torch.Tensor]:
    """Zero-filled scratch buffer of the size mixdq_workspace_bytes reported."""
    if nbytes == 0:
        return None
    return torch.zeros(nbytes, dtype=torch.uint8, device=device)


def unpack_weights(packed: torch.Tensor, N: int, K: int, bits: int, is_signed: bool,
                   layout: int = LAYOUT_DEVICE) -> torch.Tensor:
    codes = torch.empty((N, K), dtype=torch.int16, device=packed.device)
    _chk(lib().mixdq_unpack_weights(_ptr(packed), N, K, bits, int(is_signed), layout, _ptr(codes), _stream()),
         "mixdq_unpack_weights")
    return codes


def _ws(workspace):
    return (_ptr(workspace), workspace.numel() if workspace is not None else 0)


def linear_acc_i32(X, packed_W, N: int, w_bits: int, act_scale, workspace=None, status=None):
    M, K = X.shape
    acc = torch.empty((M, N), dtype=torch.int32, device=X.device)
    wp, wb = _ws(workspace)
    _chk(lib().mixdq_linear_acc_i32(_ptr(X), M, K, X.stride(0), _ptr(packed_W), N, w_bits, _ptr(act_scale),
                                    _ptr(acc), wp, wb, _ptr(status), _stream()), "mixdq_linear_acc_i32")
    return acc


def linear_a8_asym_acc_i32(X, packed_W, N: int, w_bits: int, w_code_sums, act_scale, act_zero, workspace=None,
                           status=None):
    M, K = X.shape
    acc = torch.empty((M, N), dtype=torch.int32, device=X.device)
    wp, wb = _ws(workspace)
    _chk(lib().mixdq_linear_a8_asym_acc_i32(_ptr(X), M, K, X.stride(0), _ptr(packed_W), N, w_bits,
                                            _ptr(w_code_sums), _ptr(act_scale), _ptr(act_zero), _ptr(acc), wp,
                                            wb, _ptr(status), _stream()), "mixdq_linear_a8_asym_acc_i32")
    return acc


def _out_hw(H, W, stride):
    return (H - 1) // stride + 1, (W - 1) // stride + 1


def conv3x3_a8_asym_acc_i32(X, packed_W, Cout: int, w_bits: int, w_code_sums, act_scale, act_zero,
                            stride: int = 1, workspace=None, status=None):
    B, H, W, Cin = X.shape
    Ho, Wo = _out_hw(H, W, stride)
    acc = torch.empty((B, Ho, Wo, Cout), dtype=torch.int32, device=X.device)
    wp, wb = _ws(workspace)
    _chk(lib().mixdq_conv3x3_a8_asym_acc_i32(_ptr(X), B, H, W, Cin, _ptr(packed_W), Cout, stride, w_bits,
                                             _ptr(w_code_sums), _ptr(act_scale), _ptr(act_zero), _ptr(acc), wp,
                                             wb, _ptr(status), _stream()), "mixdq_conv3x3_a8_asym_acc_i32")
    return acc


def selftest_abandoned_wait(Xq, packed_W, N: int, w_bits: int, w_scale, act_scale, drop_k_block: int, status):
    """mixdq_linear_q8 with one weight tile never requested: *status becomes MIXDQ_ERR_TIMEOUT (-6)."""
    M, K = Xq.shape
    Y = torch.empty((M, N), dtype=torch.float16, device=Xq.device)
    _chk(lib().mixdq_selftest_abandoned_wait(_ptr(Xq), M, K, _ptr(packed_W), N, w_bits, _ptr(w_scale), _ptr(act_scale),
                                             _ptr(Y), drop_k_block, _ptr(status), _stream()),
         "mixdq_selftest_abandoned_wait")
    return Y


def selftest_abandoned_chan_wait(X, packed_W, N: int, w_bits: int, w_scale, w_zero, act_bits: int, act_scale, drop_k_block: int,
                                 status, X_hi=None, packed_W_hi=None):
    """The same on the channel-major kernel that runs the layer (act_bits 8: X int8 codes, X_hi a second branch's; 16: X fp16)."""
    M, K = X.shape
    K_hi = 0 if X_hi is None else X_hi.shape[1]
    Y = torch.empty((M, N), dtype=torch.float16, device=X.device)
    _chk(lib().mixdq_selftest_abandoned_chan_wait(_ptr(X), M, K, _ptr(packed_W), _ptr(X_hi), K_hi, _ptr(packed_W_hi), N, w_bits,
                                                  _ptr(w_scale), _ptr(w_zero), act_bits, _ptr(act_scale), _ptr(Y), drop_k_block,
                                                  _ptr(status), _stream()), "mixdq_selftest_abandoned_chan_wait")
    return Y


def linear_q8_acc_i32(Xq, packed_W, N: int, w_bits: int, status=None):
    M, K = Xq.shape
    acc = torch.empty((M, N), dtype=torch.int32, device=Xq.device)
    _chk(lib().mixdq_linear_q8_acc_i32(_ptr(Xq), M, K, _ptr(packed_W), N, w_bits, _ptr(acc), _ptr(status),
                                       _stream()), "mixdq_linear_q8_acc_i32")
    return acc


def split_workspace_bytes(in_rows: int, row_len: int, split_at: int, out_rows: int, N: int) -> int:
    out = _sz(0)
    _chk(lib().mixdq_split_workspace_bytes(in_rows, row_len, split_at, out_rows, N, C.byref(out)),
         "mixdq_split_workspace_bytes")
    return out.value


def linear_a8_split_acc_i32(X, split_at: int, packed_W_lo, packed_W_hi, N: int, w_bits: int, act_scale_lo,
                            act_scale_hi, workspace=None, status=None):
    M, K = X.shape
    lo = torch.empty((M, N), dtype=torch.int32, device=X.device)
    hi = torch.empty((M, N), dtype=torch.int32, device=X.device)
    wp, wb = _ws(workspace)
    _chk(lib().mixdq_linear_a8_split_acc_i32(_ptr(X), M, K, X.stride(0), split_at, _ptr(packed_W_lo),
                                             _ptr(packed_W_hi), N, w_bits, _ptr(act_scale_lo), _ptr(act_scale_hi),
                                             _ptr(lo), _ptr(hi), wp, wb, _ptr(status), _stream()),
         "mixdq_linear_a8_split_acc_i32")
    return lo, hi


def conv3x3_a8_split_acc_i32(X, split_at: int, packed_W_lo, packed_W_hi, Cout: int, w_bits: int, act_scale_lo,
                             act_scale_hi, stride: int = 1, workspace=None, status=None):
    B, H, W, Cin = X.shape
    Ho, Wo = _out_hw(H, W, stride)
    lo = torch.empty((B, Ho, Wo, Cout), dtype=torch.int32, device=X.device)
    hi = torch.empty((B, Ho, Wo, Cout), dtype=torch.int32, device=X.device)
    wp, wb = _ws(workspace)
    _chk(lib().mixdq_conv3x3_a8_split_acc_i32(_ptr(X), B, H, W, Cin, split_at, _ptr(packed_W_lo),
                                              _ptr(packed_W_hi), Cout, stride, w_bits, _ptr(act_scale_lo),
                                              _ptr(act_scale_hi), _ptr(lo), _ptr(hi), wp, wb, _ptr(status),
                                              _stream()), "mixdq_conv3x3_a8_split_acc_i32")
    return lo, hi


def conv3x3_acc_i32(X, packed_W, Cout: int, w_bits: int, act_scale, stride: int = 1, workspace=None,
                    status=None):
    B, H, W, Cin = X.shape
    Ho, Wo = _out_hw(H, W, stride)
    acc = torch.empty((B, Ho, Wo, Cout), dtype=torch.int32, device=X.device)
    wp, wb = _ws(workspace)
    _chk(lib().mixdq_conv3x3_acc_i32(_ptr(X), B, H, W, Cin, _ptr(packed_W), Cout, stride, w_bits,
                                     _ptr(act_scale), _ptr(acc), wp, wb, _ptr(status), _stream()),
         "mixdq_conv3x3_acc_i32")
    return acc


def crossattn_kv_acc_i32(text_emb, packed_W, N: int, w_bits: int, act_scale, workspace=None, status=None):
    B, T, Kt = text_emb.shape
    assert T == TOKENS_PER_PROMPT
    acc = torch.empty((B, T - 1, N), dtype=torch.int32, device=text_emb.device)
    wp, wb = _ws(workspace)
    _chk(lib().mixdq_crossattn_kv_acc_i32(_ptr(text_emb), B, Kt, _ptr(packed_W), N, w_bits, _ptr(act_scale),
                                          _ptr(acc), wp, wb, _ptr(status), _stream()),
         "mixdq_crossattn_kv_acc_i32")
    return acc


def static_scratch_bytes() -> int:
    return lib().mixdq_static_scratch_bytes()


def probe_mma_loop(kind: int, batches: int, repeats: int = 3) -> float:
    """Tensor-core MMA-loop peak in TOP/s (kind 1: int8, kind 0: fp16), best of ``repeats``."""
    ops = C.c_double(0.0)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    best = 0.0
    for _ in range(repeats + 1):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        _chk(lib().mixdq_probe_mma_loop(kind, batches, C.byref(ops), _ptr(status), _stream()), "mixdq_probe_mma_loop")
        b.record()
        torch.cuda.synchronize()
        if int(status.item()) != 0:
            raise MixdqError("mixdq_probe_mma_loop: device-side wait timed out")
        best = max(best, ops.value / (a.elapsed_time(b) * 1e-3) / 1e12)
    return best
