"""The queries that say which kernel runs an int8 layer name the one that the layer calls launch, over sizes of every form (on
the recording runtime, recorded.py: nothing runs on a GPU)."""
import ctypes as C
import random

import pytest

import test_gpu_forms as forms
from paper_2405_17873_b200 import mixdq
from recorded import BUFFER, Recorded

BYTES = C.c_size_t(1 << 40)
KERNELS = {"chan_gemm_kernel": "chan", "chan_many_kernel": "chan_many", "pair_gemm_kernel": "pair", "fq_gemm_kernel": "fused",
           "tma_gemm_": "single"}


@pytest.fixture(scope="module")
def lib(recorded_library):
    return Recorded(recorded_library)


def _sizes(rng, n):
    """Layers spread over the logarithm of their sizes, half of them with short reductions on many rows."""
    log = lambda lo, hi, step: max(step, round(lo * (hi / lo) ** rng.random() / step) * step)
    for i in range(n):
        short = i % 2
        yield log(1024 if short else 1, 16384, 1), log(16, 1024 if short else 10240, 4), log(16, 640 if short else 20000, 16)


@pytest.mark.parametrize("bits", [4, 8])
@pytest.mark.parametrize("kind", mixdq.LAYER_KINDS)
def test_plan_names_the_kernel_that_is_launched(lib, kind, bits):
    rng, seen = random.Random(bits), set()
    t, c, sp = C.c_int(), C.c_int(), C.c_int()
    for M, N, K in _sizes(rng, 600):
        so, at = lib.so, max(16, K // 32 * 16)
        if kind == "split" and at >= K:
            continue
        if kind == "kv":
            M = -(-M // 76) * 76
        kb = -(-K // 128) if kind != "split" else -(-at // 128) + -(-(K - at) // 128)
        form = so.mixdq_int8_layer_plan(M, N, kb, bits, mixdq.LAYER_KINDS.index(kind), C.byref(t), C.byref(c), C.byref(sp))
        if kind == "linear":
            rc = so.mixdq_linear(BUFFER, M, K, K, BUFFER, N, bits, BUFFER, None, 8, BUFFER, None, BUFFER, BUFFER, BYTES, None, None)
            fused = so.mixdq_linear_fused_quant_tile(M, N, K, bits)
            assert fused == (c.value if mixdq.LAYER_FORMS[form] == "fused" else 0)
        elif kind == "codes":
            rc = so.mixdq_linear_q8(BUFFER, M, K, BUFFER, N, bits, BUFFER, BUFFER, None, BUFFER, None, None)
        elif kind == "kv":
            rc = so.mixdq_crossattn_kv(BUFFER, M // 76, K, BUFFER, N, bits, BUFFER, BUFFER, BUFFER, BUFFER, BUFFER, BYTES, None, None)
        else:
            rc = so.mixdq_linear_a8_split(BUFFER, M, K, K, at, BUFFER, BUFFER, N, bits, BUFFER, BUFFER, BUFFER, None, BUFFER, BUFFER,
                                          BYTES, None, None)
        assert rc == 0
        gemms = [form_ for name, _ in lib.launches() for part, form_ in KERNELS.items() if part in name]
        got = "branches" if kind == "split" and len(gemms) == 2 else gemms[0]
        assert mixdq.LAYER_FORMS[form] == got, (M, N, K, bits)
        seen.add(got)
    assert {"linear": {"chan", "pair", "fused", "single"}, "codes": {"chan", "pair", "single"}, "kv": {"chan", "single"},
            "split": {"chan", "pair", "branches"}}[kind] <= seen, seen
    assert ("chan_many" in seen) == (bits == 4 and kind in ("linear", "codes"))


def test_argument_errors(lib):
    t, c, sp = (C.byref(C.c_int()) for _ in range(3))
    plan = lib.so.mixdq_int8_layer_plan
    assert plan(64, 64, 1, 8, 0, t, c, sp) >= 0
    assert plan(0, 64, 1, 8, 0, t, c, sp) == -1 and plan(64, 64, 1, 8, 4, t, c, sp) == -1 and plan(64, 64, 1, 8, 0, None, c, sp) == -1
    assert plan(64, 64, 1, 3, 0, t, c, sp) == -2


def _launches(lib, kernel, case, call):
    assert call(lib.so) == 0
    names = [name for name, _ in lib.launches()]
    assert kernel in names[-1], (case, names)


def test_cases_of_the_rare_kernels_launch_them(lib):
    """(of test_gpu_forms.py)"""
    ws = lambda use: (BUFFER, BYTES) if use else (None, C.c_size_t(0))
    for bits, sym, M, K, N, use, kernel in forms.LINEAR_A16:
        _launches(lib, kernel, (bits, M, K, N), lambda so: so.mixdq_linear(
            BUFFER, M, K, -(-K // 8) * 8, BUFFER, N, bits, BUFFER, None if sym else BUFFER, 16, None, BUFFER, BUFFER, *ws(use), None, None))
    for bits, (B, H, W, Cin, Cout, stride), use, kernel in forms.CONV_A16:
        _launches(lib, kernel, (bits, B, H, W, Cin, Cout, stride), lambda so: so.mixdq_conv3x3(
            BUFFER, B, H, W, Cin, BUFFER, Cout, stride, bits, BUFFER, BUFFER, 16, None, BUFFER, BUFFER, *ws(use), None, None))
    for bits, M, N, K, kernel in forms.LINEAR_Q8:
        _launches(lib, kernel, (bits, M, N, K), lambda so: so.mixdq_linear_q8(
            BUFFER, M, K, BUFFER, N, bits, BUFFER, BUFFER, None, BUFFER, None, None))
    for bits, M, lo, hi, N, kernel in forms.SPLIT_A8:
        _launches(lib, kernel, (bits, M, lo, hi, N), lambda so: so.mixdq_linear_a8_split(
            BUFFER, M, lo + hi, lo + hi, lo, BUFFER, BUFFER, N, bits, BUFFER, BUFFER, BUFFER, None, BUFFER, BUFFER, BYTES, None, None))
