"""GPU parity of the kernels that the dispatch takes for few sizes only, on sizes that take them.  test_dispatch.py checks,
without a GPU, that every case here launches the kernel it names."""
import numpy as np
import pytest
import torch

from oracle import mixdq_oracle as orc
from paper_2405_17873_b200 import mixdq, synth
import test_gpu_int8_split as split
import test_gpu_weight_only as weight_only
from helpers import assert_close, dev, device_weights, host, oracle_weights, status_word

pytestmark = pytest.mark.gpu

PAIR_CODES, PAIR_PACKED = "pair_gemm_kernelILi2E", "pair_gemm_kernelILi3E"
# weight-only linear layers: bits, symmetric, M, K, N, workspace, kernel
WIDTHS = [(2, False), (3, False), (4, False), (4, True), (8, False), (8, True)]
LINEAR_A16 = [(bits, sym, *case) for bits, sym in WIDTHS for case in
              [(600, 136, 10000, False, "wo_tc_kernel"), (4097, 72, 1300, False, "wo_tc_kernel"),
               (600, 136, 10000, True, PAIR_CODES if bits == 8 else PAIR_PACKED), (4097, 328, 1290, True, PAIR_CODES),
               (5, 100, 40, False, f"wo_kernelILi{bits}ELb{int(sym)}ELi1E"), (13, 100, 41, False, f"wo_kernelILi{bits}ELb{int(sym)}ELi2E"),
               (30, 100, 41, False, f"wo_kernelILi{bits}ELb{int(sym)}ELi4E"),
               (7, 864, 96, False, f"wo_small_kernelILi{bits}ELb{int(sym)}ELi1ELi1E"),
               (14, 2056, 130, False, f"wo_small_kernelILi{bits}ELb{int(sym)}ELi2ELi1E"),
               (5, 864, 6720, False, f"wo_small_kernelILi{bits}ELb{int(sym)}ELi1ELi2E"),
               (12, 3288, 4738, False, f"wo_small_kernelILi{bits}ELb{int(sym)}ELi2ELi2E")]]
# weight-only 3x3 convolutions: bits, (B, H, W, Cin, Cout, stride), workspace, kernel
CONV_A16 = [(bits, *case) for bits in (2, 3, 4, 8) for case in
            [((6, 32, 32, 64, 650, 1), False, "wo_tc_kernel"), ((5, 32, 32, 64, 2600, 2), True, PAIR_CODES if bits == 8 else PAIR_PACKED),
             ((5, 33, 35, 64, 650, 1), True, PAIR_CODES)]]
# int8 layers on stored codes: bits, M, N, K, kernel
LINEAR_Q8 = [(8, *case, "tma_gemm_kernelILi256E") for case in [(868, 4007, 96), (831, 4776, 160), (514, 7030, 912)]]
# shortcut-split linear layers that run a GEMM for each branch; the second takes the first's int32 sums, on one tile, with its
# reduction split over a cluster, or persistent: bits, M, lo, hi, N, kernel
SPLIT_A8 = [(bits, *case, f"{kernel}ILi128ELi6ELb{int(bits == 4)}ELb1E") for bits in (4, 8) for *case, kernel in
            [(6023, 64, 48, 317, "tma_gemm_kernel"), (2070, 176, 32, 930, "tma_gemm_kernel"),
             (6194, 80, 320, 1252, "tma_gemm_persistent_kernel")]] + \
           [(8, 58, 18032, 1968, 21, "tma_gemm_kernelILi128ELi6ELb0ELb1E"), (8, 568, 8224, 1216, 141, "tma_gemm_kernelILi128ELi6ELb0ELb1E"),
            (4, 397, 5008, 6912, 162, "tma_gemm_kernelILi128ELi6ELb1ELb1E"), (4, 948, 9312, 3344, 151, "tma_gemm_kernelILi128ELi6ELb1ELb1E")]


@pytest.mark.parametrize("bits,symmetric,M,K,N,use_ws,kernel", LINEAR_A16)
def test_weight_only_linear(bits, symmetric, M, K, N, use_ws, kernel):
    X = synth.normal_f16((M, K), 1.0, seed=M * 7 + K)
    W = synth.normal_f16((N, K), 0.02, seed=N * 11 + K)
    b = synth.normal_f16((N,), 0.01, seed=N + 2)
    if K % 8 == 0:
        weight_only._run(X, W, b, bits, symmetric, use_ws)
        return
    # rows whose length is no multiple of eight: the C call alone takes a row stride
    s_ref, z_ref, codes = oracle_weights(W, bits, symmetric)
    y_ref = orc.linear_a16(X, codes, s_ref, z_ref, b)
    s, z, packed = device_weights(W, bits, symmetric)
    Xd, bd, y, st = dev(np.pad(X, ((0, 0), (0, -K % 8)))), dev(b), torch.empty((M, N), dtype=torch.float16, device="cuda"), status_word()
    p = lambda t: None if t is None else t.data_ptr()
    assert mixdq.lib().mixdq_linear(p(Xd), M, K, Xd.shape[1], p(packed), N, bits, p(s), p(z), 16, None, p(bd), p(y), None, 0, p(st),
                                    torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    assert int(host(st)[0]) == 0
    assert_close(host(y), y_ref)


@pytest.mark.parametrize("bits,geom,use_ws,kernel", CONV_A16)
def test_weight_only_conv3x3(bits, geom, use_ws, kernel):
    (weight_only.test_weight_only_conv3x3_with_workspace if use_ws else weight_only.test_weight_only_conv3x3)(bits, geom)


@pytest.mark.parametrize("bits,M,N,K,kernel", LINEAR_Q8)
def test_int8_linear(bits, M, N, K, kernel):
    X, W, b = synth.normal_f16((M, K), 1.0, seed=M), synth.normal_f16((N, K), 0.02, seed=N), synth.normal_f16((N,), 0.01, seed=K)
    s_ref, _, codes = oracle_weights(W, bits, True)
    acc_ref, y_ref = orc.linear_a8(X, codes, s_ref, orc.act_scale(orc.act_absmax(X), 8), b)
    Xd = dev(X)
    s, _, packed = device_weights(W, bits, True)
    sx, st = mixdq.act_scale(Xd), status_word()
    xq = mixdq.quantize_acts(Xd, sx)
    acc = mixdq.linear_q8_acc_i32(xq, packed, N, bits, st)
    y = mixdq.linear_q8(xq, packed, N, bits, s, sx, dev(b), st)
    torch.cuda.synchronize()
    assert int(host(st)[0]) == 0
    assert np.array_equal(host(acc), acc_ref)
    assert_close(host(y), y_ref)


@pytest.mark.parametrize("bits,M,C_lo,C_hi,N,kernel", SPLIT_A8)
def test_split_linear_as_two_gemms(bits, M, C_lo, C_hi, N, kernel):
    split._run_linear(M, C_lo, C_hi, N, bits, seed=M + C_lo + N + 9)
