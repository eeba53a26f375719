"""The channel-major int8 kernel (weights on the rows of the tensor-core tile) on one- and two-CTA tiles: odd and even
numbers of k-blocks from one to more than every ring holds, ragged channels, tokens and reduction tails, odd widths,
every source of activations (rows, skipped first tokens, im2col, asymmetric codes), both branches of shortcut-split
layers."""
import numpy as np
import pytest
import torch

from oracle import mixdq_oracle as orc
from paper_2405_17873_b200 import mixdq, synth
import test_gpu_int8_split as split
from helpers import assert_close, dev, device_weights, host, oracle_weights, status_word

pytestmark = pytest.mark.gpu


def _layer(M, N, K):
    return (synth.normal_f16((M, K), 1.0, seed=M + K), synth.normal_f16((N, K), 0.02, seed=N + K + 1),
            synth.normal_f16((N,), 0.01, seed=N))


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("M,N,K", [(1, 16, 16), (5, 129, 144), (16, 128, 128), (17, 320, 272), (100, 127, 640), (250, 1283, 1296),
                                   (256, 320, 320), (1000, 1280, 1552), (1023, 1288, 2576), (600, 1280, 2064), (4090, 636, 640),
                                   (2050, 640, 2576), (33, 1280, 5136)])
def test_linear(bits, M, N, K):
    channels, tokens = mixdq.int8_chan_tile(M, N, -(-K // 128), bits)
    assert channels in (128, 256) and tokens % 16 == 0 and tokens > 0
    X, W, b = _layer(M, N, K)
    s_ref, _, codes = oracle_weights(W, bits, True)
    sx_ref = orc.act_scale(orc.act_absmax(X), 8)
    acc_ref, y_ref = orc.linear_a8(X, codes, s_ref, sx_ref, b)
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


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("M,N,K", [(77, 136, 272), (1024, 640, 1280), (2048, 1280, 656)])
def test_asymmetric(bits, M, N, K):
    assert mixdq.int8_chan_tile(M, N, -(-K // 128), bits)[1] > 0
    _, W, b = _layer(M, N, K)
    X = synth.one_sided_f16((M, K), seed=5, shift=0.3)
    s_ref, _, codes = oracle_weights(W, bits, True)
    sa_ref, z_ref = orc.act_minmax_params(X)
    acc_ref, y_ref = orc.linear_a8_asym(X, codes, s_ref, sa_ref, z_ref, b)
    Xd = dev(X)
    s, _, packed = device_weights(W, bits, True)
    sums = mixdq.weight_code_sums(packed, N, K, bits)
    sa, z = mixdq.act_asym_params(Xd)
    ws, st = mixdq.new_workspace(mixdq.workspace_bytes(M, N, K, bits, 8)), status_word()
    acc = mixdq.linear_a8_asym_acc_i32(Xd, packed, N, bits, sums, sa, z, workspace=ws, status=st)
    y = mixdq.linear_a8_asym(Xd, packed, N, bits, s, sums, sa, z, dev(b), ws, st)
    torch.cuda.synchronize()
    assert int(host(st)[0]) == 0
    assert np.array_equal(host(acc), acc_ref)
    assert_close(host(y), y_ref)


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("B,H,W,Cin,Cout,stride", [(1, 4, 5, 32, 16, 1), (2, 17, 13, 160, 136, 2), (4, 16, 16, 640, 1280, 1),
                                                   (2, 32, 30, 320, 640, 1), (1, 24, 24, 224, 321, 1)])
def test_conv3x3(bits, B, H, W, Cin, Cout, stride):
    Ho, Wo = (H - 1) // stride + 1, (W - 1) // stride + 1
    assert mixdq.int8_chan_tile(B * Ho * Wo, Cout, 9 * -(-Cin // 128), bits)[1] > 0
    X = synth.normal_f16((B, H, W, Cin), 1.0, seed=H * W + Cin)
    Wt = synth.normal_f16((Cout, 3, 3, Cin), 0.02, seed=Cout + Cin)
    s_ref, _, codes = oracle_weights(Wt.reshape(Cout, -1), bits, True)
    sx_ref = orc.act_scale(orc.act_absmax(X), 8)
    acc_ref, y_ref = orc.conv3x3_a8(X, codes.reshape(Cout, 3, 3, Cin), s_ref, sx_ref, None, stride)
    Xd = dev(X)
    s, _, packed = device_weights(Wt.reshape(Cout, -1), bits, True)
    sx, st = mixdq.act_scale(Xd), status_word()
    ws = mixdq.new_workspace(mixdq.conv3x3_workspace_bytes(B, H, W, Cin, Cout, stride, bits, 8))
    acc = mixdq.conv3x3_acc_i32(Xd, packed, Cout, bits, sx, stride, workspace=ws, status=st)
    y = mixdq.conv3x3(Xd, packed, Cout, bits, s, None, 8, sx, None, stride, ws, st)
    torch.cuda.synchronize()
    assert int(host(st)[0]) == 0
    assert np.array_equal(host(acc), acc_ref)
    assert_close(host(y), y_ref)


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("batch,N,K", [(1, 40, 64), (8, 1280, 2048), (3, 321, 400)])
def test_bos(bits, batch, N, K):
    assert mixdq.int8_chan_tile(76 * batch, N, -(-K // 128), bits)[1] > 0
    E = synth.normal_f16((batch, 77, K), 1.0, seed=batch + K)
    E[:, 0] = synth.normal_f16((K,), 40.0, seed=2)
    W = synth.normal_f16((N, K), 0.02, seed=N + K)
    s_ref, _, codes = oracle_weights(W, bits, True)
    sx_ref = orc.act_scale(orc.act_absmax(np.ascontiguousarray(E[:, 1:])), 8)
    bos_ref = orc.bos_row(E[0, 0], W)
    acc_ref, y_ref = orc.crossattn_kv(E, codes, s_ref, sx_ref, bos_ref)
    s, _, packed = device_weights(W, bits, True)
    ws, st = mixdq.new_workspace(mixdq.workspace_bytes(76 * batch, N, K, bits, 8)), status_word()
    sx = dev(np.array([sx_ref], np.float32))
    acc = mixdq.crossattn_kv_acc_i32(dev(E), packed, N, bits, sx, workspace=ws, status=st)
    y = mixdq.crossattn_kv(dev(E), packed, N, bits, s, sx, dev(bos_ref), workspace=ws, status=st)
    torch.cuda.synchronize()
    assert int(host(st)[0]) == 0
    assert np.array_equal(host(acc), acc_ref)
    assert_close(host(y), y_ref)


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("M,C_lo,C_hi,N", [(1, 16, 16, 16), (100, 144, 272, 129), (1024, 1280, 1280, 1280), (250, 2064, 128, 648)])
def test_two_branches_linear(bits, M, C_lo, C_hi, N):
    split._run_linear(M, C_lo, C_hi, N, bits, seed=M + C_lo)


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("B,H,W,C_lo,C_hi,N,stride", [(2, 16, 16, 160, 96, 136, 1), (1, 8, 16, 32, 32, 16, 1), (4, 16, 16, 384, 256, 1280, 1),
                                                      (2, 32, 32, 128, 640, 328, 2)])
def test_two_branches_conv3x3(bits, B, H, W, C_lo, C_hi, N, stride):
    split._run_conv(B, H, W, C_lo, C_hi, N, bits, stride, seed=H + C_lo + N)


# int4 layers of several waves: a CTA pair's tiles follow each other through the rings, on one accumulator and on two
@pytest.mark.parametrize("M,N,K", [(3000, 5124, 272), (2050, 5121, 656), (4500, 2564, 1296), (1024, 10240, 1280), (4100, 1800, 5136)])
def test_linear_of_several_waves(M, N, K):
    channels, tokens = mixdq.int8_chan_tile(M, N, -(-K // 128), 4)
    assert channels == 256 and -(-M // tokens) * -(-N // 256) > 74
    X, W, b = _layer(M, N, K)
    X = synth.one_sided_f16((M, K), seed=5, shift=0.3)
    s_ref, _, codes = oracle_weights(W, 4, True)
    sa_ref, z_ref = orc.act_minmax_params(X)
    acc_ref, y_ref = orc.linear_a8_asym(X, codes, s_ref, sa_ref, z_ref, b)
    Xd = dev(X)
    s, _, packed = device_weights(W, 4, True)
    sums = mixdq.weight_code_sums(packed, N, K, 4)
    sa, z = mixdq.act_asym_params(Xd)
    ws, st = mixdq.new_workspace(mixdq.workspace_bytes(M, N, K, 4, 8)), status_word()
    acc = mixdq.linear_a8_asym_acc_i32(Xd, packed, N, 4, sums, sa, z, workspace=ws, status=st)
    y = mixdq.linear_a8_asym(Xd, packed, N, 4, s, sums, sa, z, dev(b), ws, st)
    torch.cuda.synchronize()
    assert int(host(st)[0]) == 0
    assert np.array_equal(host(acc), acc_ref)
    assert_close(host(y), y_ref)


@pytest.mark.parametrize("B,H,W,Cin,Cout,stride", [(4, 64, 64, 320, 320, 1), (3, 65, 63, 96, 648, 1), (2, 96, 97, 128, 1284, 2)])
def test_conv3x3_of_several_waves(B, H, W, Cin, Cout, stride):
    test_conv3x3(4, B, H, W, Cin, Cout, stride)
