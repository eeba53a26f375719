"""The channel-major weight-only kernel: one pair of k-blocks to more than its rings hold, odd and even numbers of them, ragged
channels, tokens and reduction tails, odd widths, one- and two-CTA tiles, several waves of small layers, convolutions."""
import numpy as np
import pytest
import torch

from oracle import mixdq_oracle as orc
from paper_2405_17873_b200 import mixdq, synth
from helpers import assert_close, dev, device_weights, host, oracle_weights, status_word

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [2, 3, 4, 8])
@pytest.mark.parametrize("M,N,K", [(17, 16, 64), (20, 129, 136), (33, 320, 328), (100, 1283, 1296), (255, 10240, 320), (16, 5120, 640),
                                   (600, 1280, 2064), (1000, 1284, 648), (4090, 636, 640), (64, 640, 5136)])
def test_linear(bits, M, N, K):
    X = synth.normal_f16((M, K), 1.0, seed=M + K)
    W = synth.normal_f16((N, K), 0.02, seed=N + K + 1)
    b = synth.normal_f16((N,), 0.01, seed=N)
    for symmetric in ([False, True] if bits >= 4 else [False]):
        s_ref, z_ref, codes = oracle_weights(W, bits, symmetric)
        y_ref = orc.linear_a16(X, codes, s_ref, None if symmetric else z_ref, b)
        s, z, packed = device_weights(W, bits, symmetric)
        st = status_word()
        y = [mixdq.linear(dev(X), packed, N, bits, s, None if symmetric else z, 16, None, dev(b), None, st) for _ in range(2)]
        torch.cuda.synchronize()
        assert int(host(st)[0]) == 0
        assert torch.equal(y[0], y[1])  # the order of the sums is fixed
        assert_close(host(y[0]), y_ref)


@pytest.mark.parametrize("bits", [2, 3, 4, 8])
@pytest.mark.parametrize("B,H,W,Cin,Cout,stride", [(1, 4, 5, 64, 16, 1), (2, 17, 13, 192, 137, 2), (1, 24, 24, 128, 320, 1),
                                                   (2, 32, 30, 320, 328, 1)])
def test_conv3x3(bits, B, H, W, Cin, Cout, stride):
    X = synth.normal_f16((B, H, W, Cin), 1.0, seed=H * W + Cin)
    Wt = synth.normal_f16((Cout, 3, 3, Cin), 0.02, seed=Cout + Cin)
    s_ref, z_ref, codes = oracle_weights(Wt.reshape(Cout, -1), bits, False)
    y_ref = orc.conv3x3_a16(X, codes.reshape(Cout, 3, 3, Cin), s_ref, z_ref, None, stride)
    s, z, packed = device_weights(Wt.reshape(Cout, -1), bits, False)
    st = status_word()
    y = mixdq.conv3x3(dev(X), packed, Cout, bits, s, z, 16, None, None, stride, None, st)
    torch.cuda.synchronize()
    assert int(host(st)[0]) == 0
    assert_close(host(y), y_ref)
