"""3x3 convolutions on images that do not tile into 128-pixel boxes: the im2col loads of the TMA-fed kernels, on
one-tile, cluster-split, persistent and two-CTA shapes, int8 and weight-only, with ragged last tiles, tiles that span
images, channel tails and stride 2 on odd sides."""
import numpy as np
import pytest
import torch

from oracle import mixdq_oracle as orc
from paper_2405_17873_b200 import mixdq, synth
from helpers import assert_close, dev, device_weights, host, oracle_weights, status_word

pytestmark = pytest.mark.gpu


def _inputs(B, H, W, Cin, Cout):
    return (synth.normal_f16((B, H, W, Cin), 1.0, seed=H * W + Cin), synth.normal_f16((Cout, 3, 3, Cin), 0.02, seed=Cout + Cin),
            synth.normal_f16((Cout,), 0.01, seed=Cout))


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("B,H,W,Cin,Cout,stride", [(1, 8, 9, 32, 16, 1), (5, 3, 5, 96, 40, 1), (2, 17, 13, 160, 136, 2),
                                                   (1, 24, 24, 640, 136, 1), (3, 48, 48, 64, 320, 1), (1, 48, 48, 256, 320, 1),
                                                   (2, 26, 38, 320, 648, 1), (2, 97, 61, 32, 200, 2), (1, 12, 20, 1280, 320, 1)])
def test_int8(bits, B, H, W, Cin, Cout, stride):
    X, Wt, b = _inputs(B, H, W, Cin, Cout)
    s_ref, _, codes = oracle_weights(Wt.reshape(Cout, -1), bits, True)
    sx_ref = orc.act_scale(orc.act_absmax(X), 8)
    acc_ref, y_ref = orc.conv3x3_a8(X, codes.reshape(Cout, 3, 3, Cin), s_ref, sx_ref, b, stride)
    Xd = dev(X)
    s, _, packed = device_weights(Wt.reshape(Cout, -1), bits, True)
    sx, st = mixdq.act_scale(Xd), status_word()
    ws = mixdq.new_workspace(mixdq.conv3x3_workspace_bytes(B, H, W, Cin, Cout, stride, bits, 8))
    acc = mixdq.conv3x3_acc_i32(Xd, packed, Cout, bits, sx, stride, workspace=ws, status=st)
    y = mixdq.conv3x3(Xd, packed, Cout, bits, s, None, 8, sx, dev(b), stride, workspace=ws, status=st)
    torch.cuda.synchronize()
    assert int(host(st)[0]) == 0
    assert np.array_equal(host(acc), acc_ref)
    assert_close(host(y), y_ref)


@pytest.mark.parametrize("use_ws", [True, False])
@pytest.mark.parametrize("bits", [2, 3, 4, 8])
@pytest.mark.parametrize("B,H,W,Cin,Cout,stride", [(1, 8, 9, 64, 40, 1), (2, 17, 13, 128, 136, 2), (1, 24, 24, 200, 136, 1),
                                                   (3, 48, 48, 64, 320, 1), (1, 12, 22, 640, 320, 1)])
def test_weight_only(bits, B, H, W, Cin, Cout, stride, use_ws):
    X, Wt, b = _inputs(B, H, W, Cin, Cout)
    s_ref, z_ref, codes = oracle_weights(Wt.reshape(Cout, -1), bits, False)
    y_ref = orc.conv3x3_a16(X, codes.reshape(Cout, 3, 3, Cin), s_ref, z_ref, b, stride)
    s, z, packed = device_weights(Wt.reshape(Cout, -1), bits, False)
    st = status_word()
    ws = mixdq.new_workspace(mixdq.conv3x3_workspace_bytes(B, H, W, Cin, Cout, stride, bits, 16)) if use_ws else None
    y = mixdq.conv3x3(dev(X), packed, Cout, bits, s, z, 16, None, dev(b), stride, ws, st)
    torch.cuda.synchronize()
    assert int(host(st)[0]) == 0
    assert_close(host(y), y_ref)
