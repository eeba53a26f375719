"""The kernels' bounded waits end in a status word.

Every wait on a shared-memory barrier in the tensor-core kernels has a cycle budget; when it runs out the
kernel raises an abort flag, lets its copies in flight land, reports MIXDQ_ERR_TIMEOUT through the caller's
status word, releases its tensor memory and returns.  The self-test entry points make that happen without any
fault: weight tiles are never requested.  Afterwards the same GPU context runs an ordinary layer with full parity
against the oracle."""
import time

import numpy as np
import pytest
import torch

from oracle import mixdq_oracle as orc
from paper_2405_17873_b200 import mixdq, synth
from helpers import assert_close, dev, device_weights, host, oracle_weights, status_word, workspace_for

pytestmark = pytest.mark.gpu

MIXDQ_ERR_TIMEOUT = -6


@pytest.mark.parametrize("bits,M,N,K,drop", [(8, 128, 128, 512, 2), (4, 256, 384, 1280, 7), (8, 4096, 2048, 512, 1)])
def test_abandoned_wait_reports_timeout_and_context_survives(bits, M, N, K, drop):
    X = synth.normal_f16((M, K), 1.0, seed=61)
    W = synth.normal_f16((N, K), 0.02, seed=62)
    Xd = dev(X)
    s, _, packed = device_weights(W, bits, True)
    sx = mixdq.act_scale(Xd)
    xq = mixdq.quantize_acts(Xd, sx)
    st = status_word()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    mixdq.selftest_abandoned_wait(xq, packed, N, bits, s, sx, drop, st)
    torch.cuda.synchronize()                     # returns: the kernel gave up by itself
    dt = time.perf_counter() - t0
    assert int(host(st)[0]) == MIXDQ_ERR_TIMEOUT
    assert dt < 20.0, dt
    # the context is intact and tensor memory was released: the same layer, ordinary call, full parity
    st2 = status_word()
    s_ref, _, codes = oracle_weights(W, bits, True)
    sx_ref = orc.act_scale(orc.act_absmax(X), 8)
    acc_ref, y_ref = orc.linear_a8(X, codes, s_ref, sx_ref, None)
    ws = workspace_for(M, N, K, bits)
    acc = mixdq.linear_acc_i32(Xd, packed, N, bits, sx, workspace=ws, status=st2)
    y = mixdq.linear(Xd, packed, N, bits, s, None, 8, sx, None, workspace=ws, status=st2)
    torch.cuda.synchronize()
    assert int(host(st2)[0]) == 0
    assert np.array_equal(host(acc), acc_ref)
    assert_close(host(y), y_ref)


def _gives_up(call, status):
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    call()
    torch.cuda.synchronize()                     # returns: the kernel gave up by itself
    assert time.perf_counter() - t0 < 20.0
    assert int(host(status)[0]) == MIXDQ_ERR_TIMEOUT


# one- and two-CTA tiles, tiles that a CTA pair walks one after another; the first weight tile, one in the middle, the last
# (int8 layers of one wave: always the first)
@pytest.mark.parametrize("bits,act_bits,M,N,K,drop,form", [
    (8, 8, 100, 320, 640, 1, "chan"), (4, 8, 256, 1280, 1296, 1, "chan"), (4, 8, 1024, 1280, 2560, 1, "chan"),
    (8, 8, 1024, 1280, 2560, 1, "chan"), (4, 8, 1024, 10240, 1536, 11, "chan_many"), (4, 8, 4096, 5120, 640, 3, "chan_many"), (4, 8, 1024, 10240, 1280, 1, "chan_many"),
    (3, 16, 64, 320, 1288, 1, None), (4, 16, 1024, 1280, 2560, 11, None), (8, 16, 300, 1280, 648, 5, None),
    (8, 16, 300, 1280, 1024, 8, None)])
def test_abandoned_wait_in_the_channel_major_kernels(bits, act_bits, M, N, K, drop, form):
    if form:
        assert mixdq.int8_layer_plan(M, N, -(-K // 128), bits, "codes")[0] == form
    X, W = synth.normal_f16((M, K), 1.0, seed=61), synth.normal_f16((N, K), 0.02, seed=62)
    Xd = dev(X)
    symmetric = act_bits == 8
    s, z, packed = device_weights(W, bits, symmetric)
    s_ref, z_ref, codes = oracle_weights(W, bits, symmetric)
    sx = mixdq.act_scale(Xd) if symmetric else None
    rows = mixdq.quantize_acts(Xd, sx) if symmetric else Xd
    st, st2 = status_word(), status_word()
    _gives_up(lambda: mixdq.selftest_abandoned_chan_wait(rows, packed, N, bits, s, z, act_bits, sx, drop, st), st)
    if symmetric:
        acc_ref, y_ref = orc.linear_a8(X, codes, s_ref, orc.act_scale(orc.act_absmax(X), 8), None)
        assert np.array_equal(host(mixdq.linear_q8_acc_i32(rows, packed, N, bits, st2)), acc_ref)
        y = mixdq.linear_q8(rows, packed, N, bits, s, sx, None, st2)
    else:
        y_ref = orc.linear_a16(X, codes, s_ref, z_ref, None)
        y = mixdq.linear(Xd, packed, N, bits, s, z, 16, None, None, None, st2)
    torch.cuda.synchronize()
    assert int(host(st2)[0]) == 0
    assert_close(host(y), y_ref)


@pytest.mark.parametrize("bits,M,N,lo,hi", [(8, 100, 320, 640, 640), (4, 1024, 1280, 1280, 1280), (4, 100, 320, 512, 384),
                                               # the last pair of k-blocks alone, which is not the first issuer's: that one has long finished
                                               (8, 100, 320, 640, 128), (4, 1024, 1280, 640, 128)])
def test_abandoned_wait_in_the_second_branch(bits, M, N, lo, hi):
    assert mixdq.int8_layer_plan(M, N, -(-lo // 128) - (-hi // 128), bits, "split")[0] == "chan"
    X, W = synth.normal_f16((M, lo + hi), 1.0, seed=61), synth.normal_f16((N, lo + hi), 0.02, seed=62)
    Xd, Wd = dev(X), dev(W)
    s, _ = mixdq.weight_minmax_params(Wd, bits, True)
    packed = [mixdq.pack_weights(w.contiguous(), bits, s) for w in (Wd[:, :lo], Wd[:, lo:])]
    sx = mixdq.act_scale(Xd)
    rows = [mixdq.quantize_acts(x.contiguous(), sx) for x in (Xd[:, :lo], Xd[:, lo:])]
    st, st2 = status_word(), status_word()
    _gives_up(lambda: mixdq.selftest_abandoned_chan_wait(rows[0], packed[0], N, bits, s, None, 8, sx, 1, st, rows[1], packed[1]), st)
    s_ref, _, codes = oracle_weights(W, bits, True)
    sx_ref = orc.act_scale(orc.act_absmax(X), 8)
    _, _, y_ref = orc.linear_a8_split(X, codes, s_ref, sx_ref, sx_ref, lo, None)
    ws = mixdq.new_workspace(mixdq.split_workspace_bytes(M, lo + hi, lo, M, N))
    y = mixdq.linear_a8_split(Xd, lo, packed[0], packed[1], N, bits, s, sx, sx, workspace=ws, status=st2)
    torch.cuda.synchronize()
    assert int(host(st2)[0]) == 0
    assert_close(host(y), y_ref)


def test_channel_major_self_test_on_another_kernel_is_refused():
    Xq = torch.zeros((2100, 208), dtype=torch.int8, device="cuda")
    s, _, packed = device_weights(synth.normal_f16((1000, 208), 0.02, seed=62), 8, True)
    assert mixdq.int8_layer_plan(2100, 1000, 2, 8, "codes")[0] == "single"
    with pytest.raises(mixdq.MixdqError, match="unsupported"):
        mixdq.selftest_abandoned_chan_wait(Xq, packed, 1000, 8, s, None, 8, mixdq.act_scale(dev(synth.normal_f16((8, 8), 1.0, 1))), 1,
                                           status_word())
