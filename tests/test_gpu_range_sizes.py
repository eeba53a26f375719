"""Activation ranges at the sizes where their kernels change: scalar and vector rows, one and several CTAs of the
cluster, its 8 MiB limit, skipped rows; and weight packing on both sides of the row lengths that one warp takes."""
import numpy as np
import pytest
import torch

from oracle import mixdq_oracle as orc
from paper_2405_17873_b200 import mixdq, synth
from helpers import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols", [(1, 1), (3, 7), (1, 8), (1, 8192), (1, 8200), (77, 2048), (1024, 1280), (4096, 1024),
                                       (4097, 1024), (2053, 2049)])
def test_ranges(rows, cols):
    X = synth.normal_f16((rows, cols), 1.0, seed=rows + cols)
    X[-1, -1], X[0, 0] = np.float16(-9.5), np.float16(7.25)
    Xd = dev(X)
    amax = orc.act_absmax(X)
    assert host(mixdq.act_absmax(Xd))[0] == amax == np.abs(X).max()
    assert host(mixdq.act_scale(Xd))[0] == orc.act_scale(amax, 8)
    assert host(mixdq.act_scale_from_absmax(mixdq.act_absmax(Xd)))[0] == orc.act_scale(amax, 8)
    lo, hi = (float(v) for v in host(mixdq.act_minmax(Xd)))
    assert (lo, hi) == (min(float(X.min()), 0.0), max(float(X.max()), 0.0))
    s_ref, z_ref = orc.act_minmax_params(X)
    s, z = mixdq.act_asym_params(Xd)
    assert host(s)[0] == np.float32(s_ref) and int(host(z)[0]) == int(z_ref)
    zeros = torch.zeros_like(Xd)
    assert host(mixdq.act_scale(zeros))[0] == 1.0
    s, z = mixdq.act_asym_params(zeros)
    assert host(s)[0] == 1.0 and int(host(z)[0]) == 0


@pytest.mark.parametrize("rows,cols", [(77, 2048), (154, 40), (231, 13), (77 * 40, 2048)])
def test_skipped_rows(rows, cols):
    X = synth.normal_f16((rows, cols), 1.0, seed=rows)
    X[::77] = np.float16(100.0)
    kept = np.delete(X, np.arange(0, rows, 77), axis=0)
    assert host(mixdq.act_absmax(dev(X), 77))[0] == np.abs(kept).max()


@pytest.mark.parametrize("bits,symmetric", [(2, False), (3, False), (4, True), (8, False), (8, True)])
@pytest.mark.parametrize("K", [31, 129, 4096, 4104, 5001])
def test_pack_row_lengths(bits, symmetric, K):
    W = synth.normal_f16((11, K), 0.02, seed=K)
    s_ref, z_ref = orc.weight_minmax_params(W, bits, symmetric)
    zr = None if symmetric else z_ref
    s, z = mixdq.weight_minmax_params(dev(W), bits, symmetric)
    assert np.array_equal(host(s).view(np.uint32), s_ref.view(np.uint32)) and np.array_equal(host(z), z_ref)
    codes = orc.quantize_weights(W, bits, s_ref, zr)
    for layout in (mixdq.LAYOUT_CANONICAL, mixdq.LAYOUT_DEVICE):
        packed = mixdq.pack_weights(dev(W), bits, s, None if symmetric else z, layout)
        if layout == mixdq.LAYOUT_CANONICAL:
            assert np.array_equal(host(packed).reshape(11, -1), orc.pack_codes(codes, bits, zr))
        assert np.array_equal(host(mixdq.unpack_weights(packed, 11, K, bits, symmetric, layout)), codes)
