"""Signed output codes without ReLU and without a residual, each layer directly behind a launch that fills most of the shared memory of every
SM with prepared filters of -1 (0xFF bytes, NaN as floats): what a kernel reads there without having written it shows in its codes.
The epilogue takes the oracle's binary32 operations in its order, so the codes must be equal.  And layers without a residual whose other
residual fields hold something: a null pointer means none, whatever they say, in this call and in later ones of the shape."""
import numpy as np
import pytest

import oracle
from paper_2207_08820_b200 import api, workloads as wl
from gpu_util import dev, words

pytestmark = pytest.mark.gpu

# C, O, k of layers whose prepared filters take 36 to 200 KB of a CTA's shared memory, over enough pixels for every SM
FILLERS = [(64, 64, 3), (128, 64, 3), (128, 128, 3), (256, 64, 3), (320, 32, 5), (512, 256, 1)]


@pytest.fixture(scope="module")
def fillers():
    out = []
    for C, O, k in FILLERS:
        x = api.bitpack_activations(dev(np.ones((48, C, 28, 28), np.int8)), 1.0, 2)
        wp = api.pack_weights(dev(np.full((O, C, k, k), -1, np.int8)), 2, api.SIGNED)
        wt = api.tc_prepare_weights(wp, C, api.SIGNED, 2)
        out.append(lambda x=x, wp=wp, wt=wt, C=C, k=k: api.bitserial_conv2d(x, wp, C=C, pad=k // 2, want_i32=True, wgt_tc=wt))
    return out


def signed_layer(N, C, H, W, O, k, stride, a, w, out, seed):
    """Inputs of a layer, its scale and bias (both ends of the code range in use) and the oracle's packed codes."""
    rng = np.random.default_rng(seed)
    w_sign = wl.weight_sign(w)
    x, f = wl.rand_codes(rng, (N, C, H, W), a, 0), wl.rand_codes(rng, (O, C, k, k), w, w_sign)
    acc = oracle.conv2d_i32(x, f, stride, k // 2)
    scale = np.full(O, 2 ** out / (2 * max(float(acc.std()), 1.0)), np.float32)
    bias = (-scale * acc.mean(axis=(0, 2, 3)) - np.float32(0.5)).astype(np.float32)
    codes = oracle.requantize(acc, scale, bias, False, out, oracle.SIGNED)
    assert codes.min() == -(1 << out - 1) and codes.max() == (1 << out - 1) - 1 and len(np.unique(codes)) >= (1 << out) - 1
    return x, f, w_sign, scale, bias, oracle.pack_activations(codes, out, oracle.SIGNED)


#          N   C   H   W    O  k  s  a  w  out
LAYERS = [(3, 64, 11, 13, 72, 3, 1, 2, 2, 2), (8, 64, 56, 56, 64, 3, 1, 2, 2, 3), (4, 128, 28, 28, 128, 3, 1, 2, 1, 4), (2, 96, 17, 20, 40, 3, 2, 1, 2, 2),
          (5, 64, 16, 16, 256, 1, 1, 2, 2, 4), (16, 256, 14, 14, 256, 3, 1, 2, 2, 2), (1, 512, 7, 7, 96, 3, 1, 2, 2, 3)]


@pytest.mark.parametrize("prepared", [False, True])
@pytest.mark.parametrize("layer", LAYERS)
def test_signed_codes_without_residual(fillers, layer, prepared):
    N, C, H, W, O, k, stride, a, w, out = layer
    x, f, w_sign, scale, bias, want = signed_layer(*layer, seed=C + O + out)
    if prepared and not api.tc_supported(N, C, H, W, O, k, stride, k // 2, a, 0, w, w_sign):
        pytest.skip("no prepared filters for this shape")
    xa, wp = api.bitpack_activations(dev(x), 1.0, a), api.pack_weights(dev(f), w, w_sign)
    wt = api.tc_prepare_weights(wp, C, w_sign, a) if prepared else None
    sc, bi = dev(scale), dev(bias)
    for fill in fillers:
        fill()
        _, got = api.bitserial_conv2d(xa, wp, C=C, stride=stride, pad=k // 2, w_sign=w_sign, scale=sc, bias=bi, out_bits=out, out_sign=api.SIGNED, wgt_tc=wt)
        assert np.array_equal(words(got), want)
    api.bs_check_status()


@pytest.mark.parametrize("relu,out_sign", [(False, api.SIGNED), (True, api.SIGNED), (True, api.UNSIGNED)])
@pytest.mark.parametrize("prepared", [False, True])
def test_residual_fields_without_a_residual(relu, out_sign, prepared):
    out, hw = 3, 13 + 2 * prepared + 4 * relu + 8 * out_sign       # a shape that no call has been planned for
    rng = np.random.default_rng(hw)
    x, f = wl.rand_codes(rng, (2, 64, hw, hw), 2, 0), wl.rand_codes(rng, (64, 64, 3, 3), 2, 1)
    acc = oracle.conv2d_i32(x, f, 1, 1)
    scale = np.full(64, 4 / float(acc.std()), np.float32)
    bias = (-scale * acc.mean(axis=(0, 2, 3)) + np.float32(0.25)).astype(np.float32)
    want = oracle.pack_activations(oracle.requantize(acc, scale, bias, relu, out, out_sign), out, out_sign)
    res = wl.rand_codes(rng, (2, 64, hw, hw), 2, 0)
    want_res = oracle.pack_activations(oracle.requantize(acc, scale, bias, relu, out, out_sign, res=res, res_scale=0.5), out, out_sign)
    xa, wp, rp = api.bitpack_activations(dev(x), 1.0, 2), api.pack_weights(dev(f), 2, 1), api.bitpack_activations(dev(res), 1.0, 2)
    kw = dict(C=64, pad=1, scale=dev(scale), bias=dev(bias), relu=relu, out_bits=out, out_sign=out_sign,
              wgt_tc=api.tc_prepare_weights(wp, 64, 1, 2) if prepared else None)
    left = dict(res_scale=0.5, res_bits=2, res_sign=api.UNSIGNED, res_c_offset=32, res_c_total=96)
    for fields, residual, codes in ((left, None, want), ({}, None, want), (dict(left, res_c_offset=0, res_c_total=64), rp, want_res), (left, None, want)):
        _, got = api.bitserial_conv2d(xa, wp, residual=residual, **fields, **kw)
        assert np.array_equal(words(got), codes)
    api.bs_check_status()
