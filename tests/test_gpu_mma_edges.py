"""The tensor-core kernel at the edges of its dispatch: filters prepared or packed, resident or streamed; rows fetched by tensor copies or
by threads; strips of wide images; parity planes of stride 2; items split over a cluster (few tiles, long reductions, shares of
unequal length); outputs of every width and the formula instead of the fast requantisation."""
import numpy as np
import pytest

import oracle
from paper_2207_08820_b200 import api, workloads as wl
from gpu_util import dev, words

pytestmark = pytest.mark.gpu

#        N    C   H   W    O  k  s  a  w  out
CASES = [(1, 512, 7, 7, 96, 3, 1, 2, 2, 2), (2, 416, 5, 9, 64, 3, 1, 1, 2, 1), (1, 350, 8, 6, 40, 3, 2, 3, 1, 3), (1, 2048, 7, 7, 64, 1, 1, 2, 2, 4),
         (1, 1600, 5, 5, 33, 1, 1, 2, 3, 2), (1, 1300, 3, 3, 32, 1, 2, 4, 2, 2), (1, 288, 9, 9, 32, 5, 1, 2, 2, 2), (3, 33, 17, 130, 31, 3, 1, 2, 1, 2),
         (1, 64, 5, 300, 64, 3, 2, 2, 2, 2), (2, 96, 31, 30, 160, 3, 2, 1, 1, 2), (5, 64, 16, 16, 256, 1, 1, 2, 2, 2), (1, 32, 1, 1, 32, 1, 1, 2, 2, 2)]


@pytest.mark.parametrize("N,C,H,W,O,k,s,a,w,out", CASES)
def test_layer_against_oracle(N, C, H, W, O, k, s, a, w, out):
    rng = np.random.default_rng(C + O)
    w_sign = wl.weight_sign(w)
    x, f = wl.rand_codes(rng, (N, C, H, W), a, 0), wl.rand_codes(rng, (O, C, k, k), w, w_sign)
    pad = k // 2
    want = oracle.conv2d_i32(x, f, s, pad)
    sd = max(float(want.std()), 1.0)
    scale = np.full(O, 2 ** out / (4 * sd), np.float32)
    bias = np.full(O, 2 ** (out - 1), np.float32) - scale * float(want.mean())
    codes = oracle.pack_activations(oracle.requantize(want, scale, bias, True, out, 0), out, 0)
    xa, wp = api.bitpack_activations(dev(x), 1.0, a), api.pack_weights(dev(f), w, w_sign)
    kw = dict(C=C, stride=s, pad=pad, w_sign=w_sign)
    forms = [dict()]
    if api.tc_supported(N, C, H, W, O, k, s, pad, a, 0, w, w_sign):
        forms.append(dict(wgt_tc=api.tc_prepare_weights(wp, C, w_sign, a)))
    for form in forms:
        for layout in (api.NCHW, api.NHWC):
            acc, _ = api.bitserial_conv2d(xa, wp, want_i32=True, i32_layout=layout, **kw, **form)
            assert np.array_equal(acc.cpu().numpy(), want if layout == api.NCHW else want.transpose(0, 2, 3, 1))
        _, got = api.bitserial_conv2d(xa, wp, scale=dev(scale), bias=dev(bias), relu=True, out_bits=out, **kw, **form)
        assert np.array_equal(words(got), codes)
        # a scale below the fast form's range: the formula, one output at a time
        _, got = api.bitserial_conv2d(xa, wp, scale=dev(scale * np.float32(1e-30)), bias=dev(bias), relu=True, out_bits=out, **kw, **form)
        assert np.array_equal(words(got), oracle.pack_activations(oracle.requantize(want, scale * np.float32(1e-30), bias, True, out, 0), out, 0))
    api.bs_check_status()


@pytest.mark.parametrize("M,N,K,a,w", [(1, 32, 4608, 2, 2), (129, 33, 1281, 1, 2), (200, 128, 3000, 3, 3), (256, 64, 576, 2, 1), (64, 300, 2048, 4, 4)])
def test_product_against_oracle(M, N, K, a, w):
    rng = np.random.default_rng(K)
    w_sign = wl.weight_sign(w)
    A, B = wl.rand_codes(rng, (M, K), a, 0), wl.rand_codes(rng, (N, K), w, w_sign)
    got, _ = api.bitserial_gemm(api.bs_pack_rows(dev(A), a, 0), api.bs_pack_rows(dev(B), w, w_sign), K, w_sign=w_sign)
    api.bs_check_status()
    assert np.array_equal(got.cpu().numpy(), oracle.gemm_i32(A, B))
