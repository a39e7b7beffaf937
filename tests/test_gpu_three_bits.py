"""Layers of three-bit codes on nibbles: signed codes are halves as they are, unsigned activations enter as a - 4 and the epilogue adds the filters' sums.
Whole numbers throughout, so every comparison is exact: extreme codes, padding (whose code 0 becomes -4), channels that end inside a word under
bipolar filters, resident, streamed and prepared filters (the last on int8), items split over a cluster, every kind of output."""
import numpy as np
import pytest
import torch

import oracle
from paper_2207_08820_b200 import api, workloads as wl
from gpu_util import dev

pytestmark = pytest.mark.gpu

SIGNS = [(3, 0, 3, api.SIGNED), (3, 0, 2, api.SIGNED), (3, 0, 2, api.UNSIGNED), (3, 0, 1, api.BIPOLAR), (3, 0, 1, api.SIGNED), (3, api.SIGNED, 3, api.SIGNED),
         (3, api.SIGNED, 1, api.BIPOLAR), (2, 0, 3, api.SIGNED), (1, 0, 3, api.SIGNED), (2, api.SIGNED, 3, api.SIGNED), (1, api.BIPOLAR, 3, api.SIGNED),
         (3, 0, 3, api.UNSIGNED)]       # the last one stays on int8


def codes(rng, shape, bits, sign, extreme):
    if not extreme or sign == api.BIPOLAR:
        return wl.rand_codes(rng, shape, bits, sign)
    lo, hi = wl.code_range(bits, sign)
    return rng.choice(np.array([lo, hi], np.int8), shape)


@pytest.mark.parametrize("a,a_sign,w,w_sign", SIGNS)
@pytest.mark.parametrize("N,C,H,W,O,k,s", [(2, 32, 9, 12, 40, 3, 1), (1, 70, 11, 7, 33, 3, 2), (3, 96, 8, 8, 130, 1, 1), (1, 33, 20, 5, 64, 5, 1), (2, 256, 7, 7, 96, 3, 1),
                                           (1, 640, 6, 6, 300, 3, 1)])
def test_layers(N, C, H, W, O, k, s, a, a_sign, w, w_sign):
    rng = np.random.default_rng(C + O + a)
    pad = 0 if a_sign == api.BIPOLAR else k // 2
    for extreme in (False, True):
        x, f = codes(rng, (N, C, H, W), a, a_sign, extreme), codes(rng, (O, C, k, k), w, w_sign, extreme)
        want = oracle.conv2d_i32(x, f, s, pad)
        xa, wp = api.bitpack_activations(dev(x), 1.0, a, a_sign), api.pack_weights(dev(f), w, w_sign)
        spread = np.sqrt(C * k * k) * 3.0
        scale, bias = np.full(O, 1.0 / spread, np.float32), (-want.mean((0, 2, 3)) / spread + np.linspace(-1, 4, O)).astype(np.float32)
        forms = [dict()]
        if C % 32 == 0 and api.tc_supported(N, C, H, W, O, k, s, pad, a, a_sign, w, w_sign):
            forms += [dict(wgt_tc=api.tc_prepare_weights(wp, C, w_sign, p)) for p in (a, 4)]
        kw = dict(C=C, stride=s, pad=pad, a_sign=a_sign, w_sign=w_sign)
        for form in forms:
            for layout, w_ in ((api.NCHW, want), (api.NHWC, np.moveaxis(want, 1, 3))):
                acc, _ = api.bitserial_conv2d(xa, wp, want_i32=True, i32_layout=layout, **kw, **form)
                assert np.array_equal(acc.cpu().numpy(), w_)
            for out_bits in (1, 2, 3):
                _, got = api.bitserial_conv2d(xa, wp, scale=dev(scale), bias=dev(bias), relu=True, out_bits=out_bits, **kw, **form)
                assert np.array_equal(api.bitunpack_activations(got, O, out_bits).cpu().numpy(), oracle.requantize(want, scale, bias, True, out_bits))
            # both outputs, and a scale only the formula takes
            tiny = scale.copy()
            tiny[0] = 1e-19
            for sc in (scale, tiny):
                acc, got = api.bitserial_conv2d(xa, wp, scale=dev(sc), bias=dev(bias), out_bits=3, out_sign=api.SIGNED, want_i32=sc is scale, **kw, **form)
                assert np.array_equal(api.bitunpack_activations(got, O, 3, api.SIGNED).cpu().numpy(), oracle.requantize(want, sc, bias, False, 3, api.SIGNED))
        api.bs_check_status()


@pytest.mark.parametrize("M,N,K", [(100, 64, 4608), (333, 70, 1000), (1000, 600, 576), (129, 257, 64)])
@pytest.mark.parametrize("a,a_sign,w,w_sign", SIGNS[:4] + SIGNS[5:8])
def test_products(M, N, K, a, a_sign, w, w_sign):
    """Long reductions of few tiles are split over a cluster where the filters are streamed: signed activations on nibbles, unsigned ones on int8."""
    rng = np.random.default_rng(M + K)
    x, f = codes(rng, (M, K), a, a_sign, True), codes(rng, (N, K), w, w_sign, True)
    want = oracle.gemm_i32(x, f)
    ap, wp = api.bs_pack_rows(dev(x), a, a_sign), api.bs_pack_rows(dev(f), w, w_sign)
    got, _ = api.bitserial_gemm(ap, wp, K, a_sign=a_sign, w_sign=w_sign)
    assert np.array_equal(got.cpu().numpy(), want)
    if K % 64 == 0 and api.tc_supported(1, K, 1, M, N, 1, 1, 0, a, a_sign, w, w_sign):
        wt = api.tc_prepare_weights(wp.view(N, 1, 1, -1, w), K, w_sign, a)
        got, _ = api.bitserial_gemm_tc(ap, wt, N, K, w, a_sign=a_sign, w_sign=w_sign)
        assert np.array_equal(got.cpu().numpy(), want)
    api.bs_check_status()


def test_residual_of_three_bits():
    rng = np.random.default_rng(5)
    N, C, H, O = 2, 96, 10, 64
    x, f, r = wl.rand_codes(rng, (N, C, H, H), 3, 0), wl.rand_codes(rng, (O, C, 3, 3), 3, 1), wl.rand_codes(rng, (N, O, H, H), 3, 0)
    want = oracle.conv2d_i32(x, f, 1, 1)
    scale, bias = np.full(O, 0.01, np.float32), np.linspace(-1, 4, O).astype(np.float32)
    _, got = api.bitserial_conv2d(api.bitpack_activations(dev(x), 1.0, 3), api.pack_weights(dev(f), 3, 1), C=C, pad=1, scale=dev(scale), bias=dev(bias), relu=True,
                                  out_bits=3, residual=api.bitpack_activations(dev(r), 1.0, 3), res_scale=0.5, res_bits=3)
    assert np.array_equal(api.bitunpack_activations(got, O, 3).cpu().numpy(), oracle.requantize(want, scale, bias, True, 3, 0, r, 0.5))
    api.bs_check_status()


@pytest.mark.parametrize("w_sign", [api.SIGNED, api.UNSIGNED])
def test_prepared_filters_serve_every_width(w_sign):
    """Whatever width three-bit filters were prepared for, no layer converts them: their int8 form is in front, nibbles behind it where such layers take them."""
    rng = np.random.default_rng(3)
    w = wl.rand_codes(rng, (70, 128, 3, 3), 3, w_sign)
    wp = api.pack_weights(dev(w), 3, w_sign)
    made = [api.tc_prepare_weights(wp, 128, w_sign, a) for a in (1, 2, 3, 4)]
    int8 = made[3]
    assert all(torch.equal(t[:int8.numel()], int8) for t in made) and made[2].numel() == int8.numel()
    assert all(t.numel() == (2 if w_sign == api.SIGNED else 1) * int8.numel() for t in made[:2])
    for a in (1, 2, 3, 4):
        x = wl.rand_codes(rng, (2, 128, 8, 8), a, 0)
        want, xa = oracle.conv2d_i32(x, w, 1, 1), api.bitpack_activations(dev(x), 1.0, a)
        for t in made:
            part, sign = api.tc_weights_form(t, wp.shape, 128, w_sign, a)
            assert (sign == api.SIGNED_NIBBLES) == (a <= 2 and t.numel() > int8.numel())
            assert int(part[-4:].view(torch.int32)) == -0x77777778 if sign == api.SIGNED_NIBBLES else torch.equal(part[:int8.numel()], int8)
            assert sum(v.numel() for v in api.tc_weights_read(t, wp.shape, 128, a)) == (2 * 128 * 9 * 32 + 16 if sign == api.SIGNED_NIBBLES else int8.numel())
            acc, _ = api.bitserial_conv2d(xa, wp, C=128, pad=1, w_sign=w_sign, want_i32=True, wgt_tc=t)
            assert np.array_equal(acc.cpu().numpy(), want)
    api.bs_check_status()
