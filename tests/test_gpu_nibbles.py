"""Layers of one- and two-bit codes (operands of nibbles, sums in binary32) where exactness could end: sums up to the limit of the form, all bits of
them in use, at both sides of the reduction length from which int8 takes over; every pair of signs; odd numbers of channel words."""
import numpy as np
import pytest
import torch

import oracle
from paper_2207_08820_b200 import api, workloads as wl
from gpu_util import dev

pytestmark = pytest.mark.gpu

LIMIT = 4000000 // 9 // 32 * 32         # longest reduction on nibbles: C * R * S * 9 below 4 million


@pytest.mark.parametrize("K", [LIMIT, LIMIT + 32])
@pytest.mark.parametrize("form", ["largest codes", "sums that rise and fall", "random"])
def test_longest_reductions(K, form):
    """Whole numbers stay exact in binary32 below 2^24, so the comparison has no tolerance."""
    rng = np.random.default_rng(K)
    M, N = 130, 40
    if form == "random":
        a, w, ws = wl.rand_codes(rng, (M, K), 2, 0), wl.rand_codes(rng, (N, K), 2, api.SIGNED), api.SIGNED
    else:
        a, w, ws = np.full((M, K), 3, np.int8), np.full((N, K), 3, np.int8), api.UNSIGNED
        a[rng.random((M, K)) < 0.001] = 1
        if form == "sums that rise and fall":
            w[:], ws = -2, api.SIGNED
            w[:, K // 2:] = 1
    want = oracle.gemm_i32(a, w)
    ap, wp = api.bs_pack_rows(dev(a), 2, 0), api.bs_pack_rows(dev(w), 2, ws)
    got, _ = api.bitserial_gemm(ap, wp, K, w_sign=ws)
    assert np.array_equal(got.cpu().numpy(), want)
    wt = api.tc_prepare_weights(wp.view(N, 1, 1, -1, 2), K, ws, 2)
    got, _ = api.bitserial_gemm_tc(ap, wt, N, K, 2, a_sign=0, w_sign=ws)
    api.bs_check_status()
    assert np.array_equal(got.cpu().numpy(), want)


@pytest.mark.parametrize("a,a_sign,w,w_sign", [(1, 0, 1, 2), (1, 1, 1, 0), (1, 2, 1, 2), (1, 2, 2, 1), (1, 0, 1, 1), (2, 0, 2, 0), (2, 1, 2, 1), (2, 1, 1, 2), (2, 0, 2, 1)])
@pytest.mark.parametrize("C,O,k,s", [(32, 40, 3, 1), (96, 33, 1, 1), (64, 64, 3, 2), (160, 130, 5, 1)])
def test_signs(C, O, k, s, a, a_sign, w, w_sign):
    rng = np.random.default_rng(C + a + w)
    x, f = wl.rand_codes(rng, (2, C, 9, 12), a, a_sign), wl.rand_codes(rng, (O, C, k, k), w, w_sign)
    pad = 0 if a_sign == api.BIPOLAR else k // 2
    want = oracle.conv2d_i32(x, f, s, pad)
    xa, wp = api.bitpack_activations(dev(x), 1.0, a, a_sign), api.pack_weights(dev(f), w, w_sign)
    forms = [dict()]
    if api.tc_supported(2, C, 9, 12, O, k, s, pad, a, a_sign, w, w_sign):
        forms.append(dict(wgt_tc=api.tc_prepare_weights(wp, C, w_sign, a)))
    for kw in forms:
        acc, _ = api.bitserial_conv2d(xa, wp, C=C, stride=s, pad=pad, a_sign=a_sign, w_sign=w_sign, want_i32=True, **kw)
        assert np.array_equal(acc.cpu().numpy(), want)
    api.bs_check_status()


# resident and streamed filters, an odd number of channel words, rows by tensor copies, five taps a side
@pytest.mark.parametrize("C,O,k,hw", [(32, 128, 3, 8), (64, 128, 3, 8), (96, 128, 3, 8), (64, 40, 5, 9), (512, 256, 1, 12), (1024, 300, 3, 10)])
@pytest.mark.parametrize("prepared,run", [(2, 3), (4, 1), (2, 1), (3, 4), (3, 2), (2, 4)])
@pytest.mark.parametrize("w,w_sign", [(2, api.SIGNED), (1, api.BIPOLAR), (2, api.UNSIGNED), (1, api.SIGNED)])
def test_filters_prepared_for_other_widths(C, O, k, hw, prepared, run, w, w_sign):
    """One prepared tensor serves every activation width, whatever form it has (int8 ones saved by earlier versions among them)."""
    rng = np.random.default_rng(C)
    x, f = wl.rand_codes(rng, (1, C, hw, hw), run, 0), wl.rand_codes(rng, (O, C, k, k), w, w_sign)
    xa, wp = api.bitpack_activations(dev(x), 1.0, run), api.pack_weights(dev(f), w, w_sign)
    if not api.tc_supported(1, C, hw, hw, O, k, 1, k // 2, run, 0, w, w_sign):
        pytest.skip("records of other sizes take no prepared filters")
    wt = api.tc_prepare_weights(wp, C, w_sign, prepared)
    want = oracle.conv2d_i32(x, f, 1, k // 2)
    for chained in (False, True):
        torch.cuda.synchronize()
        acc, _ = api.bitserial_conv2d(xa, wp, C=C, pad=k // 2, w_sign=w_sign, want_i32=True, wgt_tc=wt, chained=chained)
        api.bs_check_status()
        assert np.array_equal(acc.cpu().numpy(), want)


@pytest.mark.parametrize("prepared,run", [(2, 3), (4, 1)])
@pytest.mark.parametrize("M,N,K", [(300, 70, 4032), (1000, 1024, 512), (3000, 600, 64)])
def test_products_with_filters_prepared_for_other_widths(M, N, K, prepared, run):
    rng = np.random.default_rng(K)
    a, w = wl.rand_codes(rng, (M, K), run, 0), wl.rand_codes(rng, (N, K), 2, api.SIGNED)
    wp = api.bs_pack_rows(dev(w), 2, api.SIGNED)
    assert api.tc_supported(1, K, 1, M, N, 1, 1, 0, run, 0, 2, api.SIGNED)
    wt = api.tc_prepare_weights(wp.view(N, 1, 1, -1, 2), K, api.SIGNED, prepared)
    got, _ = api.bitserial_gemm_tc(api.bs_pack_rows(dev(a), run, 0), wt, N, K, 2)
    api.bs_check_status()
    assert np.array_equal(got.cpu().numpy(), oracle.gemm_i32(a, w))


# both sides of the lines at which packed filters of one- and two-bit layers go to int8: channels of 1x1 layers, one channel word and more, few outputs
# and many (a few more than 2048 for each of 148 SMs), windows of codes
@pytest.mark.parametrize("C,O,k,N,hw,out", [(9, 33, 1, 2, 13, "acc"), (192, 40, 1, 2, 13, "acc"), (193, 40, 1, 2, 13, "acc"), (32, 66, 3, 4, 34, "acc"), (33, 66, 3, 4, 34, "acc"),
                                            (20, 66, 5, 4, 34, "acc"), (20, 8, 5, 1, 9, "acc"), (32, 66, 5, 4, 34, "codes"), (31, 64, 5, 1, 9, "codes"), (32, 65, 7, 4, 35, "codes"),
                                            (32, 66, 3, 4, 34, "codes")])
@pytest.mark.parametrize("a,a_sign,w,w_sign", [(2, 0, 2, 1), (1, 0, 1, 2), (2, 1, 1, 1), (1, 0, 2, 1)])
def test_lines_between_the_forms(C, O, k, N, hw, out, a, a_sign, w, w_sign):
    rng = np.random.default_rng(C + O)
    x, f = wl.rand_codes(rng, (N, C, hw, hw), a, a_sign), wl.rand_codes(rng, (O, C, k, k), w, w_sign)
    xa, wp = api.bitpack_activations(dev(x), 1.0, a, a_sign), api.pack_weights(dev(f), w, w_sign)
    kw = dict(C=C, stride=1, pad=k // 2, a_sign=a_sign, w_sign=w_sign)
    want = oracle.conv2d_i32(x, f, 1, k // 2)
    if out == "acc":
        got, _ = api.bitserial_conv2d(xa, wp, want_i32=True, **kw)
        assert np.array_equal(got.cpu().numpy(), want)
    else:
        scale, bias = np.full(O, 0.03, np.float32), np.linspace(-1.0, 2.0, O, dtype=np.float32)
        _, got = api.bitserial_conv2d(xa, wp, scale=dev(scale), bias=dev(bias), relu=True, out_bits=2, **kw)
        assert np.array_equal(api.bitunpack_activations(got, O, 2).cpu().numpy(), oracle.requantize(want, scale, bias, True, 2))
    api.bs_check_status()
