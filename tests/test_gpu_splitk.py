"""GPU parity for the `*_ws` entry points: bit-identical to the oracle and to the calls without a workspace, workspace left zero, repeated calls
on one workspace.  Products and layers of the tensor-core kernel leave the workspace alone; what that kernel refuses (bipolar operands on
both sides with a ragged channel word, residual slices that start inside a channel word) runs on the popcount kernels and is split."""
import numpy as np
import pytest
import torch

import oracle
from paper_2207_08820_b200 import api, workloads as wl
from gpu_util import dev, words

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(256, 256, 4608), (256, 256, 576), (64, 96, 2304), (130, 40, 1000)])
@pytest.mark.parametrize("wb,wsg", [(1, 2), (2, 1)])
def test_gemm_split_matches_oracle_and_leaves_workspace_zero(M, N, K, wb, wsg):
    c = wl.gemm_case(M, N, K, seed=M + K + wb, w_bits=wb, w_sign=wsg)
    ap = api.bs_pack_rows(dev(c["a"]), 2, 0)
    wp = api.bs_pack_rows(dev(c["w"]), wb, wsg)
    ws = api.gemm_workspace(M, N, K, 2, 0, wb, wsg)
    want = oracle.gemm_i32(c["a"], c["w"])
    if ws is None:
        pytest.skip("planner does not split this shape")
    scale, bias = wl.calibrated_scale_bias(c["w"], 2, 0, 2)
    codes = oracle.requantize(want, scale, bias, True, 2, 0, channel_axis=1)
    for _ in range(3):                                   # the workspace is reused without clearing
        out, packed = api.bitserial_gemm(ap, wp, K, a_sign=0, w_sign=wsg, scale=dev(scale), bias=dev(bias), relu=True,
                                         out_bits=2, workspace=ws)
        api.bs_check_status()
        assert np.array_equal(out.cpu().numpy(), want)
        assert np.array_equal(words(packed), oracle.pack_rows(codes, 2, 0))
        assert int(ws.abs().max()) == 0
    plain, _ = api.bitserial_gemm(ap, wp, K, a_sign=0, w_sign=wsg)
    assert torch.equal(plain, out)


def test_conv_split_deep_reduction():
    """7 x 7 layer with 512 channels at batch 4: few tiles, 144 reduction words."""
    c = wl.single_conv_case(seed=21, N=4, C=512, H=7, W=7, O=512, calibrated=True)
    ws = api.conv_workspace(4, 512, 7, 7, 512, 3, 1, 1, 2, 0, 2, 1)
    assert ws is not None
    x, w = dev(c["x"]), dev(c["w"])
    xa = api.bitpack_activations(x, 1.0, 2, 0, api.NCHW)
    wp = api.pack_weights(w, 2, 1, api.NCHW)
    want = oracle.conv2d_i32(c["x"], c["w"], 1, 1)
    codes = oracle.requantize(want, c["scale"], c["bias"], True, 2, 0)
    for _ in range(2):
        acc, packed = api.bitserial_conv2d(xa, wp, C=512, stride=1, pad=1, w_sign=1, scale=dev(c["scale"]), bias=dev(c["bias"]),
                                           relu=True, out_bits=2, want_i32=True, workspace=ws)
        api.bs_check_status()
        assert np.array_equal(acc.cpu().numpy(), want)
        assert np.array_equal(words(packed), oracle.pack_activations(codes, 2, 0))
        assert int(ws.abs().max()) == 0


def test_too_small_workspace_falls_back():
    c = wl.gemm_case(256, 256, 4608, seed=3)
    ap = api.bs_pack_rows(dev(c["a"]), 2, 0)
    wp = api.bs_pack_rows(dev(c["w"]), 1, 2)
    tiny = torch.zeros(4, dtype=torch.int32, device="cuda")
    out, _ = api.bitserial_gemm(ap, wp, 4608, a_sign=0, w_sign=2, workspace=tiny)
    api.bs_check_status()
    assert np.array_equal(out.cpu().numpy(), oracle.gemm_i32(c["a"], c["w"]))


def mark_workspace(ws):
    """Adds one to the first partial sum: a kernel that sums in the workspace returns it in one accumulator and clears it."""
    ws[0] += 1


@pytest.mark.parametrize("M,N,K", [(256, 256, 4600), (64, 96, 2290), (130, 40, 3333)])
def test_bipolar_product_split_sums_in_the_workspace(M, N, K):
    c = wl.gemm_case(M, N, K, seed=M + K, a_bits=1, a_sign=2, w_bits=1, w_sign=2)
    ap, wp = api.bs_pack_rows(dev(c["a"]), 1, 2), api.bs_pack_rows(dev(c["w"]), 1, 2)
    ws = api.gemm_workspace(M, N, K, 1, 2, 1, 2)
    assert ws is not None
    want = oracle.gemm_i32(c["a"], c["w"])
    scale, bias = wl.calibrated_scale_bias(c["w"], 1, 2, 2)
    codes = oracle.requantize(want, scale, bias, True, 2, 0, channel_axis=1)
    for _ in range(3):
        out, packed = api.bitserial_gemm(ap, wp, K, a_sign=2, w_sign=2, scale=dev(scale), bias=dev(bias), relu=True, out_bits=2, workspace=ws)
        api.bs_check_status()
        assert np.array_equal(out.cpu().numpy(), want)
        assert np.array_equal(words(packed), oracle.pack_rows(codes, 2, 0))
        assert int(ws.abs().max()) == 0
    mark_workspace(ws)
    out, _ = api.bitserial_gemm(ap, wp, K, a_sign=2, w_sign=2, workspace=ws)
    diff = out.cpu().numpy() - want
    assert (diff != 0).sum() == 1 and diff.max() == 1 and int(ws.abs().max()) == 0
    plain, _ = api.bitserial_gemm(ap, wp, K, a_sign=2, w_sign=2)
    assert np.array_equal(plain.cpu().numpy(), want)


@pytest.mark.parametrize("a,w", [(1, 2), (2, 2), (3, 1), (4, 3)])
def test_layer_split_with_a_residual_slice_inside_a_word(a, w):
    """7 x 7 layers of 512 channels whose residual starts at channel 24 of a wider tensor: the popcount kernels, split."""
    N, C, HW, O = 2, 512, 7, 96
    c = wl.single_conv_case(seed=60 + a, N=N, C=C, H=HW, W=HW, O=O, a_bits=a, w_bits=w, calibrated=True)
    ws = api.conv_workspace(N, C, HW, HW, O, 3, 1, 1, a, 0, w, c["w_sign"])
    assert ws is not None
    res = wl.rand_codes(np.random.default_rng(a), (N, 160, HW, HW), 2, 0)
    xa, wp, rp = api.bitpack_activations(dev(c["x"]), 1.0, a), api.pack_weights(dev(c["w"]), w, c["w_sign"]), api.bitpack_activations(dev(res), 1.0, 2)
    want = oracle.conv2d_i32(c["x"], c["w"], 1, 1)
    codes = oracle.requantize(want, c["scale"], c["bias"], True, 2, 0, res=res[:, 24:24 + O], res_scale=0.5)
    run = lambda **kw: api.bitserial_conv2d(xa, wp, C=C, pad=1, w_sign=c["w_sign"], scale=dev(c["scale"]), bias=dev(c["bias"]), relu=True, out_bits=2,
                                            residual=rp, res_scale=0.5, res_bits=2, res_c_offset=24, res_c_total=160, want_i32=True, **kw)
    for _ in range(2):
        acc, packed = run(workspace=ws)
        api.bs_check_status()
        assert np.array_equal(acc.cpu().numpy(), want)
        assert np.array_equal(words(packed), oracle.pack_activations(codes, 2, 0))
        assert int(ws.abs().max()) == 0
    mark_workspace(ws)
    acc, _ = run(workspace=ws)
    assert (acc.cpu().numpy() != want).sum() == 1 and int(ws.abs().max()) == 0
    acc, packed = run()
    assert np.array_equal(acc.cpu().numpy(), want)
    assert np.array_equal(words(packed), oracle.pack_activations(codes, 2, 0))
