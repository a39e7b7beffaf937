"""The popcount kernels behind bitserial_conv2d, reached where the tensor-core kernel refuses a layer: residual slices that start inside a channel
word (every width of activations, filters, residual and output codes; output slices; both strides; few and many tiles), and bipolar activations
times bipolar filters with a ragged channel word.  Integers and codes equal the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2207_08820_b200 import workloads as wl
from gpu_util import gpu_conv

pytestmark = pytest.mark.gpu

#          N   C    H   W    O  k  s
SHAPES = [(2, 64, 12, 12, 64, 3, 1), (1, 33, 7, 9, 40, 3, 2), (3, 128, 28, 28, 128, 1, 1), (1, 70, 31, 56, 31, 5, 1), (8, 96, 40, 37, 96, 3, 1)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("a", [1, 2, 3, 4])
@pytest.mark.parametrize("w", [1, 2, 3, 4])
def test_residual_slice_inside_a_word(shape, a, w):
    N, C, H, W, O, k, s = shape
    out, res_bits = 1 + (a + w) % 4, 1 + (a + 2 * w) % 4
    res_sign = 1 if res_bits > 1 and w % 2 else 0
    offset = (8, 40, 1, 63)[a - 1]
    c = wl.single_conv_case(seed=100 * a + 10 * w + k, N=N, C=C, H=H, W=W, O=O, k=k, stride=s, pad=k // 2, a_bits=a, w_bits=w, out_bits=out, calibrated=True)
    want = oracle.conv2d_i32(c["x"], c["w"], s, k // 2)
    res = wl.rand_codes(np.random.default_rng(a + w), (N, offset + O + 5, *want.shape[2:]), res_bits, res_sign)
    codes = oracle.requantize(want, c["scale"], c["bias"], True, out, 0, res=res[:, offset:offset + O], res_scale=0.5)
    acc, packed = gpu_conv(c, residual=(res, res_bits, res_sign), res_scale=0.5, res_c_offset=offset, out_c_offset=32)
    assert np.array_equal(acc, want)
    assert np.array_equal(packed[:, :, :, 1:], oracle.pack_activations(codes, out, 0))
    assert not packed[:, :, :, 0].any()


@pytest.mark.parametrize("N,C,H,W,O,k,s", [(2, 70, 8, 8, 33, 3, 1), (1, 33, 15, 11, 64, 5, 2), (4, 300, 14, 14, 96, 1, 1), (16, 50, 30, 30, 128, 3, 1)])
def test_bipolar_operands_with_a_ragged_word(N, C, H, W, O, k, s):
    c = wl.single_conv_case(seed=C, N=N, C=C, H=H, W=W, O=O, k=k, stride=s, pad=0, a_bits=1, a_sign=2, w_bits=1, w_sign=2, calibrated=True)
    want = oracle.conv2d_i32(c["x"], c["w"], s, 0)
    codes = oracle.requantize(want, c["scale"], c["bias"], True, 2, 0)
    acc, packed = gpu_conv(c)
    assert np.array_equal(acc, want)
    assert np.array_equal(packed, oracle.pack_activations(codes, 2, 0))
