"""The floating-point layers at the edges of their tiles: each tile shape, 16-byte and 4-byte staging, ragged strips, pooling of rows of
every even width, and the chunks of the fully connected layer."""
import numpy as np
import pytest

import oracle
from paper_2207_08820_b200 import api
from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,O,k,stride,pad,H,W", [(3, 64, 7, 2, 3, 64, 64), (3, 65, 7, 2, 3, 16, 128), (3, 64, 7, 2, 3, 130, 32), (3, 64, 7, 2, 3, 82, 164),
                                                  (3, 64, 7, 2, 3, 33, 66), (4, 64, 3, 1, 1, 17, 40), (4, 64, 3, 1, 0, 18, 20), (4, 64, 3, 2, 1, 19, 36),
                                                  (2, 9, 1, 1, 0, 33, 8)])
def test_conv_tiles(C, O, k, stride, pad, H, W):
    rng = np.random.default_rng(H)
    x = rng.normal(0, 1, (2, C, H, W)).astype(np.float32)
    w = rng.normal(0, 0.1, (O, C, k, k)).astype(np.float32)
    b = rng.normal(0, 0.5, O).astype(np.float32)
    got = api.conv2d_f32(dev(x), dev(w), dev(b), stride, pad, True).cpu().numpy()
    assert np.array_equal(got.view(np.uint32), oracle.conv2d_f32(x, w, b, stride, pad, True).view(np.uint32))


@pytest.mark.parametrize("H,W", [(2, 2), (7, 6), (5, 10), (41, 82), (12, 8), (33, 272)])
def test_pool_widths(H, W):
    x = np.random.default_rng(W).normal(-1, 1, (2, 3, H, W)).astype(np.float32)
    got = api.maxpool2d_f32(dev(x), 3, 2, 1).cpu().numpy()
    assert np.array_equal(got, oracle.maxpool2d_f32(x, 3, 2, 1))


@pytest.mark.parametrize("N,K,J", [(17, 64, 32), (16, 65, 33), (1, 68, 1), (33, 260, 64), (2, 511, 31)])
def test_fc_chunks(N, K, J):
    rng = np.random.default_rng(K)
    x, w = rng.normal(0, 1, (N, K)).astype(np.float32), rng.normal(0, 0.1, (J, K)).astype(np.float32)
    b = rng.normal(0, 1, J).astype(np.float32)
    got = api.fc_f32(dev(x), dev(w), dev(b)).cpu().numpy()
    assert np.array_equal(got.view(np.uint32), oracle.fc_f32(x, w, b).view(np.uint32))
