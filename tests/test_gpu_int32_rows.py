"""Accumulators of matrix products whose rows are not multiples of 16 bytes (stored four bytes a lane through shared memory), at the edges of
row tiles and filter groups, on nibbles and on int8."""
import numpy as np
import pytest
import torch

import oracle
from paper_2207_08820_b200 import api, workloads as wl
from gpu_util import Guarded, dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N", [(1, 1), (31, 33), (128, 31), (129, 65), (255, 127), (300, 32), (64, 36), (513, 130)])
@pytest.mark.parametrize("a,w", [(1, 1), (2, 2), (3, 3)])
def test_rows(M, N, a, w):
    rng = np.random.default_rng(M * 7 + N)
    K, ws = 160, wl.weight_sign(w)
    x, f = wl.rand_codes(rng, (M, K), a, api.UNSIGNED), wl.rand_codes(rng, (N, K), w, ws)
    want = oracle.gemm_i32(x, f)
    ap, wp = api.bs_pack_rows(dev(x), a, api.UNSIGNED), api.bs_pack_rows(dev(f), w, ws)
    guard = Guarded()
    out = guard.empty((M, N), fill=-1)
    api.bitserial_conv2d(ap.view(1, 1, M, K // 32, a), wp.view(N, 1, 1, K // 32, w), C=K, w_sign=ws, out_i32=out.view(1, 1, M, N), i32_layout=api.NHWC)
    api.bs_check_status()
    guard.check()
    assert np.array_equal(out.cpu().numpy(), want)
