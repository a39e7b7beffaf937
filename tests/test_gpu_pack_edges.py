"""Packing at the edges of its kernels: rows that start off a word, records that are not whole channel words, the end of the tensor,
and the estimate-and-check quantiser of 3 and 4 bits on every rounding tie."""
import numpy as np
import pytest

import oracle
from paper_2207_08820_b200 import api, workloads as wl
from gpu_util import dev, words

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,sign", [(1, 0), (1, 2), (2, 1), (3, 0), (4, 1)])
@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (1, 33, 1, 3), (2, 31, 3, 43), (3, 65, 5, 51), (1, 100, 1, 129), (2, 50, 9, 29), (1, 3000, 2, 3)])
def test_codes_of_any_alignment(bits, sign, shape):
    codes = wl.rand_codes(np.random.default_rng(bits + shape[1]), shape, bits, sign)
    want = oracle.pack_activations(codes, bits, sign)
    assert np.array_equal(words(api.bitpack_activations(dev(codes), 1.0, bits, sign, api.NCHW)), want)
    assert np.array_equal(words(api.bitpack_activations(dev(codes.transpose(0, 2, 3, 1)), 1.0, bits, sign, api.NHWC)), want)


@pytest.mark.parametrize("bits,sign", [(3, 0), (3, 1), (4, 0), (4, 1)])
@pytest.mark.parametrize("s", [0.37, 1.0, 2.9e-30, 3.1e29, 1e-31, 2e30])
def test_levels_on_every_tie(bits, sign, s):
    lo, hi = wl.code_range(bits, sign)
    ties = ((np.arange(lo - 1, hi + 2) + 0.5) * np.float64(np.float32(s))).astype(np.float32)
    vals = [ties, np.arange(lo - 1, hi + 2, dtype=np.float32) * np.float32(s)]
    for d in (np.inf, -np.inf):
        v = ties
        for _ in range(3):
            v = np.nextafter(v, np.float32(d))
            vals.append(v)
    vals.append(np.array([np.nan, np.inf, -np.inf, 0.0, -0.0, 1e-45, -1e-45, 3e38, -3e38], dtype=np.float32))
    x = np.random.default_rng(bits).choice(np.concatenate(vals), size=(1, 45, 5, 33)).astype(np.float32)
    with np.errstate(all="ignore"):
        want = oracle.pack_activations(oracle.quantize(x, s, bits, sign), bits, sign)
    assert np.array_equal(words(api.bitpack_activations(dev(x), s, bits, sign, api.NCHW)), want)
    assert np.array_equal(words(api.bitpack_activations(dev(x.transpose(0, 2, 3, 1)), s, bits, sign, api.NHWC)), want)
