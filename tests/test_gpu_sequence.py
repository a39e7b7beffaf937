"""bs_sequence and the compiled binding: a bound run of layers with one of them beside its successor equals the layers called one by one
(themselves checked against the oracle elsewhere), refusals come back as statuses, and wrong tensors as ValueError."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2207_08820_b200 import api, workloads as wl
from paper_2207_08820_b200._lib import SequenceLayer, lib
from gpu_util import dev, words

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prepared", [True, False])
@pytest.mark.parametrize("aside", [0, 1])
@pytest.mark.parametrize("N,C,H", [(1, 64, 9), (3, 96, 14)])
def test_sequence(N, C, H, aside, prepared):
    rng = np.random.default_rng(C + H)
    x, act = wl.rand_codes(rng, (N, C, H, H), 2, 0), []
    ws = [wl.rand_codes(rng, (C, C, 3, 3), 2, 1) for _ in range(3)]
    s, b = np.full(C, 2.0 ** -6, np.float32), rng.normal(1, 0.3, C).astype(np.float32)
    conv = lambda a, w, r=None: oracle.requantize(oracle.conv2d_i32(a, w, 1, 1), s, b, True, 2, 0)
    want0, want1 = conv(x, ws[0]), conv(x, ws[1])
    want2 = conv(want0, ws[2])
    t = [api.bitpack_activations(dev(x), 1.0, 2)] + [torch.zeros(N, H, H, C // 32, 2, dtype=torch.int32, device="cuda") for _ in range(3)]
    wp = [api.pack_weights(dev(w), 2, 1) for w in ws]
    wt = [api.tc_prepare_weights(w, C, 1, 2) for w in wp]
    sc, bi, side = dev(s), dev(b), torch.cuda.Stream()
    torch.cuda.synchronize()
    # x -> t1, x -> t2 (possibly beside the next), t1 -> t3 (waits for it)
    plan = [(t[0], t[1], 0, 0, []), (t[0], t[2], 1, aside, []), (t[1], t[3], 2, 0, [1] if aside else [])]
    arr = (SequenceLayer * 3)()
    for q, (src, dst, k, a, join) in zip(arr, plan):
        q.act_packed, q.out_packed, q.wgt_packed = src.data_ptr(), dst.data_ptr(), wp[k].data_ptr()
        q.wgt_tc = wt[k].data_ptr() if prepared else None
        q.p = api.conv_params(src.shape, wp[k].shape, C=C, pad=1, scale=sc, bias=bi, relu=True, out_bits=2)
        q.chained, q.aside = int(prepared), a
        q.join[:] = (join + [-1] * 4)[:4]
    h = ctypes.c_void_p()
    assert lib().bs_sequence_create(arr, 3, side.cuda_stream, ctypes.byref(h)) == 0
    for _ in range(3):
        for d in t[1:]:
            d.fill_(-1)
        api.run_sequence(h.value, 3)
        api.bs_check_status()
        for d, w in zip(t[1:], (want0, want1, want2)):
            assert np.array_equal(words(d), oracle.pack_activations(w, 2, 0))
    lib().bs_sequence_destroy(h)
    # refusals: no layers, a join that does not precede its layer, a layer beside the others without a stream for it
    assert lib().bs_sequence_create(arr, 0, None, ctypes.byref(h)) != 0
    arr[0].join[0] = 0
    assert lib().bs_sequence_create(arr, 3, side.cuda_stream, ctypes.byref(h)) != 0
    arr[0].join[0] = -1
    arr[1].aside = 1
    assert lib().bs_sequence_create(arr, 3, None, ctypes.byref(h)) != 0


def test_binding_refuses_wrong_tensors():
    x = torch.zeros(1, 4, 4, 2, 2, dtype=torch.int32, device="cuda")
    w = torch.zeros(32, 3, 3, 2, 2, dtype=torch.int32, device="cuda")
    for bad in (dict(act_packed=x.cpu(), wgt_packed=w, C=64), dict(act_packed=x, wgt_packed=w.transpose(1, 2), C=64), dict(act_packed=x, wgt_packed=w, C=65)):
        with pytest.raises(ValueError):
            api.bitserial_conv2d(**bad, pad=1, want_i32=True)
    with pytest.raises(ValueError):
        api.bitpack_activations(torch.zeros(1, 32, 2, 2, dtype=torch.float16, device="cuda"), 1.0, 2)
    with pytest.raises(api.BitserialError):
        api.bitserial_conv2d(x, w, C=64, pad=1)          # no output asked for
