"""Host side of bound sequences, without a device: which stacks run on operand tensors, and by which plans."""
import ctypes

import pytest

from paper_2207_08820_b200 import api, workloads as wl
from paper_2207_08820_b200._lib import ConvParams, LayerPlan, lib
from gpu_util import layer_array
from test_gpu_oper import MANY, STACKS


def workspace(spec, **kw):
    arr = layer_array(spec, **kw)
    return lib().bs_sequence_workspace_bytes(arr, len(arr))


@pytest.mark.parametrize("w_bits,w_sign,takes", [(2, wl.SIGNED, True), (2, wl.UNSIGNED, True), (1, wl.BIPOLAR, True), (3, wl.SIGNED, False), (3, wl.UNSIGNED, False), (4, wl.SIGNED, False)])
def test_filters_that_are_prepared_as_nibbles(w_bits, w_sign, takes):
    """Stacks whose prepared filters are int8, three bits and up, stay on packed codes: on operand tensors every launch would convert them."""
    spec = wl.resnet18_body(2, 28)
    spec.w_bits = w_bits
    assert (workspace(spec, w_sign=w_sign) > 0) == takes


@pytest.mark.parametrize("a_bits,w_bits,takes", [(2, 3, True), (1, 3, True), (3, 3, False), (2, 2, False), (2, 4, False)])
def test_three_bit_filters_prepared_as_nibbles(a_bits, w_bits, takes):
    spec = wl.resnet18_body(2, 28)
    spec.a_bits, spec.w_bits = a_bits, w_bits
    assert (workspace(spec, w_sign=wl.SIGNED, prepared_sign=api.SIGNED_NIBBLES) > 0) == takes


def test_the_sign_of_nibbles_is_for_prepared_filters_only():
    p = ConvParams(N=1, C=64, H=8, W=8, O=64, R=3, S=3, stride=1, pad=1, a_bits=2, w_bits=3, w_sign=api.SIGNED_NIBBLES)
    assert lib().bs_tc_supported(ctypes.byref(p)) == 1
    assert lib().bitserial_conv2d(4096, 4096, ctypes.byref(p), 4096, None, None) == 1
    assert lib().bs_conv_workspace_bytes(ctypes.byref(p)) == 0
    assert lib().pack_weights(4096, 0, 64, 64, 3, 3, 3, api.SIGNED_NIBBLES, 4096, None) == 1
    assert lib().bs_tc_prepare_weights(4096, 64, 64, 3, 3, 3, api.SIGNED_NIBBLES, 3, 4096, None) == 2
    assert lib().bs_tc_prepare_weights(4096, 64, 64, 3, 3, 2, api.SIGNED_NIBBLES, 2, 4096, None) == 2
    arr = layer_array(STACKS["one_group"])
    arr[0].wgt_tc, arr[0].p.w_sign, arr[0].p.w_bits = None, api.SIGNED_NIBBLES, 3
    assert lib().bs_sequence_layer_plan(arr, len(arr), 0, ctypes.byref(LayerPlan())) == 1
    for field, value in (("a_bits", 3), ("a_bits", 4), ("w_bits", 2), ("a_sign", api.SIGNED_NIBBLES)):
        q = ConvParams.from_buffer_copy(p)
        setattr(q, field, value)
        assert lib().bs_tc_supported(ctypes.byref(q)) == 0


def plans(spec):
    """(layer, its plan) of every layer of a stack."""
    arr = layer_array(spec, prepared_sign=api.SIGNED_NIBBLES if spec.w_bits == 3 else None)
    for i, layer in enumerate(spec.layers):
        plan = LayerPlan()
        assert lib().bs_sequence_layer_plan(arr, len(arr), i, ctypes.byref(plan)) == 0
        yield layer, plan


def test_plan_query_refuses():
    plan, spec = LayerPlan(), STACKS["one_group"]
    arr = layer_array(spec)
    for layers, n, i, out in ((arr, len(arr), -1, plan), (arr, len(arr), len(arr), plan), (arr, 0, 0, plan), (None, 1, 0, plan), (arr, len(arr), 0, None)):
        assert lib().bs_sequence_layer_plan(layers, n, i, ctypes.byref(out) if out else None) == 1
    spec = wl.resnet18_body(2, 28)
    spec.w_bits = 3
    arr = layer_array(spec)
    assert lib().bs_sequence_layer_plan(arr, len(arr), 0, ctypes.byref(plan)) == 2


def pairs(plan):
    """Two row tiles share the scales (oper_kernel.cuh)."""
    return plan.row_tiles > 1 and plan.row_tiles * plan.filters // 32 >= 4


FORMS = {
    "64 filters": lambda l, p: p.filters == 64,
    "128 filters": lambda l, p: p.filters == 128,
    "filters that end inside a tile": lambda l, p: p.filters > 32 and l.O % p.filters,
    "two row tiles one by one": lambda l, p: p.row_tiles == 2 and not pairs(p),
    "pairs of row tiles": lambda l, p: pairs(p),
    "pairs with a residual": lambda l, p: pairs(p) and l.res,
    "four row tiles": lambda l, p: p.row_tiles == 4,
    "several items on one accumulator": lambda l, p: p.items > 1 and p.accumulators == 1,
    "more items than accumulators": lambda l, p: p.items > p.accumulators > 1,
    "more items than stages": lambda l, p: p.items > p.stages > 1,
    "streamed filters, several items": lambda l, p: not p.resident and p.items > 1,
    "a stage with one step of two": lambda l, p: p.channels > 1 and (l.C + 63) // 64 % p.channels,
    "two teams": lambda l, p: p.teams == 2,
    "two teams, pairs with a residual": lambda l, p: p.teams == 2 and pairs(p) and l.res,
    "two teams, single row tiles": lambda l, p: p.teams == 2 and not pairs(p),
    "two teams, stride 2": lambda l, p: p.teams == 2 and l.stride == 2,
    "two teams, no padding": lambda l, p: p.teams == 2 and l.k > 1 and l.pad == 0,
    "windows of 5, several items": lambda l, p: l.k == 5 and p.items > p.accumulators,
    "windows of 7": lambda l, p: l.k == 7 and p.items > 1,
    "an odd number of channel groups, several items": lambda l, p: l.C // 32 % 2 and l.C > 32 and p.items > 1,
    "one channel group, more items than accumulators": lambda l, p: l.C == 32 and p.items > p.accumulators,
}


@pytest.mark.parametrize("form", FORMS)
def test_stacks_meet_every_form(form):
    """The stacks that are compared bit for bit on the device run every form of the kernel."""
    assert any(FORMS[form](l, p) for spec in MANY.values() for l, p in plans(spec))


def test_stacks_of_few_images_are_simple():
    assert all((p.filters, p.row_tiles, p.resident, p.items, p.teams) == (32, 1, 1, 1, 1) for spec in STACKS.values() for _, p in plans(spec))
