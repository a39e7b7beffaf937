"""Host side of bound sequences, without a device: which stacks run on operand tensors, and by which plans."""
import ctypes

import pytest

from paper_2207_08820_b200 import workloads as wl
from paper_2207_08820_b200._lib import LayerPlan, lib
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


def plans(spec):
    """(layer, its plan) of every layer of a stack."""
    arr = layer_array(spec)
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
