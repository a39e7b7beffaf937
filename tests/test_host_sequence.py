"""Host side of bound sequences, without a device: which stacks run on operand tensors."""
import pytest

from paper_2207_08820_b200 import workloads as wl
from paper_2207_08820_b200._lib import lib
from gpu_util import layer_array


def workspace(spec, **kw):
    arr = layer_array(spec, **kw)
    return lib().bs_sequence_workspace_bytes(arr, len(arr))


@pytest.mark.parametrize("w_bits,w_sign,takes", [(2, wl.SIGNED, True), (2, wl.UNSIGNED, True), (1, wl.BIPOLAR, True), (3, wl.SIGNED, False), (3, wl.UNSIGNED, False), (4, wl.SIGNED, False)])
def test_filters_that_are_prepared_as_nibbles(w_bits, w_sign, takes):
    """Stacks whose prepared filters are int8, three bits and up, stay on packed codes: on operand tensors every launch would convert them."""
    spec = wl.resnet18_body(2, 28)
    spec.w_bits = w_bits
    assert (workspace(spec, w_sign=w_sign) > 0) == takes
