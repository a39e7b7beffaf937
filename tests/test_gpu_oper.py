"""Layers of a bound sequence on operand tensors: every packed tensor of a pass equals, bit for bit, what the same layers write one call at a time
(whose kernels read packed codes), and the oracle where that is quick.  Geometries at the edges of the position numbering: one channel
group and odd numbers of them, readers of both strides of one tensor, windows without padding and of 5 and 7, concatenations, tensors that
a pass only reads in part from its own layers, rows and images of one pixel.  All of them with few images, whose plans are the simplest, and with many."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from oracle import network as onet
from paper_2207_08820_b200 import api, workloads as wl
from paper_2207_08820_b200.net import BitserialFullNet, BitserialNet
from paper_2207_08820_b200.workloads import ConvSpec, NetSpec
from gpu_util import dev

pytestmark = pytest.mark.gpu

L = ConvSpec


def net(batch, in_shape, layers, a_bits=2, w_bits=2):
    return NetSpec(name="t", batch=batch, in_name="x", in_shape=in_shape, layers=layers, a_bits=a_bits, w_bits=w_bits, out_name=layers[-1].dst)


STACKS = {
    "one_group": net(3, (32, 9, 12), [L("a", "x", "a", 32, 32, 3, 1, 1), L("b", "a", "b", 32, 96, 3, 2, 1), L("c", "b", "c", 96, 64, 1, 1, 0)]),
    "odd_groups": net(2, (96, 13, 8), [L("a", "x", "a", 96, 160, 3, 1, 1), L("b", "a", "b", 160, 96, 1, 2, 0, relu=False), L("c", "b", "c", 96, 40, 3, 1, 1)]),
    # readers of stride 1 and 2, with and without padding, of one tensor
    "both_strides": net(5, (64, 15, 15), [L("a", "x", "a", 64, 64, 3, 1, 1), L("b", "a", "b", 64, 64, 3, 2, 1), L("c", "a", "c", 64, 64, 1, 2, 0),
                                          L("d", "a", "d", 64, 64, 5, 1, 2), L("e", "a", "e", 64, 64, 3, 1, 0), L("f", "b", "f", 64, 64, 3, 1, 1, res="c", res_scale=0.5),
                                          L("g", "d", "g", 64, 32, 7, 2, 3), L("h", "e", "h", 64, 32, 5, 2, 1)]),
    "concatenation": net(2, (64, 20, 20), [L("a", "x", "cat", 64, 64, 1, 1, 0, dst_c_offset=64), L("b", "x", "b", 64, 64, 3, 1, 1),
                                           L("c", "b", "cat", 64, 64, 3, 1, 1, res="x", res_scale=0.5), L("d", "cat", "d", 128, 256, 1, 1, 0)]),
    "one_bit": net(3, (64, 10, 12), [L("a", "x", "a", 64, 128, 3, 1, 1), L("b", "a", "b", 128, 64, 3, 2, 1), L("c", "b", "c", 64, 64, 1, 1, 0, res="b", res_scale=0.5)], 1, 1),
    "three_bit_filters": net(3, (96, 11, 12), [L("a", "x", "a", 96, 128, 3, 1, 1), L("b", "a", "b", 128, 64, 3, 2, 1), L("c", "b", "c", 64, 64, 1, 1, 0, res="b", res_scale=0.5)], 2, 3),
    "wide": net(1, (32, 3, 300), [L("a", "x", "a", 32, 64, 3, 1, 1), L("b", "a", "b", 64, 32, 3, 2, 1), L("c", "b", "c", 32, 32, 1, 1, 0)]),
    "deep": net(1, (512, 7, 7), [L("a", "x", "a", 512, 256, 3, 1, 1), L("b", "a", "b", 256, 512, 1, 1, 0), L("c", "b", "c", 512, 64, 3, 2, 1)]),
    # records that no prepared filters are taken for: the pass prepares them
    "odd_records": net(2, (32, 9, 11), [L("a", "x", "a", 32, 64, 3, 2, 1), L("b", "a", "b", 64, 32, 1, 1, 0), L("c", "b", "c", 32, 32, 3, 1, 1, res="b", res_scale=0.5),
                                        L("d", "c", "d", 32, 128, 1, 1, 0), L("e", "d", "e", 128, 64, 3, 1, 1), L("f", "e", "f", 64, 64, 3, 1, 1), L("g", "f", "g", 64, 64, 1, 1, 0),
                                        L("h", "g", "h", 64, 64, 3, 1, 1), L("i", "h", "i", 64, 64, 3, 1, 1)]),
    "odd_one_bit": net(3, (64, 9, 13), [L("a", "x", "a", 64, 96, 3, 1, 1), L("b", "a", "b", 96, 64, 3, 2, 1)] + [L(f"l{i}", f"l{i - 1}" if i else "b", f"l{i}", 64 if i == 0 else 128, 128, 1, 1, 0) for i in range(7)], 1, 1),
    "pixels": net(40, (64, 1, 1), [L("a", "x", "a", 64, 64, 3, 1, 1), L("b", "a", "b", 64, 64, 1, 1, 0), L("c", "b", "c", 64, 32, 3, 2, 1)]),
}


# The same geometries with so many images that the plans are those of large batches: tiles of 64 and 128 filters, pairs of row tiles and four of them,
# several items a block, one to four accumulators, streamed filters, two teams (tests/test_host_sequence.py asserts that each is met).
MANY = {name: replace(STACKS[name], batch=batch) for name, batch in dict(one_group=3000, odd_groups=1500, three_bit_filters=1500, both_strides=1500, concatenation=900, one_bit=2000,
                                                                        wide=300, deep=400, odd_records=1500, odd_one_bit=1500, pixels=100000).items()}


def runner_of(spec, seed=11):
    params = wl.network_params(spec, seed)
    r = BitserialNet(spec, params, 0.25, batch=spec.batch, engine="tc")
    return r, params, wl.network_input(spec, seed, 0.25, batch=spec.batch)


def both(r, x):
    """Every packed tensor after a pass and after the same layers called one by one.  x: float input, or the packed one."""
    xd, out = dev(x) if isinstance(x, np.ndarray) else x, []
    for one_by_one in (False, True):
        for b in r.bufs.values():
            b.fill_(-1 if one_by_one else 0x5A5A5A5A)
        if xd.dtype == torch.int32:
            r.bufs[r.net.in_name].copy_(xd)
        else:
            r.pack_input(xd)
        r.run_units() if one_by_one else r.run_layers()
        api.bs_check_status()
        out.append({k: b.clone() for k, b in r.bufs.items()})
    return out


@pytest.mark.parametrize("name", STACKS)
def test_stacks(name):
    spec = STACKS[name]
    r, params, x = runner_of(spec)
    # the layers take operand tensors, of the input by a launch of its own
    assert r._sequence.launches == len(spec.layers) + 1 + any(item["w_tc"] is None for item in r.layers)
    assert (name in ("odd_records", "odd_one_bit")) == any(item["w_tc"] is None for item in r.layers)
    for seed in (0, 1):
        got, want = both(r, np.roll(x, seed, 0) if seed else x)
        for k in want:
            assert torch.equal(got[k], want[k]), k
    r.forward(dev(x))
    ref = onet.run_stack(spec, params, x, 0.25)
    for k in ref:
        assert np.array_equal(r.unpacked(k).cpu().numpy(), ref[k]), k


def packed_input(r, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randint(-2**31, 2**31, r.bufs[r.net.in_name].shape, generator=gen, device="cuda").to(torch.int32)      # (whole channel words)


@pytest.mark.parametrize("name", MANY)
def test_many_images(name):
    spec = MANY[name]
    r = BitserialNet(spec, wl.network_params(spec, 13), 0.25, batch=spec.batch, engine="tc")
    assert r._sequence.launches > len(spec.layers)
    for seed in (0, 1):
        got, want = both(r, packed_input(r, seed))
        for k in want:
            assert torch.equal(got[k], want[k]), k


@pytest.mark.parametrize("name", ["one_group", "odd_groups", "both_strides", "concatenation", "deep", "pixels"])
def test_many_images_by_the_slow_ways(name):
    """Filters of the other form, resident and streamed, and scales that only the formula takes, with every plan of large batches."""
    spec = MANY[name]
    r = BitserialNet(spec, wl.network_params(spec, 14), 0.25, batch=spec.batch, engine="tc")
    for step in (0, 1):
        for item in r.layers:
            if step == 0:
                item["w_tc"] = api.tc_prepare_weights(item["w"], item["spec"].C, item["w_sign"], 4)
            else:
                item["scale"] = item["scale"].clone()
                item["scale"][-1] = 1e-19
        got, want = both(r, packed_input(r, step))
        assert r._sequence.launches > len(spec.layers)
        for k in want:
            assert torch.equal(got[k], want[k]), k


@pytest.mark.parametrize("name", ["one_group", "both_strides", "one_bit"])
def test_packing_writes_the_operand_tensor(name):
    """A pass from floats writes the operand tensor of the input with its codes, without the launch of its own; layers alone follow codes that
    were written since, and inputs of another shape or type go the general way."""
    spec = STACKS[name]
    r, _, x = runner_of(spec)
    xd = dev(x)
    assert r.launches_per_forward == 1 + len(spec.layers)
    before = api.launch_count
    got = r.forward(xd).clone()
    assert api.launch_count - before == r.launches_per_forward
    codes = r.bufs["x"].clone()
    assert torch.equal(codes.view(-1), api.bitpack_activations(xd, 0.25, spec.a_bits).view(-1))
    r.bufs["x"].copy_(codes.roll(1, 0))                              # codes that no float input of a pass had
    r.run_layers()
    want = r.bufs[spec.out_name].clone()
    r.run_units()
    assert torch.equal(r.bufs[spec.out_name], want) and (spec.batch == 1 or torch.equal(want, got.roll(1, 0)))
    assert torch.equal(r.forward(xd), got)
    with pytest.raises(ValueError):
        r.forward(xd.transpose(2, 3))
    with pytest.raises(ValueError):
        r.forward(xd.cpu())
    api.bs_check_status()


def test_replaced_filters_scales_and_tensors():
    """Filters prepared for other widths, scales only the formula takes, tensors that move, a graph recorded before."""
    spec = STACKS["both_strides"]
    r, _, x = runner_of(spec)
    xd = dev(x)
    graph = torch.cuda.CUDAGraph()
    r.forward(xd)
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        r.run_layers()
    want = {k: b.clone() for k, b in r.bufs.items()}
    kept = [dict(item) for item in r.layers], dict(r.bufs)
    for i, item in enumerate(r.layers):
        if i % 2 == 0:
            item["w_tc"] = api.tc_prepare_weights(item["w"], item["spec"].C, item["w_sign"], 4)
        if i % 3 == 0:
            item["scale"] = item["scale"].clone()
            item["scale"][0] = 1e-19
    for k in r.bufs:
        r.bufs[k] = torch.empty_like(r.bufs[k])
    got, one_by_one = both(r, x)
    for k in got:
        assert torch.equal(got[k], one_by_one[k]), k
    for k, b in kept[1].items():
        if k != "x":
            b.fill_(-1)
    graph.replay()
    torch.cuda.synchronize()
    for k, b in kept[1].items():
        assert torch.equal(b, want[k]), k
    api.bs_check_status()


def test_filters_prepared_in_the_pass_follow_the_packed_ones():
    spec = STACKS["odd_records"]
    (a, _, x), (b, _, _) = runner_of(spec), runner_of(spec, seed=12)
    xd = dev(x)
    want = b.forward(xd).clone()
    assert not torch.equal(a.forward(xd), want)
    for mine, theirs in zip(a.layers, b.layers):
        for key in ("w", "w_tc", "scale", "bias"):
            if theirs[key] is not None:
                mine[key].copy_(theirs[key])                         # in place: nothing is bound again
    assert torch.equal(a.forward(xd), want)
    api.bs_check_status()


def test_sequences_that_keep_packed_tensors():
    """Overlapping tensors, and stacks in which most layers have no prepared filters, run as they did."""
    spec = STACKS["one_group"]
    r, _, x = runner_of(spec)
    for item in r.layers[:2]:
        item["w_tc"] = None
    got, want = both(r, x)
    assert r.launches_per_forward == 1 + len(spec.layers)
    for k in want:
        assert torch.equal(got[k], want[k]), k
    r, _, x = runner_of(spec)
    whole = torch.zeros(r.bufs["a"].numel() + r.bufs["c"].numel(), dtype=torch.int32, device="cuda")
    n = r.bufs["c"].numel()
    r.bufs["a"] = whole[: r.bufs["a"].numel()].view_as(r.bufs["a"])
    r.bufs["c"] = whole[4: 4 + n].view_as(r.bufs["c"])              # "a" is dead once "b" has been written
    xd = dev(x)
    r.forward(xd)
    assert r.launches_per_forward == 1 + len(spec.layers)
    have = r.bufs["c"].clone()
    r.pack_input(xd)
    r.run_units()
    assert torch.equal(have, r.bufs["c"])
    api.bs_check_status()


def test_filters_taken_away_from_a_bound_runner():
    """A layer that loses its prepared filters changes what the workspace holds, not whether the stack runs on operand tensors."""
    spec = STACKS["one_group"]
    r, _, x = runner_of(spec)
    n = len(spec.layers)
    assert r._sequence.launches == n + 1
    for i in range(n):
        kept, r.layers[i]["w_tc"] = r.layers[i]["w_tc"], None
        got, want = both(r, x)
        assert r._sequence.launches == n + 2, i                      # the input's import, and one launch that prepares the filters
        for k in want:
            assert torch.equal(got[k], want[k]), k
        r.layers[i]["w_tc"] = kept
    api.bs_check_status()


def test_recorded_passes_keep_their_workspace():
    """A graph that reads tensors of its own shares no memory with passes over others: the two may run side by side.  Without a graph the workspace
    passes on, and the number of those that graphs hold is bounded."""
    spec = STACKS["both_strides"]
    r, _, x = runner_of(spec)
    xd = dev(x)
    r.forward(xd)
    first = r._sequence.workspace

    def move():
        for k in r.bufs:
            r.bufs[k] = torch.empty_like(r.bufs[k])
        torch.cuda.synchronize()

    old = dict(r.bufs)
    move()
    want = r.forward(xd).clone()
    assert r._sequence.workspace is first and len(r._workspaces) == 1
    graphs, tensors = [], []
    for i in range(r.MAX_WORKSPACES + 1):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            r.run_layers()
        graphs.append(graph)
        tensors.append(dict(r.bufs))
        move()
        r.pack_input(xd)
        r.run_layers()
        live, recorded = r._sequence.workspace, [w for w in r._workspaces if w.recorded]
        assert (live is None) == (i + 1 >= r.MAX_WORKSPACES) and len(recorded) == min(i + 1, r.MAX_WORKSPACES) and live not in recorded
        assert torch.equal(r.bufs[spec.out_name], want)
    for graph, bufs in zip(graphs, tensors):
        bufs[spec.out_name].fill_(-1)
        graph.replay()
        assert torch.equal(bufs[spec.out_name], want)
    api.bs_check_status()


@pytest.mark.parametrize("whole", [False, True])
def test_a_pass_looks_at_its_tensors_once(whole, monkeypatch):
    """Whether an entry was replaced costs host time, which passes of few images are made of."""
    if whole:
        spec = wl.resnet18_full(2, 64)
        params = wl.full_network_params(spec, 5)
        r, x = BitserialFullNet(spec, params, batch=2), torch.randn(2, 3, 64, 64, device="cuda")
        body = r.body
    else:
        r, _, x = runner_of(STACKS["both_strides"])
        x, body = dev(x), r
    r.forward(x)
    looks = []
    monkeypatch.setattr(type(body._sequence), "current", lambda self, *a, current=type(body._sequence).current: looks.append(1) or current(self, *a))
    want = r.forward(x).clone()
    assert len(looks) == 1
    for k in body.bufs:
        body.bufs[k] = torch.empty_like(body.bufs[k])
    assert torch.equal(r.forward(x), want) and len(looks) == 2
    api.bs_check_status()


def test_operand_tensors_can_be_declined():
    spec = STACKS["both_strides"]
    r, params, x = runner_of(spec)
    plain, xd = BitserialNet(spec, params, 0.25, batch=spec.batch, engine="tc", operand_tensors=False), dev(x)
    assert r.operand_bytes == r._sequence.workspace.memory.numel() > 0 and plain.operand_bytes == 0
    assert plain._sequence.launches == len(spec.layers) and plain.input_operands() is None
    assert torch.equal(r.forward(xd), plain.forward(xd))
    api.bs_check_status()


def test_an_address_that_comes_back_is_not_a_packed_input():
    """Sequences of a runner follow each other, and the next may lie where the last one lay: what was written for one is not taken for the other's."""
    spec = STACKS["both_strides"]
    r, _, x = runner_of(spec)
    xd = dev(x)
    r.forward(xd)
    r.bufs["x"].copy_(r.bufs["x"].roll(1, 0))
    r.run_layers(ready=int(str(r.input_operands())))
    got = r.bufs[spec.out_name].clone()
    r.run_units()
    assert torch.equal(got, r.bufs[spec.out_name])
    ready = r.pack_input(xd, operands=True)
    r.layers[0]["w_tc"] = None                                       # binds again, to another workspace
    r.run_layers(ready=ready)
    got = r.bufs[spec.out_name].clone()
    r.run_units()
    assert torch.equal(got, r.bufs[spec.out_name])
    api.bs_check_status()
