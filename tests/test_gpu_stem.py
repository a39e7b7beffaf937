"""The fused stem (``bs_stem_codes_f32``: convolution, ReLU, pooling, quantiser) against the oracle and against the separate layers: the codes
are equal, whatever the images, filters and scale, since outputs near a bound of the quantiser take the layers' own arithmetic."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2207_08820_b200 import api, workloads as wl
from paper_2207_08820_b200.net import BitserialFullNet
from gpu_util import Guarded, dev

pytestmark = pytest.mark.gpu


def inputs(N, H, W, seed=0, bias=0.1):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(N, 3, H, W, generator=g, device="cuda")
    w = torch.randn(64, 3, 7, 7, generator=g, device="cuda") / math.sqrt(147.0)
    return x, w, torch.randn(64, generator=g, device="cuda") * bias


def compare(x, w, b, scale=0.25):
    pool = api.maxpool2d_f32(api.conv2d_f32(x, w, b, 2, 3, True), 3, 2, 1)
    want = api.bitpack_activations(pool, scale, 2)
    guard = Guarded()
    out = guard.empty(tuple(want.shape), fill=-1)
    assert api.stem_codes_f32(x, w, b, scale, 2, out)
    api.bs_check_status()
    guard.check()
    assert torch.equal(out, want)


# one pixel pair, one pooled row, odd heights, widths whose rows end inside a tile or a slab, runs that cross images, wide rows (the widest: test_widest_rows)
@pytest.mark.parametrize("N,H,W", [(5, 1, 2), (2, 8, 8), (1, 7, 34), (2, 37, 46), (3, 64, 64), (149, 20, 24), (9, 75, 126), (2, 224, 224), (1, 90, 254), (2, 256, 256), (1, 50, 278)])
def test_sizes(N, H, W):
    compare(*inputs(N, H, W, seed=H))
    x, w, _ = inputs(N, H, W, seed=H + 1)
    compare(x, w, None)


def test_against_oracle():
    x, w, b = inputs(2, 58, 66, seed=5)
    pool = oracle.maxpool2d_f32(oracle.conv2d_f32(x.cpu().numpy(), w.cpu().numpy(), b.cpu().numpy(), 2, 3, True), 3, 2, 1)
    codes = oracle.quantize(pool, 0.25, 2, api.UNSIGNED)
    out = torch.empty(2, 15, 17, 2, 2, dtype=torch.int32, device="cuda")
    assert api.stem_codes_f32(x, w, b, 0.25, 2, out)
    assert np.array_equal(api.bitunpack_activations(out, 64, 2).cpu().numpy(), codes)


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf"), 3e38, 1e30, 2.0 ** 20, 1e6, 1e-30, 1e-42])
def test_single_values(value):
    x, w, b = inputs(2, 64, 64, seed=9)
    x[1, 2, 31, 17] = value
    compare(x, w, b)


@pytest.mark.parametrize("case", ["zero", "constant", "on the bounds", "small images", "large images", "zero filters", "one large filter", "large bias",
                                  "bad filters", "cancelling", "denormal"])
def test_values(case):
    x, w, b = inputs(2, 66, 70, seed=11)
    if case == "zero":
        x.zero_()
    elif case == "constant":
        x.fill_(0.37)
    elif case == "on the bounds":        # half of the outputs are the bias, which is a bound or its neighbour: all undecided
        x[:, :, :40] = 0.0
        b.copy_(torch.tensor([0.125, 0.375, 0.625, 0.12500001], device="cuda").repeat(16))
    elif case == "small images":
        x *= 1e-25
        w *= 1e25
    elif case == "large images":
        x *= 255.0
    elif case == "zero filters":
        w.zero_()
    elif case == "one large filter":
        w[7] *= 1e6
    elif case == "large bias":
        b *= 1e4
    elif case == "bad filters":
        w[3, 1, 2, 2], w[40, 0, 0, 0], b[7], b[9] = float("inf"), float("nan"), float("inf"), float("nan")
    elif case == "cancelling":           # the order of the chain decides
        w.fill_(1.0)
        x[:, 0], x[:, 2] = 3e5, -3e5
    else:
        x *= 1e-42
    compare(x, w, b)


@pytest.mark.parametrize("scale", [1e-20, 0.01, 0.25, 0.6, 1.5, 37.0, 1e20])
def test_scales(scale):
    compare(*inputs(2, 64, 64, seed=13), scale=scale)


@pytest.mark.parametrize("C,O,k,W,bits", [(4, 64, 7, 64, 2), (3, 32, 7, 64, 2), (3, 64, 5, 64, 2), (3, 64, 7, 63, 2), (3, 64, 7, 64, 3), (3, 64, 7, 400, 2)])
def test_other_shapes_are_refused(C, O, k, W, bits):
    x, w = torch.zeros(1, C, 64, W, device="cuda"), torch.zeros(O, C, k, k, device="cuda")
    q = (W - 1) // 2 + 1
    out = torch.full((1, 16, (q - 1) // 2 + 1, (O + 31) // 32, bits), -1, dtype=torch.int32, device="cuda")
    assert not api.stem_codes_f32(x, w, None, 0.25, bits, out)
    assert bool((out == -1).all())


@pytest.mark.parametrize("hw", [32, 64, 284])
def test_classifier_front(hw):
    """Both ways of the classifier's front, the float tensors of the stem, and filters replaced between passes."""
    net = wl.resnet18_full(batch=2, hw=hw)
    params = wl.full_network_params(net, 8300)
    images = dev(wl.full_network_input(net, 8300))
    runner = BitserialFullNet(net, params, batch=2)
    logits = runner.forward(images).clone()
    packed = runner.body.bufs[net.body.in_name].clone()
    conv, pool = runner.stem_conv.clone(), runner.stem_pool.clone()
    runner.run_stem(images)
    assert torch.equal(conv, runner.stem_conv) and torch.equal(pool, runner.stem_pool)
    runner.body.pack_input(runner.stem_pool)
    assert torch.equal(packed, runner.body.bufs[net.body.in_name])
    runner.stem_w.mul_(-1.0)
    assert not torch.equal(runner.forward(images), logits)
    runner.stem_w = -runner.stem_w
    assert torch.equal(runner.forward(images), logits)
    api.bs_check_status()


def classifier(hw=64, seed=8300):
    net = wl.resnet18_full(batch=2, hw=hw)
    images = [dev(wl.full_network_input(net, seed + k)) for k in range(3)]
    return BitserialFullNet(net, wl.full_network_params(net, seed), batch=2), images


def stem_layers(runner, images):
    conv = api.conv2d_f32(images, runner.stem_w, runner.stem_b, 2, 3, True)
    return conv, api.maxpool2d_f32(conv, 3, 2, 1)


def record(runner, static):
    runner.forward(static)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        runner.forward(static)
    return graph


def test_stem_tensors_follow_replays():
    """Python does not run on a replay: a read between two replays must not leave the first one's tensors behind."""
    runner, (a, b, c) = classifier()
    static = a.clone()
    graph = record(runner, static)

    def check(images):
        conv, pool = stem_layers(runner, images)
        assert torch.equal(runner.stem_conv, conv) and torch.equal(runner.stem_pool, pool)

    for images in (a, b, b, c):
        static.copy_(images)
        graph.replay()
        check(images)
        check(images)
    runner.forward(a)                       # launched after replays, and replayed after a launch
    check(a)
    graph.replay()
    check(c)
    runner.run_stem(b)
    check(b)
    static.copy_(a)
    graph.replay()
    check(a)
    kept = runner.stem_pool                 # recorded while held: the graph writes the tensors
    second = record(runner, static)
    static.copy_(b)
    second.replay()
    assert torch.equal(kept, stem_layers(runner, b)[1])
    check(b)
    static.copy_(c)
    graph.replay()
    check(c)


def test_stem_tensors_that_are_kept_or_assigned():
    runner, (a, b, c) = classifier()
    logits = runner.forward(a).clone()
    kept = runner.stem_pool
    assert runner.stem_pool is kept
    runner.forward(b)
    assert torch.equal(kept, stem_layers(runner, b)[1])
    b.zero_()                               # the pass wrote its tensors: its images may go
    assert torch.equal(kept, runner.stem_pool)
    assert torch.equal(runner.forward(a), logits)
    del kept
    runner.forward(c)
    d = c.clone()
    c.zero_()
    with pytest.raises(RuntimeError):       # codes only, and their images are gone
        runner.stem_conv
    runner.forward(d)
    mine = torch.zeros_like(runner.stem_pool)
    runner.stem_pool = mine
    assert bool((mine == 0).all())
    runner.forward(a)
    assert torch.equal(mine, stem_layers(runner, a)[1]) and torch.equal(runner.stem_pool, mine)
    assert torch.equal(runner.logits, logits)


@pytest.mark.parametrize("hw", [64, 308])
def test_launches_and_layers_of_the_front(hw):
    """``launches_per_forward`` counts what a pass launches, where the stem is one kernel, where its shape is refused and while its tensors are held."""
    runner, (a, b, _) = classifier(hw)
    fused = hw == 64

    def launches(images):
        before = api.launch_count
        runner.forward(images)
        return api.launch_count - before

    for images in (a, b):
        assert launches(images) == runner.launches_per_forward == runner.body.launches_per_forward + (2 if fused else 4)
        conv, pool = stem_layers(runner, images)
        assert torch.equal(runner.body.bufs[runner.net.body.in_name].view(-1), api.bitpack_activations(pool, runner.body.act_scale, 2).view(-1))
        assert torch.equal(runner.stem_conv, conv) and torch.equal(runner.stem_pool, pool)
    kept = runner.stem_pool
    assert launches(a) == runner.launches_per_forward == runner.body.launches_per_forward + 4
    assert torch.equal(kept, stem_layers(runner, a)[1])


def test_widest_rows():
    """Shared memory and the cells of a thread nearly full; the next even width is refused."""
    compare(*inputs(2, 37, 306, seed=3))
    x, w, _ = inputs(1, 16, 308)
    assert not api.stem_codes_supported(x.shape, w.shape, 0.25, 2)
    assert not api.stem_codes_f32(x, w, None, 0.25, 2, torch.empty(1, 4, 77, 2, 2, dtype=torch.int32, device="cuda"))


def test_stem_tensors_take_memory_from_their_first_use_on():
    runner, (a, _, _) = classifier()
    runner.forward(a)
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    pool = runner.stem_pool
    assert torch.cuda.memory_allocated() - before >= 4 * 2 * 64 * (32 * 32 + 16 * 16)
    assert torch.equal(pool, stem_layers(runner, a)[1])


def test_images_inside_a_larger_buffer():
    x, w, b = inputs(5, 60, 64, seed=21)
    compare(x[1:4], w, b)
    flat = torch.cat([x.reshape(-1), x.reshape(-1)])
    n = 2 * 3 * 60 * 64
    compare(flat[4:4 + n].view(2, 3, 60, 64), w, b)
    with pytest.raises(api.BitserialError):         # off a 16-byte boundary, as for the layers
        api.stem_codes_f32(flat[1:1 + n].view(2, 3, 60, 64), w, b, 0.25, 2, torch.empty(2, 15, 16, 2, 2, dtype=torch.int32, device="cuda"))
    with pytest.raises(api.BitserialError):
        api.conv2d_f32(flat[1:1 + n].view(2, 3, 60, 64), w, b, 2, 3, True)
