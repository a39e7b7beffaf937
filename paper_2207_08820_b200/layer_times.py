"""Per-layer times of a layer stack on one GPU.

    python -m paper_2207_08820_b200.layer_times resnet18_body [batch] [engine]

Every layer is timed in four ways, each inside a CUDA graph with CUDA events (warm L2, best of four replays).  As a call on packed codes: launched
once; eight times back to back; eight times back to back as launches chained by programmatic dependent launch (tensor-core engine only).  And as
:class:`net.BitserialNet` runs it, in a bound sequence on operand tensors, where the library takes it there.  The last columns are the layer's
arithmetic over the last of these times, and how the bound layer was planned.  Host logic only.
"""
from __future__ import annotations

import ctypes
import sys

import torch

from . import api, workloads as wl
from ._lib import LayerPlan, SequenceLayer, lib
from .net import BitserialNet

STACKS = {"resnet18_body": (wl.resnet18_body, 64, 3000), "detection_backbone": (wl.detection_backbone, 16, 4000),
          "resnet50_body": (wl.resnet50_body, 32, 6000), "vgg16_ssd_body": (wl.vgg16_ssd_body, 8, 7000)}
REPS = 8


class BoundLayer:
    """A sequence of one layer of a bound runner ``reps`` times over, on operand tensors: behind a small layer that reads its output, so that it writes the
    operand tensor as well.  ``handle`` is None where the library does not take it so.  Owns what the sequence reads and writes."""

    def __init__(self, runner: BitserialNet, item, reps: int):
        out, C = runner.bufs[item["spec"].dst], runner.shapes[item["spec"].dst][0]
        self.handle, self.plan, self.keep = None, LayerPlan(), [runner]
        if item["w_tc"] is None or C % 32:
            return
        codes = torch.zeros(32, C, 1, 1, dtype=torch.int8, device=out.device)
        w, rest = api.pack_weights(codes, runner.net.w_bits, item["w_sign"]), torch.zeros(*out.shape[:3], 1, runner.net.a_bits, dtype=torch.int32, device=out.device)
        scale = torch.ones(32, dtype=torch.float32, device=out.device)
        both = api.tc_prepare_weights(w, C, item["w_sign"], runner.net.a_bits)
        w_tc, sign = api.tc_weights_form(both, w.shape, C, item["w_sign"], runner.net.a_bits)
        self.keep += [w, both, rest, scale]
        self.layers = (SequenceLayer * (reps + 1))()
        for k, q in enumerate(self.layers):
            q.act_packed, q.out_packed = (runner.bufs[item["spec"].src].data_ptr(), out.data_ptr()) if k else (out.data_ptr(), rest.data_ptr())
            q.wgt_packed, q.wgt_tc = (item["w"].data_ptr(), runner._filters(item)[0].data_ptr()) if k else (w.data_ptr(), w_tc.data_ptr())
            q.p = runner._conv_params(item) if k else api.conv_params(out.shape, w.shape, C=C, w_sign=sign, scale=scale, bias=scale, out_bits=runner.net.a_bits)
            q.chained = 1
            q.join[:] = [-1] * 4
        nbytes = lib().bs_sequence_workspace_bytes(self.layers, reps + 1)
        if nbytes == 0:
            return
        workspace = torch.zeros(nbytes, dtype=torch.uint8, device=out.device)
        self.keep.append(workspace)
        handle = ctypes.c_void_p()
        torch.cuda.synchronize(out.device)
        if lib().bs_sequence_create_ws(self.layers, reps + 1, None, workspace.data_ptr(), nbytes, ctypes.byref(handle)) == 0:
            self.handle = handle.value
            lib().bs_sequence_layer_plan(self.layers, reps + 1, reps, ctypes.byref(self.plan))

    def run(self) -> None:
        api.run_sequence(self.handle, lib().bs_sequence_launches(self.handle))

    def __del__(self):
        if self.handle is not None:
            lib().bs_sequence_destroy(self.handle)


def graph_us(fn, stream) -> float:
    """Device time of ``fn`` as a graph."""
    fn()
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        fn()
    best = float("inf")
    for k in range(6):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        graph.replay()
        e1.record(stream)
        e1.synchronize()
        if k >= 2:
            best = min(best, e0.elapsed_time(e1) * 1e3)
    return best


def main(argv) -> int:
    name = argv[1] if len(argv) > 1 else "resnet18_body"
    make, batch, seed = STACKS[name]
    if len(argv) > 2:
        batch = int(argv[2])
    engine = argv[3] if len(argv) > 3 else "tc"
    net = make(batch)
    params = wl.network_params(net, seed)
    x = torch.from_numpy(wl.network_input(net, seed, 0.25, batch=batch)).cuda()
    runner = BitserialNet(net, params, 0.25, batch=batch, engine=engine, chains=False)
    runner.forward(x)
    api.bs_check_status()
    stream = torch.cuda.Stream()
    shapes = net.tensor_shapes()
    sums = [0.0, 0.0, 0.0]
    with torch.cuda.stream(stream):
        for item in runner.layers:
            L = item["spec"]
            _, P, Q = shapes[L.dst]
            macs = batch * P * Q * L.O * L.C * L.k * L.k

            def calls(reps, chained):
                for _ in range(reps):
                    runner.run_layer(item, chained=chained)

            t1, tr, tc = graph_us(lambda: calls(1, False), stream), graph_us(lambda: calls(REPS, False), stream) / REPS, graph_us(lambda: calls(REPS, True), stream) / REPS
            few, many = BoundLayer(runner, item, REPS), BoundLayer(runner, item, 2 * REPS)
            tb, plan = tc, "packed codes"
            if few.handle is not None:
                tb, p = (graph_us(many.run, stream) - graph_us(few.run, stream)) / REPS, few.plan
                plan = f"{p.filters}x{128 * p.row_tiles} {'resident' if p.resident else 'streamed'} {p.blocks} blocks of {p.items} items, {p.accumulators} accumulators, {p.teams} teams"
            for k, t in enumerate((t1, tc, tb)):
                sums[k] += t
            print(f"{L.name:14s} C{L.C:5d} O{L.O:5d} k{L.k} s{L.stride} {P:3d}x{Q:<3d} res={int(bool(L.res))}  single {t1:6.2f} us  x{REPS} {tr:6.2f}  "
                  f"chained {tc:6.2f}  bound {tb:6.2f} us  {2 * macs / tb / 1e6:7.1f} TOP/s  {plan}")
    print(f"sum of single calls {sums[0]:.1f} us, of chained calls {sums[1]:.1f} us, of bound layers {sums[2]:.1f} us")
    api.bs_check_status()
    return 0


if __name__ == "__main__":
    sys.exit(main(sys.argv))
