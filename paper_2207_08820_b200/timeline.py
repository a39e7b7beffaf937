"""Per-CTA timelines of the tensor-core kernels (trace builds only).

A library built with ``BS_EXTRA_NVCC_FLAGS=-DBS_TRACE python -m paper_2207_08820_b200.build --force`` records, for the first 148 CTAs
of a launch with 2-bit activations and filters of at most two bits and the first 48 steps of each, the SM cycle counter at the hand-offs between the kernel's roles
(expansion of a chunk, issue of its MMAs, epilogue of an item).  This tool runs chosen layers of a layer stack and prints
those timelines, of the layer in a bound sequence on operand tensors (as a runner's pass runs it) or, with "calls", of a call on packed codes:

    python -m paper_2207_08820_b200.timeline resnet18_body 0,7 [cta,cta,...] [batch] [calls]

Host logic only; the normal library has no such entry point and the tool says so.
"""
from __future__ import annotations

import ctypes
import sys

import numpy as np
import torch

from . import api, workloads as wl
from ._lib import lib
from .layer_times import BoundLayer
from .net import BitserialNet

EVENTS = ["START", "SETUP", "PDL", "WGT", "XBEG", "XEND", "MBEG", "MEND", "EBEG", "EEND", "END", "XWAIT"]
STACKS = {"resnet18_body": (wl.resnet18_body, 64, 3000), "detection_backbone": (wl.detection_backbone, 16, 4000),
          "resnet50_body": (wl.resnet50_body, 32, 6000), "vgg16_ssd_body": (wl.vgg16_ssd_body, 8, 7000)}


def main(argv) -> int:
    name = argv[1] if len(argv) > 1 else "resnet18_body"
    layers = [int(v) for v in argv[2].split(",")] if len(argv) > 2 else [0]
    ctas = [int(v) for v in argv[3].split(",")] if len(argv) > 3 else [0, 147]
    L = lib()
    if not hasattr(L, "bs_tc_trace_read"):
        print("this library was not built with -DBS_TRACE: no timeline is recorded")
        return 1
    make, batch, seed = STACKS[name]
    batch = int(argv[4]) if len(argv) > 4 else batch
    calls = "calls" in argv
    read = L.bs_tc_trace_read if calls else L.bs_oper_trace_read
    read.restype, read.argtypes = ctypes.c_int, [ctypes.c_void_p, ctypes.c_int]
    net = make(batch)
    params = wl.network_params(net, seed)
    x = torch.from_numpy(wl.network_input(net, seed, 0.25, batch=batch)).cuda()
    runner = BitserialNet(net, params, 0.25, batch=batch, engine="tc")
    runner.forward(x)
    api.bs_check_status()
    buf = np.zeros((148, len(EVENTS), 48), dtype=np.int64)
    for li in layers:
        item = runner.layers[li]
        if calls:
            run = lambda: runner.run_layer(item, chained=False)
        else:
            bound = BoundLayer(runner, item, 4)
            if bound.handle is None:
                print(f"layer {li}: not on operand tensors")
                continue
            run = bound.run
        for _ in range(3):
            run()
        read(buf.ctypes.data, 1)
        run()
        read(buf.ctypes.data, 1)
        spec = item["spec"]
        print(f"layer {li} {spec.name}: C {spec.C} O {spec.O} k {spec.k} stride {spec.stride}")
        if not calls:           # (what the table holds beyond it is of the small layer in front)
            p, chunks = bound.plan, -(-((spec.C + 63) // 64) // bound.plan.channels)
            buf[p.blocks:] = 0
            print(f"  {p.filters} filters x {p.row_tiles} row tiles, {p.blocks} blocks of up to {p.items} items of {chunks} chunks, {p.stages} stages, {p.accumulators} accumulators, "
                  f"{p.teams} teams, filters {'resident' if p.resident else 'streamed'}")
        for c in ctas:
            t0 = buf[c, 0, 0] if c < 148 else 0
            if t0 == 0:
                print(f"  CTA {c}: no timeline (fewer CTAs in this launch)")
                continue
            rel = lambda e, k=0: buf[c, EVENTS.index(e), k] - t0
            print(f"  CTA {c}: ends at {rel('END')} cycles; set-up {rel('SETUP')}, filters landed {rel('WGT')}")
            for k in range(48 if calls else min(48, p.items * chunks)):
                if buf[c, EVENTS.index("XBEG" if calls else "MBEG"), k] <= t0:
                    break
                line = f"    chunk {k}: "
                if calls:
                    line += f"expand {rel('XBEG', k)}..{rel('XEND', k)}  "
                line += f"mma issue {rel('MBEG', k)}..{rel('MEND', k)}"
                if buf[c, EVENTS.index("EBEG"), k] > t0 and (calls or k < -(-p.items // p.teams)):
                    line += f"   item {k if calls else k * p.teams}: epilogue {rel('EBEG', k)}..{rel('EEND', k)}"
                print(line)
        ends = (buf[:, EVENTS.index("END"), 0] - buf[:, 0, 0])[buf[:, 0, 0] != 0]
        if ends.size:
            print(f"  CTA durations: min {ends.min()} median {int(np.median(ends))} max {ends.max()} over {ends.size} CTAs")
    return 0


if __name__ == "__main__":
    sys.exit(main(sys.argv))
