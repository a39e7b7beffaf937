"""Runs a stack of quantised conv layers (``workloads.NetSpec``) through the C ABI.

Host logic only: buffer planning, weight packing at set-up, the layers bound once as a ``bs_sequence`` and run by one call per
pass (residual adds and concatenations are epilogue arguments), optional CUDA-graph replay.
"""
from __future__ import annotations

import ctypes
import weakref
from typing import Dict, List, Optional

import numpy as np
import torch

from . import api
from ._lib import SequenceLayer, lib, native
from .workloads import NetSpec


class _Sequence:
    """The launches of a pass bound to what they read and write.  ``handle``: the ``bs_sequence``, None where the library does not take the
    layers as one; ``launches``: kernels of a run.  ``dicts`` name the tensors and settings of the layers; ``values`` are what was found there, kept alive because a sequence
    and the graphs captured from it hold the tensors' ``addresses``."""

    def __init__(self, units, concurrent, dicts):
        self.units, self.concurrent = units, concurrent
        self.dicts = tuple(dicts)
        self.values = tuple(v for d in self.dicts for v in d.values())
        self.addresses = tuple(v.data_ptr() if isinstance(v, torch.Tensor) else None for v in self.values)
        self.handle = None
        self.launches = 0
        self.input: Optional[int] = None        # operand tensor of the network's input
        self.workspace: Optional[_Workspace] = None

    def own(self, handle: int, packed: int) -> None:
        self.handle = handle
        self.launches = lib().bs_sequence_launches(handle)
        self.input = lib().bs_sequence_input(handle, packed)
        weakref.finalize(self, lib().bs_sequence_destroy, handle).atexit = False

    def current(self, units, concurrent) -> bool:
        """Whether nothing was replaced since: the dicts hold the same objects, the tensors are where they were."""
        return units is self.units and concurrent == self.concurrent and native().unchanged(self.dicts, self.values, self.addresses)


class _Workspace:
    """Memory of the operand tensors of sequences of one ``geometry``, the last of which had its tensors at ``addresses``.  ``recorded``: a pass that
    uses it went into a graph, which may be replayed beside passes over other tensors."""

    def __init__(self, geometry, addresses, memory: torch.Tensor):
        self.geometry, self.addresses, self.memory, self.recorded = geometry, addresses, memory, False


class BitserialNet:
    MAX_CHAIN = 4
    MAX_WORKSPACES = 4      # arrangements of tensors that have memory for operand tensors; passes over further ones run on packed codes

    def __init__(self, net: NetSpec, params: Dict[str, Dict], act_scale: float, device="cuda", batch: Optional[int] = None,
                 engine: str = "popc", concurrent: bool = True, chains="auto", operand_tensors: bool = True):
        """engine: "popc" = packed filters, expanded on chip; "tc" = filters prepared as operand tiles once for every layer that
        supports it (others keep packed filters).  concurrent: launch independent neighbouring layers on
        two streams (see :meth:`schedule`).  chains: True groups, with the "tc" engine, runs of consecutive same-shaped layers that the
        library accepts into units which :meth:`run_units` issues as one ``bitserial_conv2d_tc_chain`` call each; False and "auto" = a unit per
        layer.  A pass is one call of a bound sequence whatever the units are.
        operand_tensors: with filters prepared as nibbles a pass keeps what the tensor cores read of every tensor between its layers in device memory of
        its own (``bs_sequence_create_ws``), about twice the packed tensors together: 59 MB for the 18-layer stack at 64 images, 139 MB for
        the detection stack at 16, 169 MB for the 50-layer one at 32, held while the runner lives (:attr:`operand_bytes`), once more for every
        set of tensors that a graph was recorded with.  False: no such memory, layers expand packed codes, 1.1 to 1.5 times the time."""
        self.net = net
        self.engine = engine
        self.act_scale = float(act_scale)
        self.device = torch.device(device)
        self.batch = batch or net.batch
        self.shapes = net.tensor_shapes()
        self.layers = []
        for L in net.layers:
            p = params[L.name]
            w = torch.from_numpy(np.ascontiguousarray(p["w"])).to(self.device)
            wp = api.pack_weights(w, net.w_bits, p["w_sign"])
            _, H, W = self.shapes[L.src]
            use_tc = engine == "tc" and api.tc_supported(self.batch, L.C, H, W, L.O, L.k, L.stride, L.pad, net.a_bits,
                                                         api.UNSIGNED, net.w_bits, p["w_sign"])
            self.layers.append(dict(
                spec=L,
                w=wp,
                w_tc=api.tc_prepare_weights(wp, L.C, p["w_sign"], net.a_bits) if use_tc else None,
                w_sign=p["w_sign"],
                scale=torch.from_numpy(p["scale"]).to(self.device),
                bias=torch.from_numpy(p["bias"]).to(self.device)))
        self.bufs: Dict[str, torch.Tensor] = {}
        for name, (C, H, W) in self.shapes.items():
            self.bufs[name] = torch.zeros(self.batch, H, W, (C + 31) // 32, net.a_bits, dtype=torch.int32, device=self.device)
        self.units = self._plan_units(chains is True and engine == "tc")
        torch.cuda.synchronize(self.device)   # chained layers fetch filters, scale and bias ahead of stream order
        self.sms = torch.cuda.get_device_properties(self.device).multi_processor_count
        self.concurrent = concurrent
        self.side = torch.cuda.Stream(device=self.device)
        self.graph = None
        self.static_in = None
        self.launches_per_forward = 1 + len(self.layers)
        self.operand_tensors = operand_tensors
        self._workspaces: List[_Workspace] = []
        self._sequence: Optional[_Sequence] = None
        self._captured: Optional[_Sequence] = None      # what the graph was captured from
        self._bind()

    def _layer_params(self, item):
        """``bs_conv_params`` of a layer as a chain would run it, or None when its output is a slice of a wider tensor."""
        net, L = self.net, item["spec"]
        if L.dst_c_offset != 0 or self.shapes[L.dst][0] != L.O or (L.res and self.shapes[L.res][0] != L.O):
            return None
        return self._conv_params(item)

    def _plan_units(self, chains: bool) -> List[Dict]:
        """The calls of :meth:`run_units`: single layers, and runs of up to MAX_CHAIN consecutive layers that the library
        accepts as one chain (same shape) and whose inputs come from outside the run or from an
        earlier layer of it.  Longest run first, greedily from the front."""
        units, i, n = [], 0, len(self.layers)
        while i < n:
            took = 0
            if chains:
                for length in range(min(self.MAX_CHAIN, n - i), 1, -1):
                    items = self.layers[i:i + length]
                    if any(it["w_tc"] is None for it in items):
                        continue
                    prm = [self._layer_params(it) for it in items]
                    if any(q is None for q in prm):
                        continue
                    dsts = [it["spec"].dst for it in items]
                    if len(set(dsts)) != length:
                        continue
                    if any(t in dsts[k:] for k, it in enumerate(items) for t in (it["spec"].src, it["spec"].res) if t):
                        continue
                    nbytes = api.tc_chain_workspace_bytes(prm)
                    if nbytes == 0:
                        continue
                    ws = torch.zeros((nbytes + 3) // 4, dtype=torch.int32, device=self.device)
                    units.append(dict(items=items, params=prm, workspace=ws))
                    took = length
                    break
            if not took:
                units.append(dict(items=[self.layers[i]], params=None, workspace=None))
                took = 1
            i += took
        return units

    def _run(self, x: torch.Tensor) -> torch.Tensor:
        bound = self._bind()
        self._layers(self._pack(x, self._sequence.input if bound else None), bound)
        return self.bufs[self.net.out_name]

    @property
    def operand_bytes(self) -> int:
        """Device memory of the operand tensors (see the constructor)."""
        return sum(w.memory.numel() for w in self._workspaces)

    def input_operands(self) -> Optional[int]:
        """The operand tensor of the packed input (``bs_sequence_input``), which a producer of the input may write as well, or None.  It is
        the bound sequence's: valid until an entry of the layers is replaced."""
        return self._sequence.input if self._bind() else None

    def pack_input(self, x: torch.Tensor, operands: bool = False) -> Optional[int]:
        """Quantise + bitplane-pack the fp32 input on the current stream.  operands: its operand tensor too, where the layers have one and ``x`` is
        the whole input; :meth:`run_layers` takes the object that is returned then, as long as neither is written in between."""
        return self._pack(x, self.input_operands() if operands else None)

    def _pack(self, x: torch.Tensor, operands: Optional[int]) -> Optional[int]:
        net, buf = self.net, self.bufs[self.net.in_name]
        if operands is not None and x.dtype == torch.float32 and tuple(x.shape) == (self.batch, *net.in_shape):
            api.bitpack_operands(x, self.act_scale, net.a_bits, buf, operands)
            return operands
        api.bitpack_activations(x, self.act_scale, net.a_bits, api.UNSIGNED, api.NCHW, out=buf.view(-1))
        return None

    def run_layer(self, item, chained: bool = True) -> None:
        """One conv layer through the C ABI on the current stream."""
        net, L = self.net, item["spec"]
        res = self.bufs[L.res] if L.res else None
        api.bitserial_conv2d(
            self.bufs[L.src], item["w"], C=L.C, stride=L.stride, pad=L.pad, a_sign=api.UNSIGNED,
            w_sign=item["w_sign"], scale=item["scale"], bias=item["bias"], relu=L.relu, out_bits=net.a_bits,
            out_sign=api.UNSIGNED, residual=res, res_scale=L.res_scale, res_bits=net.a_bits if L.res else 0,
            res_sign=api.UNSIGNED, res_c_offset=0, res_c_total=self.shapes[L.res][0] if L.res else 0,
            out_packed=self.bufs[L.dst], out_c_offset=L.dst_c_offset, out_c_total=self.shapes[L.dst][0],
            wgt_tc=item["w_tc"], chained=chained and item["w_tc"] is not None)

    def run_unit(self, unit, chained: bool = True) -> None:
        """One call on the current stream: a layer, or a chain of layers."""
        if unit["params"] is None:
            self.run_layer(unit["items"][0], chained=chained)
            return
        items = unit["items"]
        params = [self._layer_params(it) for it in items]       # pointers of the buffers as they are now (tests swap them)
        api.bitserial_conv2d_tc_chain([self.bufs[it["spec"].src] for it in items], [self._filters(it)[0] for it in items], params,
                                      [self.bufs[it["spec"].dst] for it in items], unit["workspace"], chained=chained)

    def schedule(self):
        """The calls in order: (unit, aside, join).  With ``concurrent`` a single layer whose successor neither reads nor
        overwrites its output (a projection shortcut beside the first conv of its block, the two 1x1 branches of a cross-stage
        block) runs ``aside`` on a second stream when it does not fill the GPU by itself: at most one 128 x 128 block of outputs per
        multiprocessor (a measure of its size; the plans cut their own tiles).  ``join``: positions of the calls that must be waited for first.

        Layers of a pass as a graph, us, never aside / by this line / always where the data allow (B200, operand tensors):
        18-layer stack, batch 1: 62.0 / 59.9 / 59.9, 8: 74.6 / 73.6 / 73.9, 16: 85.0 / 85.4 / 84.6, 64: 143.7 / 143.9 / 145.5;
        50-layer stack, 1: 173.2 / 169.4 / 169.2, 8: 231.1 / 231.6 / 232.1, 32: 382.3 / 382.6 / 386.8;
        detection stack (160 px), 1: 82.3 / 77.6 / 78.0, 4: 90.6 / 88.4 / 89.0, 16: 118.5 / 117.2 / 121.3, 32: 145.8 / 147.9 / 152.0.
        Up to 6 % gained while a layer leaves room, about 1 % lost near the line, up to 4 % where both neighbours fill the GPU."""
        out, pending = [], {}
        n = len(self.units)

        def touched(unit):
            reads, writes = set(), set()
            for it in unit["items"]:
                L = it["spec"]
                reads.update(t for t in (L.src, L.res) if t)
                writes.add((L.dst, L.dst_c_offset))
            return reads, writes

        for i, unit in enumerate(self.units):
            reads, writes = touched(unit)
            wnames = {d for d, _ in writes}
            aside = False
            if self.concurrent and i + 1 < n and len(unit["items"]) == 1:
                nreads, nwrites = touched(self.units[i + 1])
                L = unit["items"][0]["spec"]
                _, P, Q = self.shapes[L.dst]
                small = -(-self.batch * P * Q // 128) * -(-L.O // 128) <= self.sms
                aside = (small and not (wnames & nreads) and not ({d for d, _ in nwrites} & reads) and not (writes & nwrites)
                         and not (reads & set(pending)))
            join = []
            if aside:
                pending.update({d: i for d in wnames})
            else:
                join = sorted({pending.pop(t) for t in list(reads | wnames) if t in pending})
                if i + 1 == n:                      # the pass ends with its last launch
                    join = sorted(set(join) | set(pending.values()))
            out.append((unit, aside, join))
        return out

    def run_layers(self, ready: Optional[int] = None) -> None:
        """All layers on the current stream, and on the side stream those that :meth:`schedule` puts there; under stream capture the
        events between them become the edges of the graph.  ready: the operand tensor of the input, where it holds what the packed input holds."""
        self._layers(ready, self._bind())

    def _layers(self, ready: Optional[int], bound: bool) -> None:
        """:meth:`run_layers` behind a look at the tensors: a pass takes one, in front of what writes its input."""
        if bound:
            q = self._sequence
            ready = ready if ready is q.input else None         # (an address may come back with another sequence, the object does not)
            api.run_sequence(q.handle, q.launches - (ready is not None), ready=ready)
        else:
            self.run_units()

    def run_units(self) -> None:
        """The same layers one call per unit, on packed codes: what :meth:`run_layers` does where the library does not take them as one sequence."""
        main = torch.cuda.current_stream(self.device)
        done: Dict[int, torch.cuda.Event] = {}
        for i, (unit, aside, join) in enumerate(self.schedule()):
            if aside:
                fork = torch.cuda.Event()
                fork.record(main)
                self.side.wait_event(fork)
                with torch.cuda.stream(self.side):
                    self.run_unit(unit, chained=False)
                    done[i] = torch.cuda.Event()
                    done[i].record(self.side)
                continue
            for k in join:
                main.wait_event(done[k])
            self.run_unit(unit)

    def _bind(self) -> bool:
        """Binds the layers as one sequence to the tensors and settings they have now, again when one was replaced; False where the library does
        not take them as one."""
        q, recording = self._sequence, torch.cuda.is_current_stream_capturing()
        if q is not None and q.current(self.units, self.concurrent):
            if recording and q.workspace is not None:
                q.workspace.recorded = True
            return q.handle is not None
        items = [item for unit in self.units for item in unit["items"]]
        self._sequence = _Sequence(self.units, self.concurrent, [self.bufs, *items, *(vars(item["spec"]) for item in items)])
        if q is not None and not recording:
            torch.cuda.synchronize(self.device)     # as at set-up: what replaced a filter, scale or bias has to be final
        steps = self.schedule()
        at, layers = {}, []                          # position of a launch among the layers
        for i, (unit, aside, join) in enumerate(steps):
            for k, item in enumerate(unit["items"]):
                if k == 0:
                    at[i] = len(layers)
                layers.append((item, aside, [at[j] for j in join] if k == 0 else []))
        if any(len(j) > 4 for _, _, j in layers):
            return False
        arr = (SequenceLayer * len(layers))()
        for q, (item, aside, join) in zip(arr, layers):
            L = item["spec"]
            q.act_packed, q.out_packed = api._ptr(self.bufs[L.src]), api._ptr(self.bufs[L.dst])
            q.wgt_packed, q.wgt_tc = api._ptr(item["w"]), api._ptr(self._filters(item)[0])
            q.p = self._conv_params(item)
            q.chained, q.aside = 1, int(aside)
            q.join[:] = (join + [-1] * 4)[:4]
        handle = ctypes.c_void_p()
        ws = self._sequence.workspace = self._workspace(arr, recording)
        memory, nbytes = (api._ptr(ws.memory), ws.memory.numel()) if ws is not None else (None, 0)
        if lib().bs_sequence_create_ws(arr, len(layers), self.side.cuda_stream, memory, nbytes, ctypes.byref(handle)) != 0:
            return False
        if recording and ws is not None:
            ws.recorded = True
        self._sequence.own(handle.value, api._ptr(self.bufs[self.net.in_name]))
        self.launches_per_forward = 1 + self._sequence.launches - (self._sequence.input is not None)
        return True

    def _workspace(self, arr, recording: bool) -> Optional[_Workspace]:
        """Memory of the layers' operand tensors (``bs_sequence_create_ws``), or None.  What a graph was recorded with stays with its tensors while the
        runner lives; otherwise it passes on to the next arrangement of the same geometry, whose passes begin on an idle device."""
        nbytes = lib().bs_sequence_workspace_bytes(arr, len(arr)) if self.operand_tensors else 0
        if nbytes == 0:
            return None
        tensors = {}
        at = lambda address: tensors.setdefault(address, len(tensors))
        # (filters that a pass prepares lie there as well)
        geometry = (nbytes, *((at(q.act_packed), at(q.out_packed), bool(q.wgt_tc), *(getattr(q.p, f) for f in (
            "N", "C", "H", "W", "O", "R", "stride", "pad", "a_bits", "out_bits", "out_c_offset", "out_c_total"))) for q in arr))
        addresses = tuple(tensors)
        alike = [w for w in self._workspaces if w.geometry == geometry]
        for w in alike:
            if w.addresses == addresses:
                return w
        if recording:                           # (its clearing would belong to the graph, and nobody has waited for passes under way)
            return None
        for w in alike:
            if not w.recorded:
                w.addresses = addresses
                return w
        self._workspaces = [w for w in self._workspaces if w.recorded]
        if len(self._workspaces) >= self.MAX_WORKSPACES:
            return None
        try:
            memory = torch.zeros(nbytes, dtype=torch.uint8, device=self.device)
        except torch.OutOfMemoryError:
            return None
        torch.cuda.synchronize(self.device)
        self._workspaces.append(_Workspace(geometry, addresses, memory))
        return self._workspaces[-1]

    def _filters(self, item):
        """Prepared filters of a layer, or None, and the sign that goes with them."""
        return api.tc_weights_form(item["w_tc"], item["w"].shape, item["spec"].C, item["w_sign"], self.net.a_bits)

    def _conv_params(self, item):
        net, L = self.net, item["spec"]
        q = api.conv_params(
            self.bufs[L.src].shape, item["w"].shape, C=L.C, stride=L.stride, pad=L.pad, a_sign=api.UNSIGNED, w_sign=self._filters(item)[1],
            scale=item["scale"], bias=item["bias"], relu=L.relu, out_bits=net.a_bits, out_sign=api.UNSIGNED,
            residual=self.bufs[L.res] if L.res else None, res_scale=L.res_scale, res_bits=net.a_bits if L.res else 0,
            res_sign=api.UNSIGNED)
        q.res_c_total = self.shapes[L.res][0] if L.res else L.O
        q.out_c_offset, q.out_c_total = L.dst_c_offset, self.shapes[L.dst][0]
        return q

    def prefetch_filters(self) -> None:
        """A hint before a pass whose filters have left L2: they start on their way there (a separate launch; a pass does not issue it,
        since it gains nothing while the filters are still in L2)."""
        api.l2_prefetch([t for item in self.layers for t in (
            [item["w"]] if item["w_tc"] is None else api.tc_weights_read(item["w_tc"], item["w"].shape, item["spec"].C, self.net.a_bits))])

    def forward(self, x: torch.Tensor) -> torch.Tensor:
        """x: float32 [batch, C, H, W] on the device.  Returns the packed output tensor of the stack."""
        return self._run(x)

    def capture(self, x: torch.Tensor) -> None:
        """Record one forward pass into a CUDA graph replayed by :meth:`replay` (input copied into a static buffer).  The graph keeps the
        tensors it was captured with; entries replaced later take effect in :meth:`forward` and in the next capture."""
        self.static_in = x.clone()
        self._run(self.static_in)            # warm-up outside capture: plans, descriptors, module loading
        torch.cuda.synchronize()
        self.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(self.graph):
            self._run(self.static_in)
        self._captured = self._sequence

    def replay(self, x: Optional[torch.Tensor] = None) -> torch.Tensor:
        if x is not None:
            self.static_in.copy_(x, non_blocking=True)
        self.graph.replay()
        return self.bufs[self.net.out_name]

    def unpacked(self, name: str) -> torch.Tensor:
        """int8 NCHW codes of an activation tensor (debugging / tests)."""
        C = self.shapes[name][0]
        return api.bitunpack_activations(self.bufs[name], C, self.net.a_bits, api.UNSIGNED, api.NCHW)


class BitserialFullNet:
    """The whole mixed-precision classifier of ``workloads.FullNetSpec`` through the C ABI: floating-point stem and quantiser (one kernel,
    ``bs_stem_codes_f32``, or ``bs_conv2d_f32`` + ``bs_maxpool2d_f32`` + quantise and pack for shapes it does not take), the quantised body
    (:class:`BitserialNet`), floating-point head (``bs_avgpool_codes_f32`` + ``bs_fc_f32``).  Host logic only."""

    MAX_CAPTURES = 16       # recorded passes whose images are kept for :attr:`stem_conv`

    def __init__(self, net, params: Dict[str, Dict], device="cuda", batch: Optional[int] = None, engine: str = "tc", operand_tensors: bool = True):
        self.net = net
        self.batch = batch or net.batch
        self.device = torch.device(device)
        self.body = BitserialNet(net.body, params, net.stem_act_scale, device=device, batch=self.batch, engine=engine, operand_tensors=operand_tensors)
        to = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(self.device)
        self.stem_w, self.stem_b = to(params["stem"]["w"]), to(params["stem"]["bias"])
        self.fc_w, self.fc_b = to(params["fc"]["w"]), to(params["fc"]["bias"])
        h1 = (net.hw + 2 * 3 - 7) // 2 + 1
        h2 = (h1 + 2 - 3) // 2 + 1
        self._stem_sizes = dict(conv=h1, pool=h2)
        self._stem: Dict[str, torch.Tensor] = {}                # the stem's float tensors, from their first use on
        self._stem_held: Dict[str, weakref.ref] = {}            # what was handed out of them
        self._stem_assigned = False                             # the caller has put tensors of their own in their place
        self._codes_only: Optional[torch.Tensor] = None         # images of the last pass launched, where it made codes only
        self._captures: Dict[int, torch.Tensor] = {}            # ... of the passes recorded into graphs, by number
        self._recorded = 0
        # number of the recorded pass that ran last where it made codes only, -1 where it made the tensors; 0 after a launched one
        self._replayed = torch.zeros((), dtype=torch.int32, device=self.device)
        C, H, W = net.body.tensor_shapes()[net.body.out_name]
        self.pooled = torch.empty(self.batch, C, dtype=torch.float32, device=self.device)
        self.logits = torch.empty(self.batch, net.classes, dtype=torch.float32, device=self.device)
        self.inv = float(np.float32(np.float32(net.body_act_scale) / np.float32(H * W)))

    @property
    def launches_per_forward(self) -> int:
        """Kernels of a pass as it would run now: two more where the stem runs as layers of its own."""
        fused = not self._watched() and api.stem_codes_supported((self.batch, 3, self.net.hw, self.net.hw), self.stem_w.shape, self.body.act_scale,
                                                                 self.body.net.a_bits)
        return self.body.launches_per_forward + (2 if fused else 4)

    def run_stem(self, images: torch.Tensor) -> None:
        """The stem as layers of its own: images to ``stem_conv`` and ``stem_pool``."""
        self._stem_layers(images)
        self._note_pass(None)
        self._join_note()

    def run_front(self, images: torch.Tensor) -> None:
        """Images to the body's packed input.  Codes only, where the library has the stem as one kernel and nobody holds the stem's tensors."""
        self._front(images)
        self._join_note()

    def _front(self, images: torch.Tensor, ready: Optional[int] = None) -> Optional[int]:
        body = self.body
        if not self._watched() and tuple(images.shape) == (self.batch, 3, self.net.hw, self.net.hw) and api.stem_codes_f32(
                images, self.stem_w, self.stem_b, body.act_scale, body.net.a_bits, body.bufs[body.net.in_name], operands=ready):
            self._note_pass(images)
            return ready
        self._stem_layers(images)
        self._note_pass(None)
        return body._pack(self._stem["pool"], ready)

    def _stem_layers(self, images: torch.Tensor) -> None:
        conv, pool = self._stem_tensor("conv"), self._stem_tensor("pool")
        api.conv2d_f32(images, self.stem_w, self.stem_b, stride=2, pad=3, relu=True, out=conv)
        api.maxpool2d_f32(conv, 3, 2, 1, out=pool)

    def _stem_tensor(self, name: str) -> torch.Tensor:
        t = self._stem.get(name)
        if t is None:
            hw = self._stem_sizes[name]
            t = self._stem[name] = torch.empty(self.batch, 64, hw, hw, dtype=torch.float32, device=self.device)
        return t

    def _watched(self) -> bool:
        return self._stem_assigned or any(r() is not None for r in self._stem_held.values())

    def _note_pass(self, images: Optional[torch.Tensor]) -> None:
        """Records that the stem's tensors follow from ``images`` from here on, or (None) that they hold what belongs to the last pass.  A pass recorded
        into a graph records this as well: Python does not run when the graph does.  It does so beside the layers, on the body's second stream
        (between them it cost 3.6 of 299 us); :meth:`_join_note` has to follow."""
        if torch.cuda.is_current_stream_capturing():
            self._recorded += 1
            if images is not None:
                self._captures[self._recorded] = images
                if len(self._captures) > self.MAX_CAPTURES:
                    del self._captures[min(self._captures)]
            main = torch.cuda.current_stream(self.device)
            self.body.side.wait_stream(main)
            with torch.cuda.stream(self.body.side):
                self._replayed.fill_(self._recorded if images is not None else -1)
        else:
            self._codes_only = images
            if self._recorded:
                self._replayed.zero_()

    def _join_note(self) -> None:
        if torch.cuda.is_current_stream_capturing():
            torch.cuda.current_stream(self.device).wait_stream(self.body.side)

    def _read_stem(self, name: str) -> torch.Tensor:
        """The tensor ``name`` of the last pass, evaluated first where that pass made codes only."""
        images, recording = self._codes_only, torch.cuda.is_current_stream_capturing()
        if self._recorded and not recording:
            k = int(self._replayed)
            if k > 0 and k not in self._captures:
                raise RuntimeError("the last pass was a replay of a graph recorded long ago: the images it read are not known any more")
            if k != 0:
                images = self._captures[k] if k > 0 else None
        if images is not None:
            body = self.body
            self._stem_layers(images)
            if not recording and not torch.equal(api.bitpack_activations(self._stem["pool"], body.act_scale, body.net.a_bits).view(-1),
                                                 body.bufs[body.net.in_name].view(-1)):
                raise RuntimeError("images, stem or body input have changed since the last pass, which made codes only: read stem_conv or stem_pool "
                                   "before that, or hold one of them while passes run")
            if not recording:
                self._note_pass(None)       # nothing to join: not recorded
        held = self._stem_held.get(name)
        t = held() if held is not None else None
        if t is None:
            t = self._stem_tensor(name).detach()
            self._stem_held[name] = weakref.ref(t)
        return t

    def _assign_stem(self, name: str, t: torch.Tensor) -> None:
        self._read_stem(name)
        self._stem[name] = t
        self._stem_assigned = True
        self._stem_held.pop(name, None)
        self._note_pass(None)
        self._join_note()

    @property
    def stem_conv(self) -> torch.Tensor:
        """Float output of the stem convolution in the last pass, replays of recorded ones included.  While the tensor (or ``stem_pool``) is held, every
        pass that is launched or recorded writes both.  Otherwise passes make codes only, and a read evaluates the tensors from the images of the
        last pass; it raises where these have changed since.  A graph recorded while nobody held them makes codes only: after its replays a
        held tensor is brought up to date by the next read."""
        return self._read_stem("conv")

    @stem_conv.setter
    def stem_conv(self, t: torch.Tensor) -> None:
        self._assign_stem("conv", t)

    @property
    def stem_pool(self) -> torch.Tensor:
        """Float output of the stem's pooling, like :attr:`stem_conv`."""
        return self._read_stem("pool")

    @stem_pool.setter
    def stem_pool(self, t: torch.Tensor) -> None:
        self._assign_stem("pool", t)

    def run_head(self) -> None:
        body = self.net.body
        api.avgpool_codes_f32(self.body.bufs[body.out_name], body.tensor_shapes()[body.out_name][0], api.UNSIGNED, self.inv, out=self.pooled)
        api.fc_f32(self.pooled, self.fc_w, self.fc_b, out=self.logits)

    def forward(self, images: torch.Tensor) -> torch.Tensor:
        """images: float32 [batch, 3, hw, hw] on the device.  Returns the logits [batch, classes]."""
        body = self.body
        bound = body._bind()
        body._layers(self._front(images, body._sequence.input if bound else None), bound)
        self.run_head()
        self._join_note()
        return self.logits
