"""Sequences the C-ABI calls of a whole network (``workloads.networks.Net``).

PyTorch supplies device memory and the stream; every layer runs in the CUDA library.
Per-layer integer parameters (quantisation step, mul, shift, h_i, skip rescale) arrive as
a dict, e.g. read from ``workloads/params/*.json``; weights are re-created from the
network's seed with the library's own Eq. 1 (``iq_quantize_weights``).
"""
from collections.abc import ItemsView, ValuesView

import numpy as np
import torch

from workloads import generators as gen
from workloads.networks import AvgPool, Conv, MaxPool, Net
from workloads.params import load_params  # noqa: F401  (re-exported: callers read cached parameters through here too)

from . import binding as B

FLOW_MAX_LAYERS = 50      # layers of one stack the library takes at most
_TORCH = {"u8": torch.uint8, "i32": torch.int32}

def net_input(net: Net, first: int = 0, count=None) -> np.ndarray:
    t = net.tensors[net.input]
    count = net.n - first if count is None else count
    if net.input_kind == "uniform":
        return np.ascontiguousarray(gen.uniform_u8(net.seed, (net.n, t.h, t.w, t.c))[first:first + count])
    return gen.image_batch(net.seed, count, t.h, t.w, t.c, first=first)


def _stack_kernel(run) -> str:
    """The kernel in which the library runs the layers of a stack: its form for equal layers of few channels, or the general one."""
    a = run[0]
    equal = a.k == 3 and a.stride == 1 and a.pad == 1 and 32 < a.c_in <= 64 and a.c_out <= 64 and all(
        (o.c_in, o.c_out, o.k, o.stride, o.pad, o.skip) == (a.c_in, a.c_out, 3, 1, 1, None) and (i == 0 or o.src == run[i - 1].dst)
        for i, o in enumerate(run))
    return "umma_stack_kernel" if equal else "umma_flow_kernel"


class _LeftOut:
    """The output of a first layer whose kernel goes on to the max-pool (``fuse_pool``), for whoever looks at it.  The forwards leave
    the tensor out until the first look and write it, in a launch of its own, from then on.  A look fills it with what the last
    forward's would be: what that forward read is in the repacked image, which its workspace holds until the next one, while the input
    tensor may have changed since, and a graph captured before the first look does not write the tensor when it is replayed."""

    def __init__(self, kw):
        self.kw, self.plan = kw, B.iconv_plan(**kw)
        self.repacked = self.scratch = None      # the network's workspace, with the image as the last forward left it; this layer's own
        self.stream = None                       # the last forward's
        self.looked_at = False

    def __del__(self):
        try:
            B.iconv_plan_destroy(self.plan)
        except Exception:
            pass

    def write(self, x, out, stream):
        """The layer by itself, from the images at address x."""
        if self.scratch is None:
            self.scratch = torch.empty((B.iconv_workspace_bytes(self.plan),), dtype=torch.uint8, device=out.device)
        B.iconv_forward(self.plan, x, None, out.data_ptr(), self.scratch.data_ptr(), stream)

    def look(self, out) -> torch.Tensor:
        self.looked_at = True
        if self.stream is not None:
            here = torch.cuda.current_stream(out.device)
            apart = here != self.stream and not (_captured(here) or _captured(self.stream))
            if apart:
                here.wait_stream(self.stream)
            x = self.images(out)
            self.write(x.data_ptr(), out, here.cuda_stream)
            if apart:
                self.stream.wait_stream(here)               # the next forward there writes what is read here
        return out

    def images(self, out) -> torch.Tensor:
        """The images out of the repacked ones.  Those are 16-byte positions of 2 x 2 pixels x 3 channels and four bytes of zeros, two
        positions above and four to the left of the image, a row's even positions before its odd ones (``stem_repack_wide_kernel``)."""
        n, h_out, w_out, _ = out.shape
        half = (w_out + 8) // 4 * 2                         # positions of either kind in a row
        t = self.repacked[:n * (h_out + 3) * half * 32].view(n, h_out + 3, 2, half, 16)[..., :12].unflatten(4, (2, 2, 3))
        x = t.permute(0, 1, 4, 3, 2, 5, 6).reshape(n, 2 * (h_out + 3), 4 * half, 3)[:, 4:4 + self.kw["h"], 8:8 + self.kw["w"]]
        return (x ^ 128 if self.kw["in_dtype"] == B.U8_RAW128 else x).contiguous()


def _captured(stream) -> bool:
    with torch.cuda.stream(stream):
        return torch.cuda.is_current_stream_capturing()


class _Tensors(dict):
    """A network's tensors by name.  One that its forwards leave out is filled in whenever it is looked up."""

    def __init__(self):
        super().__init__()
        self.left_out = {}                       # name -> _LeftOut

    def __getitem__(self, name):
        t = super().__getitem__(name)
        return self.left_out[name].look(t) if name in self.left_out else t

    def __iter__(self):                          # (one of its own, so that dict(tensors) takes the values by __getitem__)
        return super().__iter__()

    def get(self, name, default=None):
        return self[name] if name in self else default

    def values(self):
        return ValuesView(self)

    def items(self):
        return ItemsView(self)

    def copy(self):
        return dict(self)


class Network:
    """Plans every layer once; ``forward`` enqueues the whole network on the current stream."""

    def __init__(self, net: Net, params: dict, n=None, device="cuda:0", kernel=B.KERNEL_AUTO, fuse_projection=True,
                 merge_branches=True, fuse_chain=True, stack_layers=True, fuse_pool=True):
        """fuse_projection: run a projection skip (a "raw" convolution whose int32 output only feeds
        the next layer's skip) inside that layer's kernel; its int32 tensor is then never written.
        merge_branches: plan two convolutions that read the same tensor and write neighbouring
        channel ranges of the same concatenation (a variable-filter-size block) as one layer: the
        smaller filter sits zero-padded in the middle of the larger one, every channel keeps its
        own bias, h_i, mul and shift.  The sums only gain zero terms, so the bytes are the same.
        fuse_chain: run a block-closing 1x1 layer with an 8-bit identity skip and the 1x1 layer that
        reads its output as ONE kernel where the library takes the pair (``iconv_plan_chain``): the
        wide tensor is still written (later layers read it as their skip) but not read back by the
        next layer, and one launch goes.
        stack_layers: run consecutive layers as ONE kernel where the library takes the run
        (``iconv_plan_stack``): equal 3x3 layers, or 1x1 and k x k layers with their skips and
        projections where that is the faster way (``_flow_takes``).  A tile waits for the tiles it
        reads, not for a whole layer; the launch takes the whole GPU.  A stack is bound to the
        tensors of this network and to its counters: one forward at a time.
        fuse_pool: run a first layer and the max-pool that alone reads its output as ONE kernel where that is the faster
        way (``_pool_takes``) and the library takes the pair (``iconv_plan_stem_pool``); the layer's own tensor, four times the pooled one, is then
        filled in when it is first looked up in ``tensors``, and by every forward from then on."""
        self.net, self.n, self.device = net, net.n if n is None else n, torch.device(device)
        self.plans, self.steps, self.tensors = {}, [], _Tensors()
        self.chains = {}         # name of a closing layer -> chain handle; self.chained: second op name -> closing layer
        self.chained = {}
        self.stacks = {}         # name of a run's first layer -> stack handle; self.stacked: name of a later layer -> that first layer
        self.stacked = {}
        self.fused = {}          # name of a fused projection op -> name of the layer that absorbed it
        self.pooled = {}         # name of a max-pool -> name of the first layer whose kernel runs it
        self.merged = {}         # name of a branch convolution -> name of the sibling whose plan runs both
        self._pending = {}
        self._quantised = {}     # name of a convolution -> its integer weights, until everything is planned
        self._refused = set()    # (kind of run, name of a layer) that the library takes into no such run
        torch.cuda.set_device(self.device)
        convs = {op.name: op for op in net.convs()}
        fusable = {}             # skip tensor name -> projection op
        if fuse_projection and kernel in (B.KERNEL_AUTO, B.KERNEL_UMMA):
            for op in net.convs():
                if op.role == "raw" and op.dst != net.output:
                    users = [o for o in net.ops if getattr(o, "src", None) == op.dst or getattr(o, "skip", None) == op.dst]
                    if len(users) == 1 and getattr(users[0], "skip", None) == op.dst and getattr(users[0], "src", None) != op.dst:
                        fusable[op.dst] = op
        for name, t in net.tensors.items():
            self.tensors[name] = torch.zeros((self.n, t.h, t.w, t.c), dtype=_TORCH[t.dtype], device=self.device)
        partner = self._partner = {}      # first op of a merged pair -> second
        if merge_branches and kernel in (B.KERNEL_AUTO, B.KERNEL_UMMA):
            for a, b in zip(net.ops, net.ops[1:]):
                if a.name not in self.merged and self._mergeable(a, b, params):
                    partner[a.name] = b
                    self.merged[b.name] = a.name
        for op in net.ops:
            src, dst = net.tensors[op.src], net.tensors[op.dst]
            if op.name in self.merged or op.name in self.chained or op.name in self.stacked:
                continue
            if op.name in self.fused or op.name in self.stacks or op.name in self.pooled:
                continue        # (a run may begin with a projection: it is then planned before its first layer is met)
            if fuse_pool and self._try_pool(op, params, kernel):
                continue
            if stack_layers and (self._try_stack(op, params, kernel) or self._try_flow(op, fusable, params, kernel)):
                continue
            if op.name in partner:
                self.plans[op.name] = self._plan_merged(op, partner[op.name], params, kernel)
                self.steps.append(("conv", op, None))
                continue
            if isinstance(op, MaxPool):
                self.steps.append(("max", op, None))
            elif isinstance(op, AvgPool):
                self.steps.append(("avg", op, params[op.name]))
            else:
                if op.dst in fusable and self._try_fuse(op, fusable, params, kernel):
                    continue
                p = params[op.name]
                kw = dict(n=self.n, h=src.h, w=src.w, c_in=op.c_in, c_out=op.c_out, kh=op.k, kw=op.k,
                          stride=op.stride, pad=op.pad, in_dtype=B.DTYPE_CODE[op.in_dtype], in_c_total=src.c,
                          in_c_offset=op.in_c_offset, out_c_total=dst.c, out_c_offset=op.out_c_offset,
                          weights=self._weights(op, params),
                          bias=gen.bias_i32(net.seed, op.layer, op.c_out), kernel=kernel)
                fused = self._pending.pop(op.skip, None) if op.skip else None
                if fused is not None:
                    kw.update(skip_dtype=fused["skip_dtype"], skip_mul=p["skip_mul"], skip_shift=p["skip_shift"],
                              proj=fused["proj"])
                elif op.skip:
                    kw.update(skip_dtype=B.DTYPE_CODE[op.skip_dtype], skip_c_total=net.tensors[op.skip].c,
                              skip_mul=p["skip_mul"], skip_shift=p["skip_shift"])
                if op.role == "raw":
                    kw.update(out_dtype=B.I32, brelu=0)
                else:
                    kw.update(out_dtype=B.U8, brelu=p["brelu"], mul=p["mul"], shift=p["shift"], h_i=p["h_i"],
                              out_lo=p["out_lo"], out_hi=p["out_hi"], out_zero=p["out_zero"])
                if fused is not None:
                    try:
                        self.plans[op.name] = B.iconv_plan(**kw)
                    except B.IconvError as e:
                        if e.status != B.ERR_UNSUPPORTED:
                            raise
                        raise RuntimeError("fused projection refused for %s: %s (build the network with "
                                           "fuse_projection=False)" % (op.name, e))
                    self.fused[fused["op"].name] = op.name
                    self.tensors.pop(fused["op"].dst, None)        # the projection's int32 output is never written
                    self.steps.append(("conv", op, fused["op"].src))
                    continue
                nxt = self._chain_partner(op, kernel) if fuse_chain else None
                if nxt is not None:
                    try:
                        self.chains[op.name] = B.iconv_plan_chain(kw, self._conv_kwargs(nxt, params, kernel))
                        self.chained[nxt.name] = op.name
                        self.steps.append(("chain", op, nxt))
                        continue
                    except B.IconvError as e:
                        if e.status != B.ERR_UNSUPPORTED:
                            raise
                self.plans[op.name] = B.iconv_plan(**kw)
                self.steps.append(("conv", op, None))
        self._quantised.clear()
        self._alloc_workspace()

    def _weights(self, op, params) -> np.ndarray:
        """The integer weights of a convolution (a layer may be planned in several forms before one is taken)."""
        w = self._quantised.get(op.name)
        if w is None:
            w_f = gen.weights_f(self.net.seed, op.layer, op.c_out, op.k, op.k, op.c_in)
            w = self._quantised[op.name] = B.iq_quantize_weights(w_f, params[op.name]["delta"])
        return w

    def _try_pool(self, op, params, kernel) -> bool:
        """Plan the first layer `op` and the max-pool that is the only reader of its output as one kernel."""
        ops = self.net.ops
        i = ops.index(op)
        pool = ops[i + 1] if i + 1 < len(ops) else None
        if kernel != B.KERNEL_AUTO or not isinstance(op, Conv) or not isinstance(pool, MaxPool) or pool.src != op.dst or op.dst == self.net.output:
            return False
        if (op.k, op.stride, op.pad, op.c_in) != (7, 2, 3, 3) or op.skip or op.role != "act" or (pool.k, pool.stride, pool.pad) != (3, 2, 1):
            return False
        if sum(1 for o in ops if getattr(o, "src", None) == op.dst or getattr(o, "skip", None) == op.dst) != 1:
            return False
        if not self._pool_takes(op):
            return False
        kw = self._conv_kwargs(op, params, kernel)
        try:
            self.plans[op.name] = B.iconv_plan_stem_pool(**kw)
        except B.IconvError as e:
            if e.status != B.ERR_UNSUPPORTED:
                raise
            return False
        self.pooled[pool.name] = op.name
        self.tensors.left_out[op.dst] = _LeftOut(kw)
        self.steps.append(("pool", op, pool))
        return True

    def _pool_takes(self, op) -> bool:
        """Is this first layer better off in one kernel with its max-pool?  That kernel walks down bands of the image, two images and
        two strips of 29 pooled columns at a time and two such walks a CTA, and its time is the steps of the longest CTA, about
        2 us each, however few of the lanes have a column; the two kernels apart take 0.048 us per 1000 of the layer's pixels.  Measured
        with the repack (us, one kernel / apart): 256 images of 224 x 224 80.6 / 165.7, of 64 x 64 26.6 / 21.9, of 32 x 32 17.1 / 12.5, of 1600 x 16 371
        / 83; 16 of 64 x 64 8.4 / 11.2, 7 of 231 x 315 13 / 15; always faster while the walks are no more than the SMs.  The line is drawn
        with 152 such pairs: none that is faster in one kernel is left out, what is slower in it and taken is so by 2.7 us at most."""
        t = self.net.tensors[op.dst]
        rows = (t.h + 1) // 2
        columns = -(-((t.w + 1) // 2) // 58) * -(-self.n // 2)
        steps = lambda bands: -(-columns * bands // (2 * 148)) * (-(-rows // bands) + 1)
        bands = min(range(1, rows + 1), key=steps)
        return columns * bands <= 148 or steps(bands) * 48000 <= 90000 + self.n * t.h * t.w

    def _try_stack(self, op, params, kernel) -> bool:
        """Plan the run of plain layers that starts at `op`, all of its geometry and each reading the
        one before, as one kernel; False when there is no such run or the library does not take it."""
        plain = lambda o: isinstance(o, Conv) and o.role == "act" and not o.skip and o.in_dtype == "u8" and not self._is_merged(o)
        if kernel not in (B.KERNEL_AUTO, B.KERNEL_UMMA) or not plain(op) or op.src == self.net.input:
            return False        # (the network's input is whatever tensor a forward is given: a stack is bound to its own)
        shape = lambda o: (o.c_in, o.c_out, o.k, o.stride, o.pad)
        ops = self.net.ops
        i = ops.index(op)
        run = [op]
        for o in ops[i + 1:]:
            if not plain(o) or o.src != run[-1].dst or o.in_c_offset != run[-1].out_c_offset or shape(o) != shape(op):
                break
            run.append(o)
        if len(run) < 2:
            return False
        if any(("stack", o.name) in self._refused for o in run):
            return False
        ptr = lambda name: self.tensors[name].data_ptr()
        stack = self._plan_stack("stack", run, [(self._conv_kwargs(o, params, kernel), ptr(o.src), ptr(o.dst)) for o in run])
        if stack is None:
            return False
        self.stacks[op.name] = stack
        self.stacked.update({o.name: op.name for o in run[1:]})
        self.steps.append(("stack", op, run))
        return True

    def _plan_stack(self, kind, run, entries):
        """The run's handle, or None where the library does not take it.  A layer that it names as the reason is in no run of
        that kind, and later attempts that meet it are not made: planning ResNet-50 with parameters of each channel's own, an
        attempt at every layer and all of the layers behind it planned for each, took 14 s instead of 0.5."""
        try:
            return B.iconv_plan_stack(entries)
        except B.IconvError as e:
            if e.status != B.ERR_UNSUPPORTED:
                raise
            if e.layer is not None:
                self._refused.add((kind, run[e.layer].name))
            return None

    def _is_merged(self, op) -> bool:
        """Is this one of two merged branches?  Their common plan runs both, so no run of layers may take either."""
        return op.name in self._partner or op.name in self.merged

    def _flow_takes(self, op) -> bool:
        """Is this layer better off in a run of layers (``_try_flow``) than in a launch of its own?  Measured with
        whole networks: always where both channel counts are at least 256 (the stages that run on CTA
        pairs anyway; ResNet-152 at batch 50 1662 -> 1306 us, ResNet-50 at batch 256 1699 -> 1622 with the run
        kernel's first version, 1111 and 1722 under the power limit with the present one); narrower layers
        while they have few pixels: up to 65 536 with 128 channels (batch 64 and 28 x 28: 257 -> 244 us for
        ResNet-18, 1622 -> 1715 for ResNet-50 at batch 256), up to 32 768 with 64 (batch 8 and 56 x 56: 346 -> 333
        us for ResNet-50, 438 -> 451 at batch 32), where the patch and two-layer kernels move fewer bytes."""
        dst = self.net.tensors[op.dst]
        width, pixels = min(op.c_in, op.c_out), self.n * dst.h * dst.w
        return width >= 256 or pixels <= 32768 or (width >= 128 and pixels <= 65536)

    def _try_flow(self, op, fusable, params, kernel) -> bool:
        """Plan the run of layers that starts at `op` as one kernel: 1x1 and k x k layers in any order with
        identity skips and fused projections; False when there is no such run or the library does not
        take it."""
        if kernel not in (B.KERNEL_AUTO, B.KERNEL_UMMA):
            return False
        net, ops = self.net, self.net.ops
        run, absorbed, waiting = [], {}, {}      # absorbed: layer of the run -> its projection; waiting: tensor -> projection, until its consumer comes
        for o in ops[ops.index(op):]:
            if not isinstance(o, Conv) or o.in_dtype != "u8" or o.c_in % 64 or o.c_out % 64 or self._is_merged(o) or o.src == net.input:
                break
            if o.dst in fusable and o.role == "raw":
                waiting[o.dst] = o
                continue
            if o.role != "act" or o.skip == net.input or not self._flow_takes(o) or len(run) == FLOW_MAX_LAYERS:
                break
            if o.name in self.stacks or o.name in self.stacked:
                break           # (tried at a projection that an earlier run passed over: what that run took runs there)
            if o.skip in waiting:
                absorbed[o.name] = waiting.pop(o.skip)
            elif o.skip and o.skip_dtype != "u8":
                break
            if ("flow", o.name) in self._refused:
                return False
            run.append(o)
        if len(run) < 2 or op.dst in waiting:      # (a projection whose consumer is not in the run is planned by itself first)
            return False
        ptr = lambda name: self.tensors[name].data_ptr()
        entries = []
        for o in run:
            kw, entry, p = self._conv_kwargs(o, params, kernel), (ptr(o.src), ptr(o.dst)), params[o.name]
            if o.name in absorbed:
                kw.update(skip_mul=p["skip_mul"], skip_shift=p["skip_shift"], skip_dtype=B.U8, proj=self._proj_kwargs(absorbed[o.name], params))
                entry += (ptr(absorbed[o.name].src),)
            elif o.skip:
                kw.update(skip_mul=p["skip_mul"], skip_shift=p["skip_shift"], skip_dtype=B.U8, skip_c_total=net.tensors[o.skip].c)
                entry += (ptr(o.skip),)
            entries.append((kw,) + entry)
        stack = self._plan_stack("flow", run, entries)
        if stack is None:
            return False
        self.stacks[run[0].name] = stack
        for closer, proj in absorbed.items():
            self.fused[proj.name] = closer
            self.tensors.pop(proj.dst, None)       # the projection's int32 output is never written
        self.stacked.update({o.name: run[0].name for o in run[1:]})
        self.steps.append(("stack", run[0], run))
        return True

    def _proj_kwargs(self, op, params) -> dict:
        """iconv_plan's `proj` argument for the projection `op`."""
        src = self.net.tensors[op.src]
        return dict(weights=self._weights(op, params), bias=gen.bias_i32(self.net.seed, op.layer, op.c_out),
                    h=src.h, w=src.w, c_total=src.c, c_offset=op.in_c_offset, stride=op.stride, pad=op.pad)

    def _chain_partner(self, op, kernel):
        """The layer to run in the same kernel as the closing layer `op`, or None: the next
        operation, a plain 1x1 layer (no skip, 8-bit output) that reads op's whole output."""
        if kernel not in (B.KERNEL_AUTO, B.KERNEL_UMMA) or op.k != 1 or not op.skip or op.skip_dtype != "u8" or op.role != "act":
            return None
        ops = self.net.ops
        i = ops.index(op)
        if i + 1 >= len(ops):
            return None
        nxt = ops[i + 1]
        if not isinstance(nxt, Conv) or nxt.src != op.dst or nxt.k != 1 or nxt.stride != 1 or nxt.skip or nxt.role != "act" or self._is_merged(nxt):
            return None
        if nxt.c_in != op.c_out or nxt.in_c_offset != op.out_c_offset:
            return None
        return nxt

    def _conv_kwargs(self, op, params, kernel) -> dict:
        """iconv_plan's keyword arguments of a plain layer (8-bit output, no skip)."""
        net = self.net
        src, dst = net.tensors[op.src], net.tensors[op.dst]
        p = params[op.name]
        return dict(n=self.n, h=src.h, w=src.w, c_in=op.c_in, c_out=op.c_out, kh=op.k, kw=op.k, stride=op.stride, pad=op.pad,
                    in_dtype=B.DTYPE_CODE[op.in_dtype], in_c_total=src.c, in_c_offset=op.in_c_offset, out_c_total=dst.c,
                    out_c_offset=op.out_c_offset, weights=self._weights(op, params),
                    bias=gen.bias_i32(net.seed, op.layer, op.c_out), kernel=kernel, out_dtype=B.U8, brelu=p["brelu"],
                    mul=p["mul"], shift=p["shift"], h_i=p["h_i"], out_lo=p["out_lo"], out_hi=p["out_hi"], out_zero=p["out_zero"])

    def _alloc_workspace(self):
        """One buffer of the largest workspace any plan asks for: the layers run one after another
        on one stream, so they can share it."""
        size = max([B.iconv_workspace_bytes(p) for p in self.plans.values()] + [0])
        self.workspace = torch.empty((size,), dtype=torch.uint8, device=self.device) if size else None
        self._ws_ptr = self.workspace.data_ptr() if size else None
        for layer in self.tensors.left_out.values():
            layer.repacked = self.workspace
        # the stacks' counters: zero between forwards (each launch leaves them so)
        size = max([B.iconv_stack_sync_bytes(h) for h in self.stacks.values()] + [0])
        self.sync = torch.zeros((size,), dtype=torch.uint8, device=self.device) if size else None
        if size:
            torch.cuda.current_stream(self.device).synchronize()      # a first forward under another stream does not wait for the fill

    def _mergeable(self, a, b, params) -> bool:
        if not (isinstance(a, Conv) and isinstance(b, Conv)):
            return False
        if a.role == "raw" or b.role == "raw" or a.skip or b.skip or a.dst == self.net.output:
            return False
        same = (a.src == b.src and a.dst == b.dst and a.c_in == b.c_in and a.in_c_offset == b.in_c_offset and
                a.in_dtype == b.in_dtype and a.stride == b.stride and b.out_c_offset == a.out_c_offset + a.c_out)
        if not same or (a.k - b.k) % 2 or a.pad - b.pad != (a.k - b.k) // 2:
            return False
        pa, pb = params[a.name], params[b.name]
        return all(pa[k] == pb[k] for k in ("brelu", "out_lo", "out_hi", "out_zero")) and pa["brelu"] == 1 and \
            len(pa["mul"]) == 1 and len(pb["mul"]) == 1

    def _plan_merged(self, a, b, params, kernel):
        """One plan for the sibling branches a and b (see merge_branches)."""
        net = self.net
        src, dst = net.tensors[a.src], net.tensors[a.dst]
        k = max(a.k, b.k)
        W = np.zeros((a.c_out + b.c_out, k, k, a.c_in), dtype=np.int8)
        row = 0
        for op in (a, b):
            o = (k - op.k) // 2
            W[row:row + op.c_out, o:o + op.k, o:o + op.k, :] = self._weights(op, params)
            row += op.c_out
        per = lambda key: np.concatenate([np.repeat(np.asarray(params[op.name][key], dtype=np.int32), op.c_out) for op in (a, b)])
        pa = params[a.name]
        big = a if a.k >= b.k else b
        return B.iconv_plan(n=self.n, h=src.h, w=src.w, c_in=a.c_in, c_out=a.c_out + b.c_out, kh=k, kw=k, stride=a.stride,
                            pad=big.pad, in_dtype=B.DTYPE_CODE[a.in_dtype], in_c_total=src.c, in_c_offset=a.in_c_offset,
                            out_c_total=dst.c, out_c_offset=a.out_c_offset, weights=W,
                            bias=np.concatenate([gen.bias_i32(net.seed, op.layer, op.c_out) for op in (a, b)]),
                            kernel=kernel, out_dtype=B.U8, brelu=1, mul=per("mul"), shift=per("shift"), h_i=per("h_i"),
                            out_lo=pa["out_lo"], out_hi=pa["out_hi"], out_zero=pa["out_zero"])

    def _try_fuse(self, op, fusable, params, kernel) -> bool:
        """Remember a projection op so that its consumer plans it as a fused skip."""
        src = self.net.tensors[op.src]
        if op.in_dtype != "u8" or op.c_in % 16 or src.c % 16 or op.in_c_offset % 16:
            return False
        self._pending[op.dst] = dict(op=op, skip_dtype=B.U8, proj=self._proj_kwargs(op, params))
        return True

    def kernels(self) -> dict:
        out = {k: B.KERNEL_NAME[B.iconv_plan_kernel(p)] for k, p in self.plans.items()}
        out.update({k: "umma" for k in list(self.chains) + list(self.stacks)})
        return out

    def describe(self) -> dict:
        out = {k: B.iconv_plan_describe(p) for k, p in self.plans.items()}
        out.update({k: "umma chain: this layer and %s in one kernel" % [b for b, a in self.chained.items() if a == k][0] for k in self.chains})
        for kind, op, run in self.steps:
            if kind == "stack":
                out[op.name] = "umma stack: %d layers from this one on in one %s" % (len(run), _stack_kernel(run))
        return out

    def conv_macs(self) -> dict:
        """True multiply-accumulates per forward of every convolution (M * N * K)."""
        out = {}
        for op in self.net.convs():
            dst = self.net.tensors[op.dst]
            name = self.fused.get(op.name, op.name)          # a fused projection counts with the layer that runs it
            name = self.merged.get(name, name)               # and so does a merged sibling branch
            name = self.chained.get(name, name)              # and the second layer of a two-layer kernel
            name = self.stacked.get(name, name)              # and the later layers of a stack
            out[name] = out.get(name, 0) + self.n * dst.h * dst.w * op.c_out * op.c_in * op.k * op.k
        return out

    def algorithmic_bytes(self) -> dict:
        """Bytes every executed step must move at least once when the network runs layer at a time:
        its input slice, its output slice, its skip operand and its weights (a fused projection
        adds its own input and weights to the layer that runs it and writes nothing)."""
        esz = {"u8": 1, "i32": 4}
        out = {}
        for op in self.net.ops:
            src, dst = self.net.tensors[op.src], self.net.tensors[op.dst]
            if isinstance(op, (MaxPool, AvgPool)):
                if op.name in self.pooled:                       # its layer's output stays on the chip
                    out[self.pooled[op.name]] += self.n * (dst.h * dst.w * dst.c - src.h * src.w * src.c)
                else:
                    out[op.name] = self.n * (src.h * src.w * src.c + dst.h * dst.w * dst.c)
                continue
            b = self.n * src.h * src.w * op.c_in + op.c_out * op.c_in * op.k * op.k + 4 * op.c_out
            if op.name in self.chained:                      # its input never comes back from memory
                name = self.chained[op.name]
                b += self.n * dst.h * dst.w * op.c_out * esz[dst.dtype] - self.n * src.h * src.w * op.c_in
            elif op.name in self.fused:
                name = self.fused[op.name]
            elif op.name in self.merged:                     # shares its sibling's input read
                name = self.merged[op.name]
                b += self.n * dst.h * dst.w * op.c_out * esz[dst.dtype] - self.n * src.h * src.w * op.c_in
            else:
                name = self.stacked.get(op.name, op.name)
                b += self.n * dst.h * dst.w * op.c_out * esz[dst.dtype]
                if op.skip and op.skip in self.tensors:
                    sk = self.net.tensors[op.skip]
                    b += self.n * sk.h * sk.w * op.c_out * esz[sk.dtype]
            name = self.stacked.get(name, name)
            out[name] = out.get(name, 0) + b
        return out

    def forward(self, x: torch.Tensor = None, marks: list = None) -> torch.Tensor:
        """x: uint8 device tensor [n][h][w][c] (or None to reuse the resident input).
        marks: if a list, receives (op name, event recorded after that op's launch); the
        first entry (None, event) marks the start."""
        ts = torch.cuda.current_stream(self.device)
        stream = ts.cuda_stream
        if x is not None:
            self.tensors[self.net.input] = x
        T = super(_Tensors, self.tensors).__getitem__       # (not a look)
        if marks is not None:
            ev = torch.cuda.Event(enable_timing=True)
            ev.record(ts)
            marks.append((None, ev))
        for kind, op, p in self.steps:
            src = self.net.tensors[op.src]
            if kind == "chain":
                B.iconv_forward_chain(self.chains[op.name], T(op.src).data_ptr(), T(op.skip).data_ptr(), T(op.dst).data_ptr(),
                                      T(p.dst).data_ptr(), stream)
            elif kind == "stack":
                B.iconv_forward_stack(self.stacks[op.name], self.sync.data_ptr(), stream)
            elif kind == "conv":
                skip_name = p if p is not None else op.skip       # a fused projection reads its own input
                B.iconv_forward(self.plans[op.name], T(op.src).data_ptr(),
                                T(skip_name).data_ptr() if skip_name else None, T(op.dst).data_ptr(), self._ws_ptr, stream)
            elif kind == "pool":
                B.iconv_forward(self.plans[op.name], T(op.src).data_ptr(), None, T(p.dst).data_ptr(), self._ws_ptr, stream)
                layer = self.tensors.left_out[op.dst]
                layer.stream = ts
                if layer.looked_at:
                    layer.write(T(op.src).data_ptr(), T(op.dst), stream)
            elif kind == "max":
                B.ipool_max(T(op.src).data_ptr(), T(op.dst).data_ptr(), self.n, src.h, src.w, src.c,
                            op.k, op.stride, op.pad, stream)
            else:
                B.ipool_avg_requant(T(op.src).data_ptr(), T(op.dst).data_ptr(), self.n, src.h, src.w, src.c,
                                    p["mul"], p["shift"], self.net.max_int, stream)
            if marks is not None:
                ev = torch.cuda.Event(enable_timing=True)
                ev.record(ts)
                marks.append((op.name, ev))
        return T(self.net.output)

    def close(self):
        for p in self.plans.values():
            B.iconv_plan_destroy(p)
        for c in self.chains.values():
            B.iconv_chain_destroy(c)
        for s in self.stacks.values():
            B.iconv_stack_destroy(s)
        self.plans, self.chains, self.stacks = {}, {}, {}

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass
