"""What a ``Network`` plans and launches, without a GPU: the library's calls are stood in for by recorders that take
every run of layers, and every operation of the network has to reach exactly one launch."""
import contextlib
import itertools

import numpy as np
import pytest
import torch

from paper_2006_11735_b200 import binding as B
from paper_2006_11735_b200 import network as NW
from workloads.networks import Conv, MaxPool, Net


class Recorder:
    """Takes every plan; a forward notes the channel slices it writes and the projections it computes."""

    def __init__(self):
        self.written, self.projections = [], []

    def plan(self, **kw):
        return [kw]

    def plan_stack(self, entries):
        return [(kw, out) for kw, _, out, *_ in entries]

    def _launch(self, kw, out):
        o = kw.get("out_c_offset", 0)
        self.written.append((out, o, o + kw["c_out"]))
        if kw.get("proj"):
            self.projections.append(kw["proj"]["weights"].tobytes())

    def forward(self, plan, x, skip, out, ws, stream=0):
        self._launch(plan[0], out)

    def forward_stack(self, stack, sync, stream=0):
        for kw, out in stack:
            self._launch(kw, out)


@pytest.fixture
def recorder(monkeypatch):
    r = Recorder()

    def refuse(*a):
        raise B.IconvError(B.ERR_UNSUPPORTED, "not here")
    for name, f in dict(iconv_plan=r.plan, iconv_plan_stack=r.plan_stack, iconv_plan_chain=refuse, iconv_forward=r.forward,
                        iconv_forward_stack=r.forward_stack, iconv_workspace_bytes=lambda p: 0, iconv_stack_sync_bytes=lambda s: 64,
                        iconv_plan_destroy=lambda p: None, iconv_stack_destroy=lambda s: None).items():
        monkeypatch.setattr(NW.B, name, f)
    stream = type("Stream", (), dict(cuda_stream=0, synchronize=lambda self: None))()
    monkeypatch.setattr(torch.cuda, "set_device", lambda d: None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda d=None: stream)
    return r


def _covered(net, g, r):
    """Every operation's output slice is written once; a fused projection's weights are in one launch instead."""
    g.forward()
    for op in net.convs():
        if op.name in g.fused:
            assert r.projections.count(g._proj_kwargs(op, PARAMS[id(net)])["weights"].tobytes()) == 1, op.name
            continue
        ptr = g.tensors[op.dst].data_ptr()
        hits = [w for w in r.written if w[0] == ptr and w[1] <= op.out_c_offset and op.out_c_offset + op.c_out <= w[2]]
        assert len(hits) == 1, (op.name, hits)


PARAMS = {}


def _network(net, changes={}, **kw):
    params = {op.name: dict(dict(delta=0.01, mul=[200], shift=[16], h_i=[83558], brelu=1, out_lo=0, out_hi=255, out_zero=0, skip_mul=100,
                                 skip_shift=8), **changes.get(op.name, {})) for op in net.ops}
    PARAMS[id(net)] = params
    return NW.Network(net, params, device="cpu", **kw)


def _net(h, w, tensors, ops, n=1):
    net = Net("t", 3, n, "x", ops[-1].dst)
    net.add_tensor("x", h, w, 64)
    for name, c, dtype in tensors:
        net.add_tensor(name, h, w, c, dtype)
    net.ops.extend(ops)
    return net


@pytest.mark.parametrize("k", [1, 3], ids=["run_of_any_layers", "run_of_equal_layers"])
def test_both_of_two_merged_branches_run_behind_a_run_of_layers(recorder, k):
    net = _net(8, 8, [("t0", 64, "u8"), ("t1", 64, "u8"), ("cat", 128, "u8"), ("out", 64, "u8")],
               [Conv("c0", 0, "x", "t0", 64, 64, 3, 1, 1), Conv("c1", 1, "t0", "t1", 64, 64, k, 1, k // 2),
                Conv("a", 2, "t1", "cat", 64, 64, k, 1, k // 2), Conv("b", 3, "t1", "cat", 64, 64, 4 - k, 1, (4 - k) // 2, out_c_offset=64),
                Conv("c2", 4, "cat", "out", 128, 64, 1)])
    g = _network(net)
    assert g.merged == {"b": "a"}
    _covered(net, g, recorder)


def test_a_projection_ahead_of_a_run_that_ends_before_its_consumer_is_not_lost(recorder, monkeypatch):
    """The projection stands first in its block, the layer it closes is left out of the run."""
    monkeypatch.setattr(NW.Network, "_flow_takes", lambda self, op: op.name in ("c1", "c2"))
    net = _net(8, 8, [("t0", 128, "u8"), ("s", 64, "i32"), ("t1", 128, "u8"), ("t2", 128, "u8"), ("out", 64, "u8")],
               [Conv("c0", 0, "x", "t0", 64, 128, 1), Conv("proj", 1, "t0", "s", 128, 64, 1, role="raw"), Conv("c1", 2, "t0", "t1", 128, 128, 1),
                Conv("c2", 3, "t1", "t2", 128, 128, 1), Conv("c3", 4, "t2", "out", 128, 64, 1, skip="s", skip_dtype="i32")])
    g = _network(net)
    assert list(g.stacks) == ["c1"] and g.fused == {"proj": "c3"}
    _covered(net, g, recorder)


def test_layers_of_a_run_that_is_full_are_not_taken_again(recorder, monkeypatch):
    """A run ends at the longest the library takes, between a projection and its consumer."""
    monkeypatch.setattr(NW, "FLOW_MAX_LAYERS", 3)
    monkeypatch.setattr(NW.Network, "_flow_takes", lambda self, op: True)
    t = [("t%d" % i, 64, "u8") for i in range(5)]
    net = _net(8, 8, t + [("s", 64, "i32"), ("out", 64, "u8")],
               [Conv("c0", 0, "x", "t0", 64, 64, 1), Conv("c1", 1, "t0", "t1", 64, 64, 1), Conv("proj", 2, "t1", "s", 64, 64, 1, role="raw"),
                Conv("c2", 3, "t1", "t2", 64, 64, 3, 1, 1), Conv("c3", 4, "t2", "t3", 64, 64, 1), Conv("c4", 5, "t3", "t4", 64, 64, 1, skip="s", skip_dtype="i32"),
                Conv("c5", 6, "t4", "out", 64, 64, 1)])
    g = _network(net)
    _covered(net, g, recorder)
    assert [s[1].name for s in g.steps] == ["c0", "c1", "c4", "c5"]


def test_both_of_two_merged_branches_run_behind_a_closing_layer(recorder, monkeypatch):
    monkeypatch.setattr(NW.B, "iconv_plan_chain", lambda a, b: pytest.fail("the first branch was chained by itself"))
    net = _net(8, 8, [("t0", 64, "u8"), ("t1", 64, "u8"), ("cat", 128, "u8"), ("out", 64, "u8")],
               [Conv("c0", 0, "x", "t0", 64, 64, 1), Conv("c1", 1, "t0", "t1", 64, 64, 1, skip="t0", skip_dtype="u8"),
                Conv("a", 2, "t1", "cat", 64, 64, 1), Conv("b", 3, "t1", "cat", 64, 64, 3, 1, 1, out_c_offset=64),
                Conv("c2", 4, "cat", "out", 128, 64, 1)])
    g = _network(net)
    assert g.merged == {"b": "a"}
    _covered(net, g, recorder)


def test_the_counters_are_zero_before_the_constructor_returns(recorder, monkeypatch):
    """The first forward may be under another stream than the one that fills them."""
    done = []
    zeros, stream = torch.zeros, torch.cuda.current_stream()
    monkeypatch.setattr(torch, "zeros", lambda *a, **kw: (done.append("fill"), zeros(*a, **kw))[1])
    monkeypatch.setattr(type(stream), "synchronize", lambda self: done.append("wait"))
    monkeypatch.setattr(NW.Network, "_flow_takes", lambda self, op: True)
    g = _network(_net(8, 8, [("t0", 64, "u8"), ("t1", 64, "u8"), ("t2", 64, "u8")],
                      [Conv("c0", 0, "x", "t0", 64, 64, 1), Conv("c1", 1, "t0", "t1", 64, 64, 1), Conv("c2", 2, "t1", "t2", 64, 64, 1)]))
    assert g.stacks and g.sync is not None and done[-2:] == ["fill", "wait"]


@pytest.mark.parametrize("equal", [False, True], ids=["run_of_any_layers", "run_of_equal_layers"])
def test_a_run_that_is_refused_for_one_layer_is_not_tried_at_every_layer(recorder, monkeypatch, equal):
    """Planning stays linear: few attempts at the run, and every layer's weights are made once."""
    depth, tried, quantised = 30, [], []

    def refuse_late(entries):
        tried.append(len(entries))
        late = [i for i, e in enumerate(entries) if e[0]["out_zero"]]
        if late:
            raise B.IconvError(B.ERR_UNSUPPORTED, "iconv_plan_stack: layer %d: a zero point" % late[0])
        return recorder.plan_stack(entries)
    quantise = NW.B.iq_quantize_weights
    monkeypatch.setattr(NW.B, "iconv_plan_stack", refuse_late)
    monkeypatch.setattr(NW.B, "iq_quantize_weights", lambda w, d: (quantised.append(0), quantise(w, d))[1])
    k = 3 if equal else 1
    ops = [Conv("c%d" % i, i, "t%d" % (i - 1) if i else "x", "t%d" % i, 64, 64, k, 1, k // 2) for i in range(depth)]
    zero = {"c%d" % (depth - 4): dict(out_zero=3)}
    g = _network(_net(8, 8, [("t%d" % i, 64, "u8") for i in range(depth)], ops), zero)
    assert len(tried) <= 4 and len(quantised) == depth, (tried, len(quantised))
    assert [len(s[2]) for s in g.steps if s[0] == "stack"] == [3]               # what stands behind that layer is a run as before
    _covered(g.net, g, recorder)


def test_the_kernel_of_every_step_is_named(recorder, monkeypatch):
    """What the benchmark calls a step's kernel is the one that the library runs it in."""
    from bench import kernel_of
    monkeypatch.setattr(NW.B, "iconv_plan_describe", lambda p: "umma window(strips) block_n=64")
    tensors = [("t%d" % i, 64, "u8") for i in range(6)]
    convs = lambda k: [Conv("c%d" % i, i, "t%d" % (i - 1) if i else "x", "t%d" % i, 64, 64, k if i % 3 else 1, 1, k // 2 if i % 3 else 0) for i in range(6)]
    for k, want in ((3, "umma_stack_kernel"), (1, "umma_flow_kernel")):
        monkeypatch.setattr(NW.Network, "_flow_takes", lambda self, op: k == 1)
        g = _network(_net(8, 8, tensors, convs(k)))
        names = {s[1].name: kernel_of(g.describe()[s[1].name], "umma") for s in g.steps}
        assert {names[s[1].name] for s in g.steps if s[0] == "stack"} == {want}
        assert names["c0"] == "umma_window_kernel"
    for text, want in (("umma window(rolling) block_n=48", "umma_roll_kernel"), ("umma im2col(cta pairs) block_n=256", "umma_conv_kernel (cta pairs)"),
                       ("umma chain: this layer and c2 in one kernel", "umma_chain_kernel"), ("umma im2col block_n=64", "umma_conv_kernel"),
                       ("stem(in place) -> umma block_n=64", "picture_kernel"),
                       ("stem and max-pool -> umma block_n=64", "stem_repack_kernel + stem_pool_kernel"), ("stem -> umma block_n=64", "stem_repack_kernel + umma_window_kernel")):
        assert kernel_of(text, "stem" if text.startswith("stem") else "umma") == want
    assert kernel_of("", "avgpool") == "avgpool"


def _pooled_net(extra=(), pool=MaxPool("maxpool", "stem", "pool"), between=(), output="out"):
    net = Net("t", 3, 2, "x", output)
    net.add_tensor("x", 20, 24, 3)
    net.add_tensor("stem", 10, 12, 64)
    net.add_tensor("pool", (10 + 2 * pool.pad - pool.k) // pool.stride + 1, (12 + 2 * pool.pad - pool.k) // pool.stride + 1, 64)
    net.add_tensor("out", net.tensors["pool"].h, net.tensors["pool"].w, 64)
    net.add_tensor("more", 10, 12, 64)
    net.ops.extend([Conv("stem", 0, "x", "stem", 3, 64, 7, 2, 3, in_dtype="u8_raw128"), *between, pool, Conv("c1", 1, "pool", "out", 64, 64, 1), *extra])
    return net


@pytest.fixture
def pooling(recorder, monkeypatch):
    """The library takes a first layer and its max-pool; launches of the max-pool alone are noted."""
    pools = []
    monkeypatch.setattr(NW.B, "iconv_plan_stem_pool", lambda **kw: recorder.plan(**kw))
    monkeypatch.setattr(NW.B, "ipool_max", lambda x, out, *a: pools.append((x, out)))
    monkeypatch.setattr(torch.cuda, "stream", lambda s: contextlib.nullcontext())
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: False)
    monkeypatch.setattr(NW._LeftOut, "images", lambda self, out: torch.zeros(1))
    return pools


def test_a_first_layer_and_its_max_pool_are_one_launch_and_all_tensors_are_there(recorder, pooling):
    net = _pooled_net()
    g = _network(net)
    assert g.pooled == {"maxpool": "stem"} and [s[0] for s in g.steps] == ["pool", "conv"]
    g.forward()
    at = {name: dict.__getitem__(g.tensors, name).data_ptr() for name in net.tensors}
    assert [w[0] for w in recorder.written] == [at["pool"], at["out"]] and not pooling
    assert list(g.tensors) == list(net.tensors) == [name for name, _ in g.tensors.items()] and len(g.tensors) == len(net.tensors) and "stem" in g.tensors
    recorder.written.clear()
    stem = g.tensors["stem"]
    assert [w[0] for w in recorder.written] == [at["stem"]]                     # (the look, in order with the forward before it)
    ways = [g.tensors.get("stem"), dict(g.tensors.items())["stem"], dict(g.tensors)["stem"], {**g.tensors}["stem"], g.tensors.copy()["stem"],
            list(g.tensors.values())[list(net.tensors).index("stem")]]
    assert all(t is stem for t in ways) and tuple(stem.shape) == (2, 10, 12, 64) and g.tensors.get("nothing", 5) == 5
    with pytest.raises(KeyError):
        g.tensors["nothing"]
    recorder.written.clear()
    g.forward()
    assert sorted(w[0] for w in recorder.written) == sorted([at["pool"], at["stem"], at["out"]])


@pytest.mark.parametrize("net", [
    _pooled_net(extra=[Conv("c2", 2, "stem", "more", 64, 64, 1)]),                                                    # a second reader
    _pooled_net(extra=[Conv("c2", 2, "stem", "more", 64, 64, 1, skip="stem", skip_dtype="u8")]),
    _pooled_net(between=[Conv("c0", 2, "x", "more", 3, 64, 7, 2, 3, in_dtype="u8_raw128")]),                          # the pool is not the next operation
    _pooled_net(pool=MaxPool("maxpool", "stem", "pool", 2, 2, 0)), _pooled_net(pool=MaxPool("maxpool", "stem", "pool", 3, 1, 1)),
    _pooled_net(output="stem")], ids=["reader", "skip", "order", "pool_2x2", "pool_stride_1", "output"])
def test_first_layers_whose_output_is_needed_are_launched_by_themselves(recorder, pooling, net):
    g = _network(net)
    assert not g.pooled and not g.tensors.left_out
    _covered(net, g, recorder)
    assert len(pooling) == 1


@pytest.mark.parametrize("n, h, w, one", [(256, 224, 224, True), (1, 224, 224, True), (50, 224, 224, True), (7, 231, 315, True), (2, 1080, 1920, True), (16, 64, 64, True),
                                          (1, 32, 32, True), (256, 160, 160, True), (256, 64, 64, False), (128, 64, 64, False), (256, 32, 32, False),
                                          (1, 1600, 16, False), (256, 1600, 16, False)])
def test_a_first_layer_takes_its_max_pool_where_that_is_faster(recorder, pooling, n, h, w, one):
    net = _pooled_net()
    g = _network(net)
    t = net.tensors["stem"]
    g.n, t.h, t.w = n, (h + 1) // 2, (w + 1) // 2
    assert g._pool_takes(net.ops[0]) == g._try_pool(net.ops[0], PARAMS[id(net)], B.KERNEL_AUTO) == one


def test_a_max_pool_is_run_by_itself_on_request_or_where_the_library_refuses(recorder, pooling, monkeypatch):
    net = _pooled_net()
    for kw in (dict(fuse_pool=False), dict(kernel=B.KERNEL_DIRECT)):
        assert [s[0] for s in _network(net, **kw).steps] == ["conv", "max", "conv"]

    def fail(status):
        def f(**kw):
            raise B.IconvError(status, "not here")
        return f
    monkeypatch.setattr(NW.B, "iconv_plan_stem_pool", fail(B.ERR_UNSUPPORTED))
    assert [s[0] for s in _network(net).steps] == ["conv", "max", "conv"]
    monkeypatch.setattr(NW.B, "iconv_plan_stem_pool", fail(B.ERR_ARG))
    with pytest.raises(B.IconvError):
        _network(net)


@pytest.mark.parametrize("h, w", [(1, 1), (7, 6), (20, 24), (21, 26), (9, 31), (5, 33)])
@pytest.mark.parametrize("in_dtype", [B.U8, B.U8_RAW128])
def test_the_images_are_found_again_in_the_repacked_ones(h, w, in_dtype):
    n, ho, wo = 2, (h - 1) // 2 + 1, (w - 1) // 2 + 1
    pitch = (wo + 3 + 2 + 3) // 4 * 4
    x = np.random.default_rng(w).integers(0, 256, size=(n, h, w, 3), dtype=np.uint8)
    T = np.zeros((n, ho + 3, pitch, 16), dtype=np.uint8)
    for Y, X, dy, dx in itertools.product(range(ho + 3), range(pitch), range(2), range(2)):
        r, c = 2 * (Y - 2) + dy, 2 * (X - 4) + dx
        if 0 <= r < h and 0 <= c < w:
            T[:, Y, (X & 1) * (pitch // 2) + X // 2, (dy * 2 + dx) * 3:(dy * 2 + dx) * 3 + 3] = x[:, r, c] ^ (128 if in_dtype == B.U8_RAW128 else 0)
    layer = NW._LeftOut.__new__(NW._LeftOut)
    layer.kw, layer.plan, layer.repacked = dict(h=h, w=w, in_dtype=in_dtype), None, torch.from_numpy(np.concatenate([T.ravel(), np.full(4096, 9, np.uint8)]))
    assert np.array_equal(layer.images(torch.empty(n, ho, wo, 64)).numpy(), x)
