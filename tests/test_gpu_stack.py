"""Consecutive layers of one geometry in one kernel (``iconv_plan_stack``): every layer's output against
the oracle where it is affordable, against the layers launched one by one (which other tests tie to the
oracle) where there are more tiles than CTAs, and the refusals."""
import numpy as np
import pytest
import torch

from oracle import networks as ON
from paper_2006_11735_b200 import binding as B
from paper_2006_11735_b200.network import Network, load_params
from workloads import generators as gen
from workloads import networks as N

pytestmark = pytest.mark.gpu


def _check():
    B.iconv_check(torch.cuda.current_stream().cuda_stream)


@pytest.mark.parametrize("shape", [(1, 16, 16), (2, 23, 19), (1, 40, 131)], ids=lambda s: "x".join(map(str, s)))
def test_stacked_layers_match_oracle(shape):
    """One tile or a few: every tile waits for its whole neighbourhood, fewer CTAs than SMs."""
    n, h, w = shape
    net = N.vdsr(n=n, h=h, w=w, depth=6)
    params = ON.calibrate(net)
    x = ON.net_input(net)
    want = ON.forward(net, params, x)
    g = Network(net, params)
    assert list(g.stacks) == ["conv2"] and len(g.stacked) == 3, g.describe()
    for _ in range(2):                  # the second forward finds the counters the first one left
        g.forward(torch.from_numpy(x).cuda())
        _check()
        for op in net.ops:
            assert np.array_equal(g.tensors[op.dst].cpu().numpy(), want[op.dst]), op.name
    assert int(g.sync.sum()) == 0
    g.close()


@pytest.mark.parametrize("shape", [(1, 148 * 16, 8), (1, 149 * 16, 8), (3, 150, 271), (5, 129, 257)], ids=lambda s: "x".join(map(str, s)))
def test_stacked_layers_equal_single_launches(shape):
    """As many tiles as SMs, one more, and several waves with a remainder, across image borders."""
    n, h, w = shape
    net = N.vdsr(n=n, h=h, w=w)
    params = load_params("vdsr")
    a, b = Network(net, params), Network(net, params, stack_layers=False)
    assert len(a.stacked) == 17 and not b.stacks
    for k in range(2):
        x = torch.from_numpy(gen.uniform_u8(k, (n, h, w, 1))).cuda()
        a.forward(x)
        _check()
        b.forward(x)
        for op in net.ops:
            assert torch.equal(a.tensors[op.dst], b.tensors[op.dst]), op.name
    a.close()
    b.close()


@pytest.mark.parametrize("name,n,h,w", [("vdsr", 1, 97, 321), ("resnet18", 1, 96, 96), ("resnet50", 3, 64, 96)])
def test_many_forwards_of_one_network_stay_equal(name, n, h, w):
    """Layers of few tiles, where the waits between the CTAs are on the path of every tile: hundreds of forwards
    back to back, all of them equal to the layers launched one by one."""
    net, params = N.by_name(name, n=n, h=h, w=w), dict(load_params(name))
    if "avgpool" in params:
        last = net.tensors[next(op.src for op in net.ops if op.name == "avgpool")]
        params["avgpool"] = dict(params["avgpool"], mul=65536 // (last.h * last.w), shift=16)
    a, b = Network(net, params), Network(net, params, stack_layers=False)
    assert a.stacks and not b.stacks
    x = torch.from_numpy(gen.uniform_u8(1, (n, h, w, net.tensors[net.input].c))).cuda()
    b.forward(x)
    different = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(300):
        for op in net.ops:
            if op.name in a.stacked and op.dst in a.tensors:
                a.tensors[op.dst].zero_()        # a tile read too early is then seen
        a.forward(x)
        different += (a.tensors[net.output] != b.tensors[net.output]).sum()
    _check()
    assert int(different) == 0 and int(a.sync.sum()) == 0
    a.close()
    b.close()


def test_two_networks_on_two_streams():
    """Launches that take the whole GPU, from two streams at a time and with other kernels between them."""
    nets = [N.by_name("vdsr", n=1, h=97, w=321), N.by_name("resnet18", n=1, h=96, w=96)]
    params = [load_params("vdsr"), dict(load_params("resnet18"), avgpool=dict(load_params("resnet18")["avgpool"], mul=65536 // 9, shift=16))]
    gs = [Network(net, p) for net, p in zip(nets, params)]
    xs = [torch.from_numpy(gen.uniform_u8(1, (1, net.tensors[net.input].h, net.tensors[net.input].w, net.tensors[net.input].c))).cuda() for net in nets]
    want = [g.forward(x).clone() for g, x in zip(gs, xs)]
    _check()
    streams, different = [torch.cuda.Stream() for _ in gs], [torch.zeros((), dtype=torch.int64, device="cuda") for _ in gs]
    torch.cuda.synchronize()
    for _ in range(100):
        for g, x, s, d, w in zip(gs, xs, streams, different, want):
            with torch.cuda.stream(s):
                d += (g.forward(x) != w).sum()
    torch.cuda.synchronize()
    _check()
    assert [int(d) for d in different] == [0, 0]
    for g in gs:
        g.close()


@pytest.mark.parametrize("name,h,w", [("vdsr", 97, 321), ("resnet18", 96, 96)])
def test_forwards_in_a_captured_graph(name, h, w):
    net, params = N.by_name(name, n=1, h=h, w=w), dict(load_params(name))
    if "avgpool" in params:
        params["avgpool"] = dict(params["avgpool"], mul=65536 // 9, shift=16)
    g = Network(net, params)
    assert g.stacks
    x = torch.from_numpy(gen.uniform_u8(1, (1, h, w, net.tensors[net.input].c))).cuda()
    want = g.forward(x).clone()
    _check()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(3):
            out = g.forward(x)
    for op in net.ops:
        if op.dst in g.tensors:
            g.tensors[op.dst].zero_()
    for _ in range(20):
        graph.replay()
    _check()
    assert torch.equal(out, want) and int(g.sync.sum()) == 0
    del graph
    g.close()


def test_an_empty_batch():
    """A rank without images."""
    net = N.vdsr(n=1, h=40, w=56)
    g = Network(net, load_params("vdsr"), n=0)
    assert not g.stacks
    assert tuple(g.forward(torch.zeros((0, 40, 56, 1), dtype=torch.uint8, device="cuda")).shape) == (0, 40, 56, 1)
    _check()
    g.close()


@pytest.fixture
def part_of_the_gpu():
    """A stream that has 32 SMs of the GPU to itself."""
    driver = pytest.importorskip("cuda.bindings.driver")

    def ok(r):
        assert int(r[0]) == 0, r[0]
        return r[1] if len(r) == 2 else r[1:]
    torch.zeros(1, device="cuda")
    device = ok(driver.cuDeviceGet(0))
    sms = ok(driver.cuDeviceGetDevResource(device, driver.CUdevResourceType.CU_DEV_RESOURCE_TYPE_SM))
    groups, _, _ = ok(driver.cuDevSmResourceSplitByCount(1, sms, 0, 32))
    ctx = ok(driver.cuGreenCtxCreate(ok(driver.cuDevResourceGenerateDesc(groups, 1)), device, driver.CUgreenCtxCreate_flags.CU_GREEN_CTX_DEFAULT_STREAM))
    stream = ok(driver.cuGreenCtxStreamCreate(ctx, driver.CUstream_flags.CU_STREAM_NON_BLOCKING, 0))
    yield torch.cuda.ExternalStream(int(stream))
    torch.cuda.synchronize()
    driver.cuStreamDestroy(stream)
    driver.cuGreenCtxDestroy(ctx)


@pytest.mark.parametrize("name,n,h,w", [("vdsr", 1, 97, 321), ("resnet18", 2, 96, 96)])
def test_where_the_launch_is_refused_the_layers_run_one_after_another(name, n, h, w, part_of_the_gpu):
    """On a part of a GPU that does not hold all CTAs, by the library itself; and by the test hook on all of it."""
    net, params = N.by_name(name, n=n, h=h, w=w), dict(load_params(name))
    if "avgpool" in params:
        params["avgpool"] = dict(params["avgpool"], mul=65536 // 9, shift=16)
    a, b = Network(net, params), Network(net, params, stack_layers=False)
    x = torch.from_numpy(gen.uniform_u8(1, (n, h, w, net.tensors[net.input].c))).cuda()
    b.forward(x)
    _check()
    with torch.cuda.stream(part_of_the_gpu):
        a.forward(x)
        _check()
    assert "not all of its CTAs" in B.iconv_last_error()
    assert torch.equal(a.tensors[net.output], b.tensors[net.output])
    for first, stack in a.stacks.items():
        run = next(s[2] for s in a.steps if s[0] == "stack" and s[1].name == first)
        for op in run:
            a.tensors[op.dst].zero_()
        B.iconv_selftest_stack_apart(stack, torch.cuda.current_stream().cuda_stream)
        _check()
        for op in run:
            assert torch.equal(a.tensors[op.dst], b.tensors[op.dst]), op.name
    assert int(a.sync.sum()) == 0
    a.close()
    b.close()


def test_stack_refuses_what_it_cannot_take():
    x, y, z = (torch.zeros((1, 32, 32, 64), dtype=torch.uint8, device="cuda") for _ in range(3))
    kw = dict(n=1, h=32, w=32, c_in=64, c_out=64, kh=3, kw=3, pad=1, weights=np.ones((64, 3, 3, 64), np.int8), bias=np.zeros(64, np.int32),
              mul=[200], shift=[16], h_i=[83558])
    p = [t.data_ptr() for t in (x, y, z)]
    B.iconv_stack_destroy(B.iconv_plan_stack([(kw, p[0], p[1]), (kw, p[1], p[2])]))
    for bad in ([(kw, p[0], p[1])],                                              # one layer
                [(kw, p[0], p[1]), (kw, p[1], p[0])],                            # the second would overwrite the first one's input
                [(kw, p[0], p[1]), (kw, p[0], p[1])],                            # two layers into one tensor
                [(kw, p[0], p[1]), (dict(kw, shift=[33]), p[1], p[2])],          # a shift beyond 32 bits
                [(kw, p[0], p[1]), (dict(kw, skip_dtype=B.U8, skip_c_total=64), p[1], p[2])]):
        with pytest.raises(B.IconvError) as e:
            B.iconv_plan_stack(bad)
        assert e.value.status == B.ERR_UNSUPPORTED


def test_first_forward_under_another_stream_than_the_constructor(monkeypatch):
    """The constructor's stream has work queued when the counters are filled."""
    net = N.vdsr(n=1, h=40, w=131, depth=6)
    params = ON.calibrate(net)
    x = ON.net_input(net)
    want = ON.forward(net, params, x)
    xd, side = torch.from_numpy(x).cuda(), torch.cuda.Stream()
    busy = torch.ones((1 << 28,), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    alloc = Network._alloc_workspace

    def queue_then_alloc(self):                 # (planning's blocking copies have gone before)
        for _ in range(100):
            busy.mul_(1.0)
        alloc(self)
    monkeypatch.setattr(Network, "_alloc_workspace", queue_then_alloc)
    g = Network(net, params)
    assert g.stacks
    with torch.cuda.stream(side):
        out = g.forward(xd)
        _check()
    assert np.array_equal(out.cpu().numpy(), want[net.output])
    g.close()


# ---- runs of different layers

@pytest.fixture
def flow_everywhere(monkeypatch):
    monkeypatch.setattr(Network, "_flow_takes", lambda self, op: True)


def test_run_of_layers_that_begins_with_a_projection(monkeypatch):
    """The layer before a block's projection runs apart; the projection and the layer it closes are in the run."""
    monkeypatch.setattr(Network, "_flow_takes", lambda self, op: op.name not in ("s1b0_3x3a", "s1b0_3x3b", "s2b0_3x3a"))
    net = N.resnet_basic(2, (1, 2), h=48, w=40, widths=(64, 128), classes=16)
    params = ON.calibrate(net)
    x = ON.net_input(net)
    want = ON.forward(net, params, x)
    g = Network(net, params)
    assert list(g.stacks) == ["s2b0_3x3b"] and g.fused == {"s2b0_proj": "s2b0_3x3b"}
    g.forward(torch.from_numpy(x).cuda())
    _check()
    for op in net.ops:
        if op.name not in g.fused:
            assert np.array_equal(g.tensors[op.dst].cpu().numpy(), want[op.dst]), op.name
    g.close()


@pytest.mark.parametrize("build", [lambda: N.resnet(1, (2, 2), h=40, w=56, widths=(64, 128), classes=16),
                                   lambda: N.resnet(3, (1, 2, 1), h=72, w=61, widths=(64, 64, 128), classes=16),
                                   lambda: N.resnet_basic(2, (2, 2, 1), h=51, w=64, widths=(64, 128, 256), classes=16)],
                         ids=["bottleneck", "bottleneck_ragged", "basic"])
def test_run_of_layers_matches_oracle(build, flow_everywhere):
    """Bottleneck and basic blocks, identity skips and fused projections, strides, units that are partly
    or, for the second CTA of a pair, wholly outside the tensor."""
    net = build()
    params = ON.calibrate(net)
    x = ON.net_input(net)
    want = ON.forward(net, params, x)
    g = Network(net, params)
    assert len(g.stacks) == 1 and sum(len(s[2]) for s in g.steps if s[0] == "stack") >= 5, g.describe()
    for _ in range(2):                  # the second forward finds the counters the first one left
        out = g.forward(torch.from_numpy(x).cuda())
        _check()
        for op in net.ops:
            if op.name not in g.fused:
                assert np.array_equal(g.tensors[op.dst].cpu().numpy(), want[op.dst]), op.name
        assert np.array_equal(out.cpu().numpy(), want[net.output])
    assert int(g.sync.sum()) == 0
    g.close()


@pytest.mark.parametrize("name,n,h,w", [("resnet50", 1, 224, 224), ("resnet50", 19, 97, 130), ("resnet18", 33, 131, 224), ("resnet50", 96, 160, 160)])
def test_run_of_layers_equals_single_launches(name, n, h, w, flow_everywhere):
    """Every tile width (32 columns at one image, 256 at many), less than a wave of tiles and many, as one launch
    of 16 or 48 layers against the layers launched one by one, which other tests tie to the oracle."""
    net = N.by_name(name, n=n, h=h, w=w)
    params = dict(load_params(name))
    last = net.tensors[next(op.src for op in net.ops if op.name == "avgpool")]
    params["avgpool"] = dict(params["avgpool"], mul=65536 // (last.h * last.w), shift=16)
    a, b = Network(net, params), Network(net, params, stack_layers=False, fuse_chain=False)
    assert len(a.stacks) == 1 and not b.stacks
    for k in range(2):
        x = torch.from_numpy(gen.uniform_u8(k, (n, h, w, 3))).cuda()
        a.forward(x)
        _check()
        b.forward(x)
        for op in net.ops:
            if op.name not in a.fused:
                assert torch.equal(a.tensors[op.dst], b.tensors[op.dst]), op.name
    a.close()
    b.close()


def test_run_of_layers_refuses_what_it_cannot_take():
    x, y, z = (torch.zeros((1, 16, 16, 128), dtype=torch.uint8, device="cuda") for _ in range(3))
    kw = dict(n=1, h=16, w=16, c_in=128, c_out=128, kh=1, kw=1, weights=np.ones((128, 1, 1, 128), np.int8), bias=np.zeros(128, np.int32),
              mul=[200], shift=[16], h_i=[83558])
    p = [t.data_ptr() for t in (x, y, z)]
    half = dict(kw, c_in=64, in_c_total=128, weights=np.ones((128, 1, 1, 64), np.int8))
    B.iconv_stack_destroy(B.iconv_plan_stack([(kw, p[0], p[1]), (kw, p[1], p[2])]))
    for bad in ([(kw, p[0], p[1]), (half, p[1], p[2])],                          # reads half of another layer's output
                [(kw, p[0], p[1]), (kw, p[1], p[0])],                            # overwrites a tensor the run has read
                [(kw, p[0], p[1]), (dict(kw, out_zero=3), p[1], p[2])],          # a zero point
                [(kw, p[0], p[1]), (dict(kw, mul=[200] * 128, shift=[16] * 128, h_i=[83558] * 128), p[1], p[2])],
                [(kw, p[0], p[1]), (dict(kw, skip_dtype=B.U8, skip_c_total=128, skip_shift=8), p[1], p[2])]):     # a skip without its tensor
        with pytest.raises(B.IconvError) as e:
            B.iconv_plan_stack(bad)
        assert e.value.status == B.ERR_UNSUPPORTED
