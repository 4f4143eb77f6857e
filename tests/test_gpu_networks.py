"""GPU parity of whole networks: every layer of small instances of the five
configurations against the oracle, bit for bit."""
import numpy as np
import pytest
import torch

from oracle import networks as ON
from paper_2006_11735_b200 import binding as B
from paper_2006_11735_b200.network import Network
from workloads import networks as N
from workloads.networks import Conv, MaxPool, Net

pytestmark = pytest.mark.gpu

SMALL = [
    N.single_conv(),
    N.vdsr(n=2, h=40, w=48),
    N.vrcnn(n=2, h=40, w=56),
    N.resnet50(n=2, h=64, w=64),
    N.resnet152(n=1, h=64, w=64),
    N.resnet18(n=2, h=64, w=64),
]


@pytest.mark.parametrize("net", SMALL, ids=lambda n: n.name)
@pytest.mark.parametrize("kernel,fuse", [(B.KERNEL_DIRECT, False), (B.KERNEL_AUTO, False), (B.KERNEL_AUTO, True)],
                         ids=["direct", "auto", "auto-fused"])
def test_every_layer_of_small_networks_matches_oracle(net, kernel, fuse):
    params = ON.calibrate(net)
    x = ON.net_input(net)
    want = ON.forward(net, params, x)
    g = Network(net, params, kernel=kernel, fuse_projection=fuse, merge_branches=fuse)
    out = g.forward(torch.from_numpy(x).cuda())
    B.iconv_check(torch.cuda.current_stream().cuda_stream)
    if fuse and net.name.startswith("resnet"):
        # one projection per stage (per strided or widening stage of the basic-block network), each
        # absorbed by its block's closing layer
        assert len(g.fused) == (3 if net.name == "resnet18" else 4)
    if net.name.startswith("vrcnn"):      # both variable-filter-size blocks run as one layer each
        assert len(g.merged) == (2 if fuse else 0) and len(g.plans) == (4 if fuse else 6)
    for op in net.ops:
        if op.name in g.fused:            # its int32 tensor never exists; the absorbing layer's output is checked
            continue
        got = g.tensors[op.dst].cpu().numpy()
        assert np.array_equal(got, want[op.dst]), "%s: %d mismatches" % (op.name, (got != want[op.dst]).sum())
    assert np.array_equal(out.cpu().numpy(), want[net.output])
    g.close()


def test_smoke_entry_point_runs():
    """The smoke entry point (one small invocation checked against the oracle) stays runnable."""
    import __graft_entry__
    __graft_entry__.smoke()


def _pooled(n=3, h=61, w=75, seed=3):
    """A first layer, the max-pool behind it and one more layer: the network that pools in the layer's kernel, the one that does not,
    and batches of images."""
    net = Net("t", seed, n, "x", "out")
    net.add_tensor("x", h, w, 3)
    net.add_tensor("stem", (h - 1) // 2 + 1, (w - 1) // 2 + 1, 64)
    ho, wo = (net.tensors["stem"].h - 1) // 2 + 1, (net.tensors["stem"].w - 1) // 2 + 1
    net.add_tensor("pool", ho, wo, 64)
    net.add_tensor("out", ho, wo, 64)
    net.ops.extend([Conv("stem", 0, "x", "stem", 3, 64, 7, 2, 3, in_dtype="u8_raw128"), MaxPool("maxpool", "stem", "pool"),
                    Conv("c1", 1, "pool", "out", 64, 64, 1)])
    params = {op.name: dict(delta=0.01, mul=[11983], shift=[16], h_i=[1395], brelu=1, out_lo=0, out_hi=255, out_zero=0) for op in net.ops}
    a, b = Network(net, params), Network(net, params, fuse_pool=False)
    assert a.pooled == {"maxpool": "stem"} and b.pooled == {} and [s[0] for s in b.steps] == ["conv", "max", "conv"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return a, b, [torch.randint(0, 256, (n, h, w, 3), dtype=torch.uint8, device="cuda", generator=gen) for _ in range(4)]


@pytest.mark.parametrize("n, h, w", [(3, 61, 75), (1, 64, 66), (2, 33, 68), (2, 40, 80), (1, 7, 6), (1, 1, 1)])
def test_the_first_layers_tensor_is_the_last_forwards(n, h, w):
    """It is left out of the forwards until somebody looks at it, and has to hold what they would have written: before the first forward,
    after one whose images are no longer there, and after more of them for somebody who has kept it."""
    a, b, x = _pooled(n, h, w)
    for q in x:                                      # (never looked at: the outputs alone)
        assert torch.equal(a.forward(q), b.forward(q))
    b.forward(x[0])
    q = x[0].clone()
    a.forward(q)
    q.fill_(7)
    held = a.tensors["stem"]
    assert torch.equal(held, b.tensors["stem"]) and (h == 1 or held.float().std() > 10)
    assert a.tensors["stem"] is held and a.tensors.get("stem") is held and dict(a.tensors)["stem"] is held
    for q in x[1:]:
        assert torch.equal(a.forward(q), b.forward(q)) and torch.equal(held, b.tensors["stem"])
    a.close()
    assert torch.equal(a.tensors["stem"], b.tensors["stem"])
    b.close()
    fresh = _pooled(n, h, w)[0]
    assert not fresh.tensors["stem"].any()


def test_the_first_layers_tensor_and_captured_forwards():
    """A graph from before the first look does not write the tensor, one from after it does; a look may be part of a graph."""
    a, b, x = _pooled()
    static = x[0].clone()
    a.forward(static)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        a.forward(static)
    for q in x:
        static.copy_(q)
        g.replay()
        b.forward(q)
        assert torch.equal(a.tensors["stem"], b.tensors["stem"])
    c, looks = _pooled()[0], torch.cuda.CUDAGraph()
    c.forward(static)
    with torch.cuda.graph(looks):
        c.forward(static)
        seen = c.tensors["stem"].clone()
        c.forward(static)
    for q in x:
        static.copy_(q)
        looks.replay()
        b.forward(q)
        assert torch.equal(seen, b.tensors["stem"]) and torch.equal(c.tensors["stem"], b.tensors["stem"])
    del g, looks


def test_a_look_at_the_first_layers_tensor_waits_for_the_forward():
    """The forward runs under another stream than the one that looks."""
    a, b, x = _pooled(16, 200, 200)
    s = torch.cuda.Stream()
    for q in x:
        b.forward(q)
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            torch.cuda._sleep(2_000_000)
            a.forward(q)
        assert torch.equal(a.tensors["stem"], b.tensors["stem"])
    B.iconv_check(s.cuda_stream)
