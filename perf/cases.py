"""Performance cases: the work a user of the library has it do, from the smallest call to the largest.

Four kinds.  "net": one forward of a network (``Network.forward``), the ResNets for classification, the
VDSR and VRCNN shapes for pictures.  "layer": one convolution through ``iconv_plan`` / ``iconv_forward``.
"add": the stand-alone feature-map addition (``iadd_requant``).  "calib": the n-sigma bound of an int32
feature map (``iq_sigma_bound``), the step a calibration run repeats for every layer.

All outputs are whole numbers and have to be the same bit for bit.
"""
import math

import numpy as np
import torch

from paper_2006_11735_b200 import binding as B
from paper_2006_11735_b200.network import Network, load_params
from workloads import networks

DEVICE = "cuda:0"
RESNETS = ("resnet18", "resnet50", "resnet152")


def _net(name, model, n, h, w):
    return {"name": name, "kind": "net", "model": model, "n": n, "h": h, "w": w}


def listed():
    return [
        # bulk classification: the batch the throughput benchmark runs
        _net("resnet50_b256", "resnet50", 256, 224, 224),
        # one image at a time, as a latency-bound service asks: about fifty small launches
        _net("resnet50_b1", "resnet50", 1, 224, 224),
        # the deep network at the batch the paper times it with (its Table 2)
        _net("resnet152_b50", "resnet152", 50, 224, 224),
        # a few images of an odd size: no tile, row or batch divides evenly
        _net("resnet18_b7_odd", "resnet18", 7, 231, 315),
        # super-resolution of a batch of patches: twenty equal 3x3 layers
        _net("vdsr_16x256x256", "vdsr", 16, 256, 256),
        # ... and of one small picture of odd size
        _net("vdsr_1x481x321", "vdsr", 1, 481, 321),
        # the in-loop filter on one large picture (the size of the paper's Table 6)
        _net("vrcnn_1x1600x2560", "vrcnn", 1, 1600, 2560),
        # ... and on a small one
        _net("vrcnn_1x240x416", "vrcnn", 1, 240, 416),
        # the smallest call: one 3x3 layer on one small feature map
        {"name": "conv_1x32x32x64", "kind": "layer", "n": 1, "h": 32, "w": 32, "c_in": 64, "c_out": 64, "k": 3, "stride": 1,
         "dtype": "u8", "per_channel": False, "skip": False},
        # a strided layer with batch normalisation folded in (a multiplier, shift and bound for every channel), 7-bit
        # activations held in int8 as the paper's own networks have them, ragged in every direction
        {"name": "conv_24x57x57x128s2_bn", "kind": "layer", "n": 24, "h": 57, "w": 57, "c_in": 128, "c_out": 256, "k": 3, "stride": 2,
         "dtype": "s8", "per_channel": True, "skip": False},
        # adding two feature maps of different ratios outside a convolution, at an element count that is odd
        {"name": "add_51m", "kind": "add", "elems": 64 * 56 * 56 * 256 + 5},
        # calibrating one layer of a batch of 64: the bound of its int32 outputs
        {"name": "calib_51m", "kind": "calib", "elems": 64 * 56 * 56 * 256},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.random()
    if kind < 0.40:
        model = rng.choice(RESNETS)
        h, w = rng.randint(160, 320), rng.randint(160, 320)
        top = {"resnet18": 256, "resnet50": 256, "resnet152": 64}[model] * 224 * 224 // (h * w)
        return {"kind": "net", "model": model, "n": _log_int(rng, 1, max(1, min(256, top))), "h": h, "w": w}
    if kind < 0.70:
        model = rng.choice(("vdsr", "vrcnn"))
        h, w = _log_int(rng, 128, 1600), _log_int(rng, 128, 2560)
        top = {"vdsr": 1500000, "vrcnn": 4200000}[model]
        h = min(h, top // w)
        n = _log_int(rng, 1, max(1, min(16, top // (h * w))))
        return {"kind": "net", "model": model, "n": n, "h": h, "w": w}
    if kind < 0.88:
        k, stride = rng.choice((1, 3, 3, 5)), rng.choice((1, 1, 2))
        c_in, c_out = rng.choice((32, 48, 64, 128, 256, 512)), rng.choice((32, 48, 64, 128, 256, 512))
        h, w = _log_int(rng, 7, 112), _log_int(rng, 7, 112)
        top = min(200000, int(2e11) // (c_in * c_out * k * k)) // (h * w)
        n = _log_int(rng, 1, max(1, min(64, top)))
        s8 = rng.random() < 0.3
        return {"kind": "layer", "n": n, "h": h, "w": w, "c_in": c_in, "c_out": c_out, "k": k, "stride": stride,
                "dtype": "s8" if s8 else "u8", "per_channel": rng.random() < 0.4, "skip": k != 5 and stride == 1 and rng.random() < 0.4}
    return {"kind": "add" if kind < 0.94 else "calib", "elems": _log_int(rng, 200000, 64 * 56 * 56 * 256)}


# ---------------------------------------------------------------- inputs

def _images(gen, n, h, w, c):
    """Low-passed noise of standard deviation 40 around 128 with a few flat patches: uint8 NHWC pictures."""
    x = torch.randn((n, c, h, w), generator=gen, device=DEVICE)
    for _ in range(3):
        x = torch.nn.functional.avg_pool2d(x, 9, stride=1, padding=4, count_include_pad=False)
    x = x / x.std(dim=(2, 3), keepdim=True) * 40.0 + 128.0
    for _ in range(8):
        y0, y1 = sorted(torch.randint(0, h + 1, (2,), generator=gen, device=DEVICE).tolist())
        x0, x1 = sorted(torch.randint(0, w + 1, (2,), generator=gen, device=DEVICE).tolist())
        x[:, :, y0:y1, x0:x1] += 40.0
    return x.round_().clamp_(0, 255).to(torch.uint8).permute(0, 2, 3, 1).contiguous()


def _activations(gen, shape, top):
    """What a bounded ReLU leaves: half zeros, the rest a half-normal that rarely reaches the bound."""
    return (torch.randn(shape, generator=gen, device=DEVICE) * (top / 3.0)).round_().clamp_(0, top)


class _Layer:
    """A planned convolution with its tensors."""

    def __init__(self, case, gen, rng):
        n, h, w, c_in, c_out, k, stride = (case[q] for q in ("n", "h", "w", "c_in", "c_out", "k", "stride"))
        signed, pad = case["dtype"] == "s8", k // 2
        top, code = (127, B.S8) if signed else (255, B.U8)
        kind = torch.int8 if signed else torch.uint8
        ho, wo = (h + 2 * pad - k) // stride + 1, (w + 2 * pad - k) // stride + 1
        w_f = rng.normal(0.0, 0.05, size=(c_out, k, k, c_in)).astype(np.float32)
        W = B.iq_quantize_weights(w_f, B.iq_weight_delta(w_f))
        # three standard deviations of Y is where the bound lies (the n-sigma rule); with batch normalisation folded in,
        # every channel has its own
        sigma = math.sqrt(c_in * k * k) * float(W.astype(np.float32).std()) * top / 3.0 / math.sqrt(2.0)
        bounds = 3.0 * sigma * (rng.uniform(0.7, 1.4, size=c_out) if case["per_channel"] else np.ones(1))
        q = [B.iq_brelu_params(float(b), 1.0, top) for b in bounds]
        kw = {}
        self.skip = None
        if case["skip"]:
            s = B.iq_skip_sync(float(bounds[0]) / (2.0 * top), 1.0)
            kw = dict(skip_dtype=code, skip_c_total=c_out, skip_mul=s["skip_mul"], skip_shift=s["skip_shift"])
            self.skip = _activations(gen, (n, ho, wo, c_out), top).to(kind)
        self.plan = B.iconv_plan(n=n, h=h, w=w, c_in=c_in, c_out=c_out, kh=k, kw=k, stride=stride, pad=pad, in_dtype=code, out_dtype=code,
                                 out_hi=top, weights=W, bias=rng.integers(-4096, 4097, size=c_out, dtype=np.int32),
                                 mul=[p["mul"] for p in q], shift=[p["shift"] for p in q], h_i=[p["h_i"] for p in q], **kw)
        self.x = _activations(gen, (n, h, w, c_in), top).to(kind)
        self.out = torch.empty((n, ho, wo, c_out), dtype=kind, device=DEVICE)

    def __del__(self):
        try:
            B.iconv_plan_destroy(self.plan)
        except Exception:       # planning failed, or the interpreter is going
            pass


def _spec(case):
    return networks.by_name(case["model"], n=case["n"], h=case["h"], w=case["w"])


def prepare(case, seed):
    gen = torch.Generator(device=DEVICE).manual_seed(int(seed))
    if case["kind"] == "net":
        net = _spec(case)
        params = dict(load_params(case["model"]))
        if "avgpool" in params:                 # the average over this picture size's last feature map
            last = net.tensors[next(op.src for op in net.ops if op.name == "avgpool")]
            params["avgpool"] = dict(params["avgpool"], mul=(65536 * 2 + last.h * last.w) // (2 * last.h * last.w), shift=16)
        t = net.tensors[net.input]
        return {"net": Network(net, params, device=DEVICE), "x": _images(gen, case["n"], t.h, t.w, t.c)}
    if case["kind"] == "layer":
        return {"layer": _Layer(case, gen, np.random.default_rng(int(seed)))}
    n = case["elems"]
    if case["kind"] == "add":
        # Y = A + B rescaled to A's ratio, then the bounded ReLU and Eq. 4, as behind two branches of different ratios
        s = B.iq_skip_sync(500.0, 333.0)
        q = B.iq_brelu_params(600.0, 1.0, 255)
        return {"a": _activations(gen, (n,), 255).to(torch.uint8), "b": _activations(gen, (n,), 255).to(torch.uint8),
                "out": torch.empty((n,), dtype=torch.uint8, device=DEVICE),
                "desc": dict(n_elems=n, a_dtype=B.U8, b_dtype=B.U8, out_dtype=B.U8, a_zero=0, b_zero=0, mul_a=1, sh_a=0,
                             mul_b=s["skip_mul"], sh_b=s["skip_shift"], brelu=1, h_i=q["h_i"], mul=q["mul"], shift=q["shift"],
                             out_zero=0, out_lo=0, out_hi=255)}
    y = torch.randn((n,), generator=gen, device=DEVICE).mul_(90000.0).sub_(2000.0).round_().to(torch.int32)
    return {"y": y}


# ---------------------------------------------------------------- one pass

def run(state):
    if "net" in state:
        return state["net"].forward(state["x"])
    stream = torch.cuda.current_stream().cuda_stream
    if "layer" in state:
        q = state["layer"]
        B.iconv_forward(q.plan, q.x.data_ptr(), None if q.skip is None else q.skip.data_ptr(), q.out.data_ptr(), None, stream)
        return q.out
    if "desc" in state:
        B.iadd_requant(state["a"].data_ptr(), state["b"].data_ptr(), state["out"].data_ptr(), stream, **state["desc"])
        return state["out"]
    return B.iq_sigma_bound(state["y"].data_ptr(), state["y"].numel(), 0.0015, stream)


def work(case):
    if case["kind"] == "net":
        # the picture in, the result out, every weight and bias once: what lies between could stay on the chip
        net = _spec(case)
        n, tin, tout = case["n"], net.tensors[net.input], net.tensors[net.output]
        size = n * (tin.h * tin.w * tin.c + tout.h * tout.w * tout.c * (4 if tout.dtype == "i32" else 1))
        macs = 0
        for op in net.convs():
            dst = net.tensors[op.dst]
            size += op.c_out * op.c_in * op.k * op.k + 4 * op.c_out
            macs += n * dst.h * dst.w * op.c_out * op.c_in * op.k * op.k
        return {"bytes": size, "flops": 2 * macs}
    if case["kind"] == "layer":
        n, h, w, c_in, c_out, k, stride = (case[q] for q in ("n", "h", "w", "c_in", "c_out", "k", "stride"))
        ho, wo = (h + 2 * (k // 2) - k) // stride + 1, (w + 2 * (k // 2) - k) // stride + 1
        outs = n * ho * wo * c_out
        return {"bytes": n * h * w * c_in + outs * (2 if case["skip"] else 1) + c_out * (c_in * k * k + 4), "flops": 2 * outs * c_in * k * k}
    if case["kind"] == "add":
        return {"bytes": 3 * case["elems"], "flops": 6 * case["elems"]}
    return {"bytes": 4 * case["elems"], "flops": case["elems"]}


def tolerance(case):
    return "exact"          # integers throughout
