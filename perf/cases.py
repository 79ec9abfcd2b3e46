"""The workloads this repository's speed is measured on.

Each listed case is one call (or one training step, or one network forward)
that a program using the library makes, through the entry points of
paper_2109_03513_gb300: projection of fp32 tensors onto ESB codes, the coded
GEMM and convolutions with their fused epilogues, the quantisation-aware
training step, and a whole network replayed from a CUDA graph.  Shapes are
those of the repository's networks (ResNet18, MobileNetV2, AlexNet's
classifier) and sweeps; draw() spreads the same kinds over odd sizes, small
batches and the other formats.

Codes and integer accumulators are exact, so almost every case is compared
exactly.  exact() gives the fp32 outputs (y, alpha, statistics, gradients)
in 64 bits from plain torch.
"""
from __future__ import annotations

import math

import torch

from paper_2109_03513_gb300 import esb, netrun

DEV = "cuda"
ACTS = {"none": esb.ESB_ACT_NONE, "relu": esb.ESB_ACT_RELU, "relu6": esb.ESB_ACT_RELU6}
# contraction formats: the four of the ResNet18 configuration, and the ternary, power-of-two and (4,1) sets
FORMATS = [(4, 2), (4, 2), (4, 2), (3, 1), (5, 2), (6, 3), (4, 1), (3, 0), (2, 0)]
# formats of the projection sweep
SWEEP = [(b, k) for b in range(3, 7) for k in range(1, b)]


def listed():
    return [
        # one 3x3x64 convolution tile as a GEMM with fp32 results: the smallest call, all latency
        dict(name="gemm_64x64x576", kind="gemm", m=64, n=64, k=576, b=4, kb=2, act="relu", out="y+codes", tiled=False),
        # the first layer of AlexNet's classifier at batch 256 (weights 9216 -> 4096)
        dict(name="fc_256x4096x9216", kind="gemm", m=256, n=4096, k=9216, b=4, kb=2, act="relu", out="codes", tiled=True),
        # a square GEMM of 6-bit codes, whose sums need K in exact chunks
        dict(name="gemm_4096_b6", kind="gemm", m=4096, n=4096, k=4096, b=6, kb=3, act="relu", out="codes", tiled=True),
        # weights or activations of a large model projected with a known scale: the largest tensor of the sweep
        dict(name="project_2p28", kind="project", rows=1, cols=1 << 28, b=4, kb=2, signed=True, dist="normal"),
        # a layer's post-ReLU input calibrated and projected in one call (ResNet18 stage 1, batch 32)
        dict(name="project_dda_56x56x64", kind="project_dda", rows=32 * 56 * 56, cols=64, b=4, kb=2, signed=False, dist="half"),
        # ResNet18 stage 1 at batch 32, the flagship 4-bit convolution
        dict(name="conv3x3_56x64_b4", kind="conv", batch=32, h=56, w=56, c=64, cout=64, r=3, stride=1, pad=1, b=4, kb=2, act="relu", res=False, affine=False),
        # ResNet18 stage 2, second convolution of a block (residual added), 5-bit codes
        dict(name="conv3x3_28x128_res_b5", kind="conv", batch=64, h=28, w=28, c=128, cout=128, r=3, stride=1, pad=1, b=5, kb=2, act="relu", res=True, affine=False),
        # ResNet18 stage 4 entry: stride 2, many channels, few pixels, 6-bit codes
        dict(name="conv3x3s2_14x256_b6", kind="conv", batch=64, h=14, w=14, c=256, cout=512, r=3, stride=2, pad=1, b=6, kb=3, act="relu", res=False, affine=False),
        # ResNet18 stem: 7x7/2 on three-channel images
        dict(name="conv7x7s2_stem_b4", kind="conv", batch=64, h=224, w=224, c=3, cout=64, r=7, stride=2, pad=3, b=4, kb=2, act="relu", res=False, affine=False),
        # MobileNetV2 depthwise layer with folded batch norm (per-channel scale and bias) and ReLU6
        dict(name="dwconv3x3_56x144_b4", kind="dwconv", batch=64, h=56, w=56, c=144, stride=1, b=4, kb=2, act="relu6"),
        # one quantisation-aware training step of a layer input: statistics, moving average, forward, backward
        dict(name="qat_64x28x28x128", kind="qat", rows=64 * 28 * 28, cols=128, b=4, kb=2),
        # MobileNetV2 inference at batch 64, the captured forward pass replayed
        dict(name="mobilenetv2_b64", kind="net", net="mobilenetv2", batch=64, b=4, kb=2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gemm", "gemm", "project", "project_dda", "conv", "conv", "conv", "dwconv", "qat", "net"])
    b, kb = rng.choice(FORMATS)
    if kind == "gemm":
        m, n, k = _log(rng, 1, 4096), _log(rng, 8, 4096), _log(rng, 16, 9216)
        while not _in_range(k, b, kb):
            k = k // 2
        tiled = rng.random() < 0.5
        while m * n * k > (1 << 34 if tiled else 1 << 32):
            m = m // 2
        return dict(kind="gemm", m=m, n=n, k=k, b=b, kb=kb, act=rng.choice(["none", "relu"]),
                    out=rng.choice(["codes", "codes", "y+codes", "acc"]), tiled=tiled)
    if kind == "project":
        b, kb = rng.choice(SWEEP)
        cols = rng.choice([_log(rng, 1, 4096), 64 * rng.randint(1, 64)])
        rows = max(1, _log(rng, 1000, 1 << 26) // cols)
        return dict(kind="project", rows=rows, cols=cols, b=b, kb=kb, signed=rng.random() < 0.6, dist=rng.choice(["normal", "laplace", "half"]))
    if kind == "project_dda":
        b, kb = rng.choice(SWEEP)
        cols = rng.choice([16, 24, 32, 64, 96, 128, 144, 256, 512, 3, 63, 1000])
        rows = max(1, _log(rng, 4000, 1 << 25) // cols)
        return dict(kind="project_dda", rows=rows, cols=cols, b=b, kb=kb, signed=rng.random() < 0.5, dist=rng.choice(["normal", "half"]))
    if kind == "qat":
        cols = rng.choice([64, 96, 128, 256, 512, 77])
        return dict(kind="qat", rows=max(1, _log(rng, 20000, 1 << 24) // cols), cols=cols, b=b, kb=kb)
    if kind == "net":
        net = rng.choice(["mobilenetv2", "resnet18", "alexnet_fc"])
        if net != "mobilenetv2":
            b, kb = rng.choice([(4, 2), (3, 1), (5, 2), (6, 3)])
        else:
            b, kb = 4, 2
        return dict(kind="net", net=net, batch=_log(rng, 1, {"resnet18": 12, "mobilenetv2": 48, "alexnet_fc": 256}[net]), b=b, kb=kb)
    if kind == "dwconv":
        h = rng.choice([7, 14, 28, 56, 112, 19, 33])
        return dict(kind="dwconv", batch=max(1, min(64, _log(rng, 1, 64) * 56 // h)), h=h, w=h + rng.choice([0, 0, 3]), c=rng.choice([32, 96, 144, 192, 384, 50]),
                    stride=rng.choice([1, 1, 2]), b=4, kb=2, act="relu6")
    # convolutions: stage shapes of the networks, with odd sizes beside them
    r, h, c, cout, stride = rng.choice([(3, 56, 64, 64, 1), (3, 28, 128, 128, 1), (3, 14, 256, 256, 1), (3, 7, 512, 512, 1),
                                        (3, 56, 64, 128, 2), (3, 28, 128, 256, 2), (1, 56, 64, 128, 2), (7, 224, 3, 64, 2), (3, 224, 3, 32, 2),
                                        (1, 56, 24, 144, 1), (1, 28, 192, 32, 1), (1, 14, 384, 96, 1), (1, 7, 320, 1280, 1),
                                        (3, 33, 48, 80, 1), (3, 19, 100, 72, 1), (5, 27, 96, 256, 1), (3, 13, 60, 44, 2)])
    res = stride == 1 and rng.random() < 0.4
    return dict(kind="conv", batch=min(64, _log(rng, 1, 64)), h=h, w=h + rng.choice([0, 0, 0, 2]), c=c, cout=cout, r=r, stride=stride, pad=r // 2,
                b=b, kb=kb, act=rng.choice(["relu", "relu", "relu6", "none"]), res=res, affine=rng.random() < 0.3)


# ------------------------------------------------------------------ formats in plain torch

def _fmt_n(b, k):
    return (1 << (b - k - 1)) - 1


def _images(b, k):
    """Integer image of each of the 2^b codes (sign | exponent | fraction)."""
    n = _fmt_n(b, k)
    out = []
    for c in range(1 << b):
        e, f = (c >> k) & n, c & ((1 << k) - 1)
        v = f if e == n else ((1 << k) + f) << e
        out.append(-v if c >> (b - 1) else v)
    return out


def _max_image(b, k):
    return max(_images(b, k))


def _in_range(terms, b, k):
    return terms * _max_image(b, k) ** 2 < 1 << 24


def _decode(codes, cols, b, k):
    """Integer images (rows, cols) float64 of packed code words."""
    cpw = 32 // b
    t = torch.tensor(_images(b, k), dtype=torch.float64, device=codes.device)
    w = codes.to(torch.int64) & 0xFFFFFFFF
    sh = torch.arange(cpw, device=codes.device) * b
    return t[((w[..., None] >> sh) & ((1 << b) - 1)).reshape(codes.shape[0], -1)[:, :cols]]


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _values(shape, dist, g):
    x = torch.randn(shape, generator=g, device=DEV, dtype=torch.float32)
    if dist == "half":
        return x.abs_()
    if dist == "laplace":
        u = torch.rand(shape, generator=g, device=DEV, dtype=torch.float32) - 0.5
        return -torch.sign(u) * torch.log1p(-2.0 * u.abs().clamp_(max=0.4999999))
    return x


def _coded(rows, cols, dist, std, f, g):
    """A projected tensor as a program holds it: packed codes and their scale."""
    x = _values((rows, cols), dist, g) * std
    a, _ = esb.esb_calibrate_dda(x, f)
    a = float(a.item())
    return esb.esb_project(x, f, alpha=a), a


# ------------------------------------------------------------------ cases

def _conv_dims(c):
    p, q = esb.conv_out_hw(c["h"], c["w"], c["r"], c["r"], c["stride"], c["pad"])
    return p, q, c["batch"] * p * q


def prepare(case, seed):
    c, g = case, _gen(seed)
    kind, b, k = c["kind"], c["b"], c["kb"]
    s = dict(case=c)
    if kind in ("gemm", "conv", "dwconv"):
        fu, fs = esb.Fmt(b, k, False), esb.Fmt(b, k, True)
        s.update(fx=fu, fw=fs)
        if kind == "gemm":
            m, n, terms = c["m"], c["n"], c["k"]
            s["X"], ax = _coded(m, terms, "half", 1.0, fu, g)
            s["W"], aw = _coded(n, terms, "normal", math.sqrt(2.0 / terms), fs, g)
        elif kind == "conv":
            _, _, m = _conv_dims(c)
            n, terms = c["cout"], c["r"] * c["r"] * c["c"]
            s["X"], ax = _coded(c["batch"] * c["h"] * c["w"], c["c"], "half", 1.0, fu, g)
            s["W"], aw = _coded(n * c["r"] * c["r"], c["c"], "normal", math.sqrt(2.0 / terms), fs, g)
        else:
            p, q = esb.conv_out_hw(c["h"], c["w"], 3, 3, c["stride"], 1)
            m, n, terms = c["batch"] * p * q, c["c"], 9
            s["X"], ax = _coded(c["batch"] * c["h"] * c["w"], n, "half", 1.0, fu, g)
            s["W"], aw = _coded(9, n, "normal", math.sqrt(2.0 / 9), fs, g)
        act = ACTS[c["act"]]
        fo = esb.Fmt(b, k, c["act"] == "none")
        a_out = 1.3 * esb.esb_alpha_star(b, k)[0]
        ep = dict(scale0=esb.esb_dequant_scale(ax, fu, aw, fs), act=act, alpha_out=a_out, fmt_out=fo)
        if c.get("affine") or kind == "dwconv":
            ep["scale"] = ep["scale0"] * (0.7 + 0.6 * torch.rand(n, generator=g, device=DEV))
            ep["bias"] = 0.2 * torch.randn(n, generator=g, device=DEV)
        if c.get("res"):
            s["R"], ar = _coded(m, n, "half", 1.0, fu, g)
            ep.update(residual=s["R"], res_fmt=fu, res_scale=ar / (1 << k))
        s["ep"] = esb.Epilogue(**ep)
        out = c.get("out", "codes")
        if "codes" in out:
            s["codes"] = torch.empty((m, esb.esb_row_words(n, b)), dtype=torch.int32, device=DEV)
        if "y" in out:
            s["y"] = torch.empty((m, n), dtype=torch.float32, device=DEV)
        if out == "acc":
            s["acc"] = torch.empty((m, n), dtype=torch.int32, device=DEV)
        if c.get("tiled"):
            s["ws"] = torch.empty(max(16, esb.esb_gemm_tiled_workspace_bytes(m, n, terms)), dtype=torch.uint8, device=DEV)
    elif kind == "project":
        s["x"] = _values((c["rows"], c["cols"]), c["dist"], g)
        s["f"] = esb.Fmt(b, k, c["signed"])
        s["alpha"] = esb.esb_alpha_star(b, k)[0]
        s["codes"] = torch.empty((c["rows"], esb.esb_row_words(c["cols"], b)), dtype=torch.int32, device=DEV)
    elif kind == "project_dda":
        s["x"] = _values((c["rows"], c["cols"]), c["dist"], g)
        s["f"] = esb.Fmt(b, k, c["signed"])
        s["codes"] = torch.empty((c["rows"], esb.esb_row_words(c["cols"], b)), dtype=torch.int32, device=DEV)
        s["alpha"] = torch.empty(1, dtype=torch.float32, device=DEV)
        s["stats"] = torch.empty(3, dtype=torch.float64, device=DEV)
        s["ws"] = torch.zeros(max(16, esb.esb_calibrate_dda_workspace_bytes(s["x"].numel())), dtype=torch.uint8, device=DEV)
    elif kind == "qat":
        # activations before normalisation and a gradient of the loss with respect to the quantised ones
        s["x"] = _values((c["rows"], c["cols"]), "normal", g) * 1.7 + 0.3
        s["grad"] = _values((c["rows"], c["cols"]), "normal", g) * 1e-3 + 1e-4
        s["f"] = esb.Fmt(b, k, True)
        s["alpha"] = torch.empty(1, dtype=torch.float32, device=DEV)
        s["stats"] = torch.empty(3, dtype=torch.float64, device=DEV)
        s["run0"] = torch.tensor([0.1, 1.5], dtype=torch.float64, device=DEV)
        s["run"] = s["run0"].clone()
        n = s["x"].numel()
        s["ws"] = torch.zeros(max(16, esb.esb_calibrate_dda_workspace_bytes(n)), dtype=torch.uint8, device=DEV)
        s["bws"] = torch.empty(max(16, int(esb.lib().esb_dn_backward_workspace_bytes(n))), dtype=torch.uint8, device=DEV)
    else:
        fn, (h, w, ch) = netrun.NETWORKS[c["net"]]
        n = c["batch"]
        rn = netrun.Runner(b, k, seed=int(seed) % 1000003, device=DEV)
        rn.begin("calibrate")
        fn(rn, _values((n * h * w, ch), "normal", g), n)
        s["rn"] = rn                                        # weights and buffers the graph reads
        s["x"] = _values((n * h * w, ch), "normal", g)
        st = torch.cuda.Stream()
        st.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(st):
            rn.begin("infer")
            fn(rn, s["x"], n)                               # warm up before the capture
            st.synchronize()
            s["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s["graph"], stream=st):
                rn.begin("infer")
                s["codes"] = fn(rn, s["x"], n).codes
        torch.cuda.current_stream().wait_stream(st)
    return s


def run(state):
    s = state
    c = s["case"]
    kind = c["kind"]
    if kind == "gemm":
        return esb.esb_gemm(s["X"], s["fx"], s["W"], s["fw"], c["k"], ep=s["ep"], want_acc=False, out_acc=s.get("acc"),
                            out_y=s.get("y"), out_codes=s.get("codes"), workspace=s.get("ws"))
    if kind == "conv":
        return esb.esb_conv2d_nhwc(s["X"], s["fx"], s["W"], s["fw"], c["batch"], c["h"], c["w"], c["c"], c["cout"], c["r"], c["r"],
                                   c["stride"], c["pad"], ep=s["ep"], want_acc=False, out_codes=s["codes"])
    if kind == "dwconv":
        return esb.esb_conv2d_nhwc(s["X"], s["fx"], s["W"], s["fw"], c["batch"], c["h"], c["w"], c["c"], c["c"], 3, 3, c["stride"], 1,
                                   groups=c["c"], ep=s["ep"], want_acc=False, out_codes=s["codes"])
    if kind == "project":
        return esb.esb_project(s["x"], s["f"], alpha=s["alpha"], codes=s["codes"], ldc=s["codes"].shape[1])
    if kind == "project_dda":
        codes, alpha = esb.esb_project_dda(s["x"], s["f"], alpha_out=s["alpha"], stats_out=s["stats"], workspace=s["ws"],
                                           codes=s["codes"], ldc=s["codes"].shape[1])
        return dict(codes=codes, alpha=alpha, stats=s["stats"])
    if kind == "qat":
        esb.esb_calibrate_dda(s["x"], s["f"], alpha_out=s["alpha"], stats_out=s["stats"], workspace=s["ws"])
        s["run"].copy_(s["run0"])
        esb.esb_ema_update(s["stats"], s["run"], 0.1)
        codes, xq = esb.esb_dn_project(s["x"], s["stats"], s["f"])
        gx = esb.esb_dn_backward(s["grad"], s["x"], s["stats"], workspace=s["bws"])
        return dict(codes=codes, xq=xq, grad_x=gx, alpha=s["alpha"], stats=s["stats"], running=s["run"])
    s["graph"].replay()
    return s["codes"]


# ------------------------------------------------------------------ what a pass cannot do without

def _code_bytes(rows, cols, b):
    return rows * cols * b / 8.0


def _net_work(net, n, b):
    """(bytes, flops) of a forward: images and weights in, every layer's codes written once and read once."""
    tot = [0.0, 0.0]

    def conv(h, c, cout, r, stride, groups=1, res=False):
        o = (h + stride - 1) // stride
        terms = r * r * c // groups
        tot[1] += 2.0 * n * o * o * cout * terms
        tot[0] += (n * o * o * cout * (2 + (1 if res else 0)) + cout * terms) * b / 8.0
        return o

    if net == "alexnet_fc":
        tot[0] += n * 9216 * (4 + b / 8.0)
        for i, o in ((9216, 4096), (4096, 4096), (4096, 1000)):
            conv(1, i, o, 1, 1)
        return tot
    tot[0] += n * 224 * 224 * 3 * (4 + b / 8.0)
    if net == "resnet18":
        h = conv(224, 3, 64, 7, 2)
        h, c = h // 2, 64
        tot[0] += n * h * h * c * b / 8.0
        for co, st in ((64, 1), (64, 1), (128, 2), (128, 1), (256, 2), (256, 1), (512, 2), (512, 1)):
            o = conv(h, c, co, 3, st)
            if st == 2:
                conv(h, c, co, 1, 2)
            conv(o, co, co, 3, 1, res=True)
            h, c = o, co
        conv(1, 512, 1000, 1, 1)
        return tot
    h = conv(224, 3, 32, 3, 2)
    c = 32
    for t, co, reps, st in netrun.MBV2:
        for i in range(reps):
            e, st1 = c * t, st if i == 0 else 1
            if t > 1:
                conv(h, c, e, 1, 1)
            h = conv(h, e, e, 3, st1, groups=e)
            conv(h, e, co, 1, 1, res=st1 == 1 and c == co)
            c = co
    conv(h, 320, 1280, 1, 1)
    conv(1, 1280, 1000, 1, 1)
    return tot


def work(case):
    c = case
    kind, b = c["kind"], c["b"]
    if kind == "gemm":
        m, n, k = c["m"], c["n"], c["k"]
        out = {"codes": b / 8.0, "y+codes": 4 + b / 8.0, "acc": 4.0}[c["out"]]
        return dict(bytes=_code_bytes(m + n, k, b) + m * n * out, flops=2.0 * m * n * k)
    if kind == "conv":
        _, _, m = _conv_dims(c)
        terms = c["r"] * c["r"] * c["c"]
        return dict(bytes=_code_bytes(c["batch"] * c["h"] * c["w"], c["c"], b) + _code_bytes(c["cout"], terms, b) +
                    _code_bytes(m, c["cout"], b) * (2 if c["res"] else 1), flops=2.0 * m * c["cout"] * terms)
    if kind == "dwconv":
        p, q = esb.conv_out_hw(c["h"], c["w"], 3, 3, c["stride"], 1)
        m = c["batch"] * p * q
        return dict(bytes=_code_bytes(c["batch"] * c["h"] * c["w"] + m + 9, c["c"], b) + 8.0 * c["c"], flops=18.0 * m * c["c"])
    if kind in ("project", "project_dda"):
        n = c["rows"] * c["cols"]
        return dict(bytes=n * (4 + b / 8.0), flops=0.0)
    if kind == "qat":
        n = c["rows"] * c["cols"]
        return dict(bytes=n * (4 + 4 + 4 + 4 + b / 8.0), flops=0.0)   # x and grad in; codes, xq and grad_x out
    by, fl = _net_work(c["net"], c["batch"], b)
    return dict(bytes=by, flops=fl)


def tolerance(case):
    kind = case["kind"]
    if kind == "project_dda":
        # alpha and the statistics within the library's stated 1e-6; an alpha one ulp away moves the few
        # values that lie between the two sets of thresholds (about 1e-7 of them, several to a word)
        return dict(rel=1e-6, max=1e-6, differ=1e-5)
    if kind == "qat":
        # a mean or sigma one ulp of fp32 away moves x_hat by 1e-7 relative: gradients accordingly, and a few
        # values across a threshold by one set element (xq: at most 3 apart of rms 1, 1e-6 of them)
        return dict(rel=2e-5, max=0.9, differ=1e-5)
    # integer sums are exact and the epilogue's operation order is fixed
    return "exact"


# ------------------------------------------------------------------ 64-bit results

def _alpha_star64(b, k):
    """First local minimum on [1e-4, 4] of the expected squared projection error of N(0,1) data."""
    q = sorted({v / float(1 << k) for v in _images(b, k) if v >= 0})

    def slope(a):                                           # dD/dalpha over the non-negative half
        cdf = lambda t: 0.5 * math.erfc(-t / math.sqrt(2.0))
        pdf = lambda t: math.exp(-0.5 * t * t) / math.sqrt(2.0 * math.pi)
        tot = 0.0
        for i, v in enumerate(q):
            lo = 0.0 if i == 0 else 0.5 * a * (q[i - 1] + v)
            hi = math.inf if i == len(q) - 1 else 0.5 * a * (v + q[i + 1])
            p1, c1 = (0.0, 1.0) if hi == math.inf else (pdf(hi), cdf(hi))
            tot += v * (a * v * (c1 - cdf(lo)) - (pdf(lo) - p1))
        return tot

    grid = [1e-4 * (4e4 ** (i / 4000.0)) for i in range(4001)]
    lo = grid[0]
    for hi in grid[1:]:
        if slope(lo) < 0.0 <= slope(hi):
            for _ in range(100):
                mid = 0.5 * (lo + hi)
                lo, hi = (mid, hi) if slope(mid) < 0.0 else (lo, mid)
            return 0.5 * (lo + hi)
        lo = hi
    return lo


def _stats64(x, signed):
    d = x.to(torch.float64)
    mean = d.mean()
    spread = ((d - mean).square().mean() if signed else d.square().mean()).sqrt()
    return mean, spread


def exact(case, seed):
    c = case
    kind, b, k = c["kind"], c["b"], c["kb"]
    if kind == "gemm":
        if "y" not in c["out"]:
            return None                                     # whole numbers only
        s = prepare(case, seed)
        e = s["ep"]
        y = _decode(s["X"], c["k"], b, k) @ _decode(s["W"], c["k"], b, k).T * e.scale0 + e.bias0
        return None, (y.clamp_min(0) if c["act"] == "relu" else y), None
    if kind == "project_dda":
        s = prepare(case, seed)
        mean, spread = _stats64(s["x"], c["signed"])
        n = torch.tensor(float(s["x"].numel()), dtype=torch.float64, device=DEV)
        return dict(codes=None, alpha=(_alpha_star64(b, k) * (spread + 1e-7)).reshape(1), stats=torch.stack([mean, spread, n]))
    if kind == "qat":
        s = prepare(case, seed)
        a = _alpha_star64(b, k)
        mean, sigma = _stats64(s["x"], True)
        d = s["x"].to(torch.float64) - mean
        q = torch.tensor(sorted({v / float(1 << k) for v in _images(b, k) if v >= 0}), dtype=torch.float64, device=DEV)
        t = d / (sigma + 1e-7) / a
        xq = a * torch.sign(t) * q[torch.bucketize(t.abs(), 0.5 * (q[1:] + q[:-1]), right=True)]
        gr = s["grad"].to(torch.float64)
        sc = sigma + 1e-7
        gx = (gr - gr.mean()) / sc - d * (gr * d).mean() / (sigma * sc * sc)
        st = torch.stack([mean, sigma])
        n = torch.tensor(float(d.numel()), dtype=torch.float64, device=DEV)
        return dict(codes=None, xq=xq, grad_x=gx, alpha=(a * sc).reshape(1), stats=torch.stack([mean, sigma, n]),
                    running=0.9 * s["run0"] + 0.1 * st)
    return None                                             # packed codes: whole numbers
