"""What a user of this library runs, as cases that can be timed and compared.

Each case is one call sequence of a user's program through the public binding
(paper_2003_04296_gb300.minw): a quantized layer on bit-planes or on level
codes, the quantizer passes of a training layer, a training step, or the
forward of a whole network.  A case is a dict of plain values; its "kind"
names the sequence.  Sizes come from the library's configurations (the CIFAR
ConvNet and its narrower models, the ResNet-18-shaped network, the weight-only
networks, the 256 x 512 x 14 x 14 sweep), draw() spreads over the ranges they
stand for.

`work` counts what a sequence cannot do without: each input read once, each
output written once (packed operands at their packed size), 2 flops per
multiply-add of its products.
"""
import numpy as np
import torch
import torch.nn.functional as F

from paper_2003_04296_gb300 import inputs, minw

ALPHA, LR = 0.75, 1e-3


def listed():
    return [
        # the smallest call: one 1-bit layer of a small batch, quantized and convolved on
        # bit-planes, raw accumulators and the scaled output (latency)
        dict(name="planes_conv_small", kind="planes_conv", B=4, C=128, H=32, W=32, O=128, k=3, stride=1, pad=1,
             ba=1, bw=1),
        # the widest operands on the sweep's layer: 3-bit x 3-bit as implicit GEMM (largest)
        dict(name="planes_conv_sweep", kind="planes_conv", B=256, C=512, H=14, W=14, O=512, k=3, stride=1, pad=1,
             ba=3, bw=3),
        # a block of a low-bit network on bit-planes, pooled and repacked, with ragged batch and
        # channels (96 in, 200 out)
        dict(name="planes_block_ragged", kind="planes_block", B=37, C=96, H=32, W=32, O=200, k=3, stride=1, pad=1,
             ba=2, bw=1, bo=2, pool=1),
        # a residual block's second convolution on FP4 level codes (ResNet-18, second stage)
        dict(name="codes_block_resid", kind="codes_block", B=128, C=128, H=28, W=28, O=128, k=3, stride=1, pad=1,
             ba=3, bw=3, bo=3, pool=0, fp4=1, res=1),
        # the quantizer passes of a training layer: AQE forward with packing and mask, its
        # backward from the mask, and the latent weights' forward and backward
        dict(name="aqe_train", kind="aqe", B=256, C=512, H=14, W=14, n=512 * 512 * 9, bits=2, bw=3),
        # Algorithm 1 on a fully connected layer (fc1 of the CIFAR ConvNet).  Training cases take 3-bit
        # activations: a 1-bit output whose sign flips with the order of a sum is off by its whole size,
        # which no tolerance tells from a wrong answer
        dict(name="fc_train", kind="fc_train", B=256, K=8192, O=1024, ba=3, bw=1),
        # Algorithm 1 on a convolutional layer (conv4 of the CIFAR ConvNet)
        dict(name="conv_train", kind="conv_train", B=256, C=256, H=16, W=16, O=256, k=3, stride=1, pad=1, ba=3, bw=1),
        # inference of the CIFAR ConvNet at the batch it is quoted on
        dict(name="convnet_b256", kind="convnet", model="A", B=256, ba=1, bw=1),
        # the same family serving a few images at a time (latency of a forward)
        dict(name="convnet_b8", kind="convnet", model="B", B=8, ba=2, bw=2),
        # inference of the ResNet-18-shaped network on ImageNet-sized images
        dict(name="resnet18_b128", kind="resnet18", B=128, hw=224, ba=3, bw=3),
        # inference of the weight-only networks
        dict(name="wresnet110_b128", kind="wresnet", n=18, B=128, bw=3),
        dict(name="wdense100_b128", kind="wdense", layers=16, growth=12, B=128, bw=3),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["planes_conv", "planes_conv", "planes_block", "codes_block", "aqe", "fc_train", "conv_train",
                       "convnet", "resnet18", "wresnet", "wdense"])
    if kind in ("planes_conv", "planes_block", "codes_block"):
        while True:
            k = rng.choice([1, 3, 3, 3])
            c = dict(kind=kind, B=_log(rng, 1, 256), C=32 * _log(rng, 1, 16), H=rng.randint(7, 56), W=0,
                     O=_log(rng, 10, 512), k=k, stride=rng.choice([1, 1, 1, 2]), pad=k // 2,
                     ba=rng.randint(1, 3), bw=rng.randint(1, 3))
            c["W"] = c["H"] if rng.random() < 0.6 else rng.randint(7, 56)
            if kind != "planes_conv":
                c["bo"] = rng.randint(1, 3)
                c["pool"] = rng.choice([0, 0, 1])
                if c["pool"]:
                    c["H"] = c["W"] = rng.choice([8, 16, 32])
                    c["stride"] = 1
            if kind == "codes_block":
                c["fp4"] = rng.randint(0, 1)
                c["C"] = 128 * rng.randint(1, 4) if c["fp4"] else 64 * rng.randint(1, 8)
                c["O"] = 32 * _log(rng, 2, 16)
                c["res"] = 0 if c["pool"] else rng.randint(0, 1)
            ho, wo = _out(c)
            if c["B"] * c["C"] * c["H"] * c["W"] <= 25_690_112 and c["B"] * c["O"] * ho * wo <= 25_690_112 and \
                    _macs(c) <= 118_380_000_000:
                return c
    if kind == "aqe":
        while True:
            c = dict(kind=kind, B=_log(rng, 1, 256), C=_log(rng, 3, 512), H=rng.randint(4, 56), W=rng.randint(4, 56),
                     n=_log(rng, 1000, 2_500_000), bits=rng.randint(1, 3), bw=rng.randint(1, 3))
            if c["B"] * c["C"] * c["H"] * c["W"] <= 25_690_112:
                return c
    if kind == "fc_train":
        return dict(kind=kind, B=64 * rng.randint(1, 4), K=64 * _log(rng, 4, 128), O=_log(rng, 10, 1024),
                    ba=3, bw=rng.randint(1, 3))
    if kind == "conv_train":
        while True:
            k = rng.choice([1, 3, 3, 3])
            c = dict(kind=kind, B=32 * rng.randint(1, 8), C=64 * rng.randint(1, 4), H=rng.randint(7, 32), W=0,
                     O=_log(rng, 16, 256), k=k, stride=rng.choice([1, 1, 2]), pad=k // 2, ba=3,
                     bw=rng.randint(1, 3))
            c["W"] = c["H"]
            ho, wo = _out(c)
            if c["B"] * ho * wo % 64 == 0 and c["B"] * c["C"] * c["H"] * c["W"] <= 16_777_216:
                return c
    if kind == "convnet":
        return dict(kind=kind, model=rng.choice("ABCD"), B=_log(rng, 1, 256), ba=rng.randint(1, 3),
                    bw=rng.randint(1, 3))
    if kind == "resnet18":
        return dict(kind=kind, B=_log(rng, 1, 128), hw=32 * rng.randint(2, 7), ba=rng.randint(1, 3),
                    bw=rng.randint(1, 3))
    if kind == "wresnet":
        return dict(kind=kind, n=rng.randint(1, 18), B=_log(rng, 1, 128), bw=rng.randint(1, 3))
    return dict(kind=kind, layers=rng.randint(4, 16), growth=12, B=_log(rng, 1, 128), bw=rng.randint(1, 3))


def _out(c):
    return (c["H"] + 2 * c["pad"] - c["k"]) // c["stride"] + 1, (c["W"] + 2 * c["pad"] - c["k"]) // c["stride"] + 1


def _macs(c):
    ho, wo = _out(c)
    return c["B"] * c["O"] * ho * wo * c["C"] * c["k"] ** 2


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(g, *shape):
    return torch.randn(shape, generator=g, device="cuda")


def _uniform(g, *shape):
    return torch.rand(shape, generator=g, device="cuda") * 2 - 1


def _i32(n):
    return torch.empty(n, dtype=torch.int32, device="cuda")


def _u8(*shape):
    return torch.empty(shape, dtype=torch.uint8, device="cuda")


def _f32(*shape):
    return torch.empty(shape, device="cuda")


_LEVEL_MS = {1: 1.0, 2: 0.6, 3: 0.4}          # rough second moment of the levels of N(0, 1) values


def _layer(c, seed):
    """Activations N(0, 1), latent weights N(0, 0.05) with the per-channel prescale of the
    multi-level quantizers, and a folded BN that spreads the outputs over the levels."""
    g = _gen(seed)
    x = _normal(g, c["B"], c["C"], c["H"], c["W"])
    w = 0.05 * _normal(g, c["O"], c["C"], c["k"], c["k"])
    ws = 1.0 / w.abs().amax(dim=(1, 2, 3)) if c["bw"] > 1 else torch.ones(c["O"], device="cuda")
    unit = (4.0 if c["ba"] == 3 else 1.0) * (4.0 if c["bw"] == 3 else 1.0)
    wms = 1.0 if c["bw"] == 1 else ((w * ws[:, None, None, None]) ** 2).mean(dim=(1, 2, 3)).clamp_min(1e-3)
    sigma = (c["C"] * c["k"] ** 2 * _LEVEL_MS[c["ba"]] * wms) ** 0.5
    scale = (1.0 + 0.1 * _normal(g, c["O"])) / (sigma * unit)
    shift = 0.1 * _normal(g, c["O"])
    if c.get("pool"):
        shift = shift - 1.03
    return x.contiguous(), w.contiguous(), ws.contiguous(), scale.contiguous(), shift.contiguous()


def _quant(bits):
    return minw.quant(bits, inputs.DEFAULT_THR[bits])


def _codes(c, x, q):
    out = _u8(x.shape[0], x.shape[2], x.shape[3], x.shape[1] // (2 if c["fp4"] else 1))
    (minw.aqe_quantize_codes_e2m1 if c["fp4"] else minw.aqe_quantize_codes)(x, q, out)
    return out


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind in ("planes_conv", "planes_block", "codes_block"):
        x, w, ws, scale, shift = _layer(c, seed)
        ho, wo = _out(c)
        s = dict(c=c, x=x, scale=scale, shift=shift, qa=_quant(c["ba"]))
        qw = _quant(c["bw"])
        if kind == "codes_block":
            s["act"] = _codes(c, x, s["qa"])
            div = 2 if c["fp4"] else 1
            s["wgt"] = _u8(c["O"], c["k"], c["k"], c["C"] // div)
            (minw.minw_pack_weight_codes_e2m1 if c["fp4"] else minw.minw_pack_weight_codes)(w, qw, s["wgt"], ws)
            s["qo"] = _quant(c["bo"])
            s["out"] = _u8(c["B"], ho >> c["pool"], wo >> c["pool"], c["O"] // div)
            if c["res"]:
                s["res"] = _codes(c, _normal(_gen(seed + 1000), c["B"], c["O"], ho, wo), s["qo"])
            return s
        s["act"] = _i32(minw.packed_words(c["B"], c["C"], c["H"], c["W"], c["ba"]))
        s["wgt"] = _i32(minw.packed_words(c["O"], c["C"], c["k"], c["k"], c["bw"]))
        minw.minw_pack_weights(w, qw, s["wgt"], ws)
        if kind == "planes_conv":
            s["acc"] = torch.empty((c["B"], c["O"], ho, wo), dtype=torch.int32, device="cuda")
            s["y"] = _f32(c["B"], c["O"], ho, wo)
        else:
            s["qo"] = _quant(c["bo"])
            s["out"] = _i32(minw.packed_words(c["B"], c["O"], ho >> c["pool"], wo >> c["pool"], c["bo"]))
        return s
    if kind == "aqe":
        g = _gen(seed)
        shape = (c["B"], c["C"], c["H"], c["W"])
        m = c["B"] * c["C"] * c["H"] * c["W"]
        return dict(c=c, x=_normal(g, *shape), g=_normal(g, *shape), w=_uniform(g, c["n"]), gw=_normal(g, c["n"]),
                    qa=_quant(c["bits"]), qw=_quant(c["bw"]), y=_f32(*shape), gx=_f32(*shape),
                    planes=_i32(minw.packed_words(*shape, c["bits"])), mask=_i32((m + 31) // 32), yw=_f32(c["n"]),
                    gxw=_f32(c["n"]))
    if kind in ("fc_train", "conv_train"):
        g = _gen(seed)
        a, w, go = _train_inputs(c, g)
        s = dict(c=c, A=a, W=w, g=go, qa=_quant(c["ba"]), qw=_quant(c["bw"]), a_out=torch.empty_like(go),
                 a_pre=torch.empty_like(go), g_in=torch.empty_like(a))
        if kind == "fc_train":
            n = minw.minw_fc_train_workspace_bytes(c["B"], c["K"], c["O"])
        else:
            n = minw.minw_conv_train_workspace_bytes(c["B"], c["C"], c["H"], c["W"], c["O"], c["k"], c["k"],
                                                     c["stride"], c["pad"])
        s["ws"] = _u8(n)
        return s
    s = dict(c=c)
    if kind == "convnet":
        m = inputs.CIFAR_MODELS[c["model"]]
        p = inputs.convnet_params(seed, bits_a=c["ba"], bits_w=c["bw"], widths=m["widths"], fcs=m["fcs"])
        s["net"] = minw.Net(minw.layer_descs(p, torch.device("cuda")), c["B"])
        s["x"] = _uniform(_gen(seed), c["B"], 3, 32, 32)
        s["logits"] = _f32(c["B"], 10)
    elif kind == "resnet18":
        p = inputs.resnet18_params(seed, bits_a=c["ba"], bits_w=c["bw"], hw=c["hw"])
        s["net"] = minw.Net.resnet18(p, c["B"], torch.device("cuda"))
        s["x"] = _normal(_gen(seed), c["B"], 3, c["hw"], c["hw"])
        s["logits"] = _f32(c["B"], 1000)
    else:
        s["net"] = (minw.Net.wresnet if kind == "wresnet" else minw.Net.wdense)(_wonly_params(c, seed), c["B"],
                                                                                 torch.device("cuda"))
        s["x"] = _uniform(_gen(seed), c["B"], 3, 32, 32)
        s["logits"] = _f32(c["B"], 10)
    return s


def _wonly_params(c, seed):
    if c["kind"] == "wresnet":
        # residual branches a fifth of their shortcuts, as training leaves them: with branches of
        # the shortcuts' size and random weights, 54 blocks amplify any rounding to the logits' size
        p = inputs.wresnet_params(seed, n=c["n"], bits_w=c["bw"])
        for blk in p["blocks"]:
            blk["c2"]["scale"] = blk["c2"]["scale"] * np.float32(0.2)
        return p
    return inputs.wdense_params(seed, layers=c["layers"], growth=c["growth"], bits_w=c["bw"])


def _train_inputs(c, g):
    """Layer inputs whose pre-activations spread around the unit interval the activation
    quantizer and its mask act on, latent weights over [-1, 1], upstream gradients N(0, 0.1)."""
    if c["kind"] == "fc_train":
        k, ash, wsh, gsh = c["K"], (c["B"], c["K"]), (c["O"], c["K"]), (c["B"], c["O"])
    else:
        k = c["C"] * c["k"] ** 2
        ash, wsh = (c["B"], c["C"], c["H"], c["W"]), (c["O"], c["C"], c["k"], c["k"])
        gsh = (c["B"], c["O"]) + _out(c)
    a = (_normal(g, *ash) * (1.3 / k ** 0.5)).contiguous()
    return a, _uniform(g, *wsh), _normal(g, *gsh) * 0.1


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(s):
    c, kind = s["c"], s["c"]["kind"]
    if kind == "planes_conv":
        minw.aqe_quantize_pack(s["x"], s["qa"], s["act"])
        minw.minw_conv2d(s["act"], c["B"], c["C"], c["H"], c["W"], c["ba"], s["wgt"], c["O"], c["k"], c["k"], c["bw"],
                         c["stride"], c["pad"], s["acc"], s["scale"], s["shift"], s["y"])
        return {"acc": s["acc"], "y": s["y"]}
    if kind == "planes_block":
        minw.aqe_quantize_pack(s["x"], s["qa"], s["act"])
        minw.minw_conv_block(s["act"], c["B"], c["C"], c["H"], c["W"], c["ba"], s["wgt"], c["O"], c["k"], c["k"],
                             c["bw"], c["stride"], c["pad"], c["pool"], s["scale"], s["shift"], s["qo"], s["out"])
        return s["out"]
    if kind == "codes_block":
        fmt = minw.CODES_E2M1 if c["fp4"] else minw.CODES_E4M3
        (minw.aqe_quantize_codes_e2m1 if c["fp4"] else minw.aqe_quantize_codes)(s["x"], s["qa"], s["act"])
        minw.minw_conv_block_codes_ex(s["act"], c["B"], c["C"], c["H"], c["W"], c["ba"], s["wgt"], c["O"], c["k"],
                                      c["k"], c["bw"], c["stride"], c["pad"], c["pool"], s["scale"], s["shift"],
                                      s["qo"], s["out"], res_codes=s.get("res"), res_bits=c["bo"] if c["res"] else 0,
                                      in_format=fmt, out_format=fmt, res_format=fmt)
        return s["out"]
    if kind == "aqe":
        minw.aqe_quantize_pack(s["x"], s["qa"], s["planes"], ALPHA, s["y"], s["mask"])
        minw.aqe_backward_masked(s["mask"], s["g"], s["gx"], ALPHA)
        minw.aqe_forward(s["w"], s["yw"], ALPHA, s["qw"])
        minw.aqe_backward(s["w"], s["gw"], s["gxw"], ALPHA)
        return {"planes": s["planes"], "y": s["y"], "mask": s["mask"], "gx": s["gx"], "yw": s["yw"], "gxw": s["gxw"]}
    if kind == "fc_train":
        minw.minw_fc_train_step(s["A"], s["W"], s["g"], ALPHA, LR, s["qw"], s["qa"], s["a_out"], s["g_in"], s["ws"],
                                s["a_pre"])
        return {k: s[k] for k in ("a_pre", "a_out", "g_in", "W")}
    if kind == "conv_train":
        minw.minw_conv_train_step(s["A"], s["W"], s["g"], c["stride"], c["pad"], ALPHA, LR, s["qw"], s["qa"],
                                  s["a_out"], s["g_in"], s["ws"], s["a_pre"])
        return {k: s[k] for k in ("a_pre", "a_out", "g_in", "W")}
    s["net"].forward(s["x"], s["logits"])
    return s["logits"]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(c):
    kind = c["kind"]
    if kind in ("planes_conv", "planes_block", "codes_block"):
        ho, wo = _out(c)
        x, w, y = c["B"] * c["C"] * c["H"] * c["W"], c["O"] * c["C"] * c["k"] ** 2, c["B"] * c["O"] * ho * wo
        if kind == "planes_conv":
            out, wbits = 8 * y, c["bw"]
        elif kind == "planes_block":
            out, wbits = (y >> (2 * c["pool"])) * c["bo"] / 8, c["bw"]
        else:
            wbits = 4 if c["fp4"] else 8
            out = ((y >> (2 * c["pool"])) + (y if c["res"] else 0)) * wbits / 8
        return {"bytes": 4 * x + w * wbits / 8 + out, "flops": 2 * _macs(c)}
    if kind == "aqe":
        m = c["B"] * c["C"] * c["H"] * c["W"]
        return {"bytes": m * (4 + 4 + c["bits"] / 8 + 1 / 8 + 4 + 4) + 16 * c["n"], "flops": 6 * m + 6 * c["n"]}
    if kind == "fc_train":
        B, K, O = c["B"], c["K"], c["O"]
        return {"bytes": 4 * (2 * B * K + 2 * O * K + 3 * B * O), "flops": 6 * B * K * O}
    if kind == "conv_train":
        ho, wo = _out(c)
        x, w, y = c["B"] * c["C"] * c["H"] * c["W"], c["O"] * c["C"] * c["k"] ** 2, c["B"] * c["O"] * ho * wo
        return {"bytes": 4 * (2 * x + 2 * w + 3 * y), "flops": 6 * _macs(c)}
    macs, params, bits, classes, hw = 0, 0, c["bw"], 10, 32
    if kind == "convnet":
        m, size, ci = inputs.CIFAR_MODELS[c["model"]], 32, 3
        for i, co in enumerate(m["widths"]):
            macs, params = macs + 9 * ci * co * size ** 2, params + 9 * ci * co
            ci, size = co, size // 2 if i % 2 else size
        k = ci * size * size
        for o in list(m["fcs"]) + [10]:
            macs, params, k = macs + k * o, params + k * o, o
    elif kind == "resnet18":
        hw, classes = c["hw"], 1000
        size, ci = hw // 4, 64
        macs = 147 * 64 * (hw // 2) ** 2 + 512 * 1000
        for i, co in enumerate((64, 128, 256, 512)):
            size //= 2 if i else 1
            for j in range(2):
                cin = ci if j == 0 else co
                n = 9 * cin * co + 9 * co * co + (cin * co if i and j == 0 else 0)
                macs, params = macs + n * size ** 2, params + n
            ci = co
    elif kind == "wresnet":
        macs, ci, size = 27 * 16 * 1024, 16, 32
        for i, co in enumerate((16, 32, 64)):
            size //= 2 if i else 1
            for j in range(c["n"]):
                cin = ci if j == 0 else co
                n = 9 * cin * co + 9 * co * co + (cin * co if i and j == 0 else 0)
                macs, params = macs + n * size ** 2, params + n
            ci = co
    else:
        g, size = c["growth"], 32
        ch, macs = 2 * g, 27 * 2 * g * 1024
        for blk in range(3):
            for _ in range(c["layers"]):
                n = ch * 4 * g + 9 * 4 * g * g
                macs, params, ch = macs + n * size ** 2, params + n, ch + g
            if blk < 2:
                macs, params = macs + ch * (ch // 2) * size ** 2, params + ch * (ch // 2)
                ch, size = ch // 2, size // 2
    return {"bytes": c["B"] * (3 * hw * hw + classes) * 4 + params * bits / 8, "flops": 2 * macs * c["B"]}


# ---------------------------------------------------------------------------
# tolerances and the 64-bit results
# ---------------------------------------------------------------------------

def tolerance(c):
    if c["kind"] in ("fc_train", "conv_train"):
        # bf16 operands with fp32 sums: another order of the sums moves a~ by about 1e-6 and, where a~
        # lies at a threshold of the activation quantizer or at the mask's bound, one level (0.4 of an
        # output) or one gradient term: 9e-4 measured against the same bf16 operands summed in 64 bits
        return {"rel": 4e-3, "max": 0.9}
    if c["kind"] in ("wresnet", "wdense"):
        # every layer rounds its input to bf16: a change of the fp32 summation order flips a few
        # roundings, which travel through all layers that follow (1.4e-3, largest 4e-3, measured against
        # the same roundings with 64-bit sums)
        return {"rel": 5e-3, "max": 2e-2}
    # integer accumulators and the fp32 operations the interface states: every bit
    return "exact"


def _levels(x, bits):
    """The levels of x (their values; thresholds compared as the interface states)."""
    t = inputs.DEFAULT_THR[bits]
    if bits == 1:
        return torch.where(x > 0, 1.0, -1.0).double()
    a = x.abs()
    if bits == 2:
        m = (a > t[0]).double()
    else:
        m = torch.where(a > t[0], 1.0, torch.where(a > t[1], 0.5, torch.where(a > t[2], 0.25, 0.0))).double()
    return torch.where(x < 0, -m, m)


def _conv64(x, w, stride, pad):
    n = max(1, (1 << 26) // max(1, x[0].numel() * w.shape[-1] ** 2))
    return torch.cat([F.conv2d(x[i:i + n], w, stride=stride, padding=pad) for i in range(0, x.shape[0], n)])


def exact(c, seed):
    kind = c["kind"]
    if kind == "planes_conv":
        x, w, ws, scale, shift = _layer(c, seed)
        acc = _conv64(_levels(x, c["ba"]), _levels(w * ws[:, None, None, None], c["bw"]), c["stride"], c["pad"])
        acc = acc * (4.0 if c["ba"] == 3 else 1.0) * (4.0 if c["bw"] == 3 else 1.0)
        y = acc * scale.double()[:, None, None] + shift.double()[:, None, None]
        return {"acc": acc.round().to(torch.int32), "y": y}
    if kind == "aqe":
        s = prepare(c, seed)
        x, w = s["x"], s["w"]
        two = 2.0 * ALPHA
        return {"planes": None, "y": ALPHA * _levels(x, c["bits"]) + (1 - ALPHA) * x.double(), "mask": None,
                "gx": s["g"].double() * two * (x.abs() <= 1), "yw": ALPHA * _levels(w, c["bw"]) + (1 - ALPHA) * w.double(),
                "gxw": s["gw"].double() * two * (w.abs() <= 1)}
    if kind in ("fc_train", "conv_train"):
        a, w, g = _train_inputs(c, _gen(seed))
        a64, g64 = a.double(), g.double()
        wq = ALPHA * _levels(w, c["bw"]) + (1 - ALPHA) * w.double()
        if kind == "fc_train":
            pre = a64 @ wq.t()
        else:
            pre = _conv64(a64, wq, c["stride"], c["pad"])
        gm = 2 * ALPHA * g64 * (pre.abs() <= 1)
        if kind == "fc_train":
            g_in, gw = gm @ wq, gm.t() @ a64
        else:
            g_in, gw = torch.zeros_like(a64), torch.zeros_like(wq)
            n = max(1, (1 << 26) // (a64[0].numel() * c["k"] ** 2))
            for i in range(0, a64.shape[0], n):
                g_in[i:i + n] = torch.nn.grad.conv2d_input(a64[i:i + n].shape, wq, gm[i:i + n], c["stride"], c["pad"])
                gw += torch.nn.grad.conv2d_weight(a64[i:i + n], wq.shape, gm[i:i + n], c["stride"], c["pad"])
        w64 = w.double()
        return {"a_pre": pre, "a_out": ALPHA * _levels(pre, c["ba"]) + (1 - ALPHA) * pre, "g_in": g_in,
                "W": (w64 - LR * 2 * ALPHA * gw * (w64.abs() <= 1)).clamp(-1, 1)}
    if kind == "wresnet":
        return _wresnet64(_wonly_params(c, seed), _uniform(_gen(seed), c["B"], 3, 32, 32).double())
    if kind == "wdense":
        return _wdense64(_wonly_params(c, seed), _uniform(_gen(seed), c["B"], 3, 32, 32).double())
    # quantized networks and blocks return whole levels, or logits behind many layers of fp32 level
    # decisions that 64-bit arithmetic takes differently at ties: no such value
    return None


def _t64(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda().double()


def _bn64(y, r):
    return y * _t64(r["scale"])[:, None, None] + _t64(r["shift"])[:, None, None]


def _wq64(r, bits):
    w = torch.from_numpy(r["w"]).cuda() * torch.from_numpy(r["w_scale"]).cuda()[:, None, None, None]
    return _levels(w, bits) * (4.0 if bits == 3 else 1.0)


def _qconv64(x, r, bits, stride, pad):
    return _bn64(_conv64(x, _wq64(r, bits), stride, pad), r)


def _wresnet64(p, x):
    bits = p["bits_w"]
    x = _bn64(_conv64(x, _t64(p["stem"]["w"]), 1, 1), p["stem"]).clamp(-1, 1)
    for b in p["blocks"]:
        h = _qconv64(x, b["c1"], bits, b["stride"], 1).clamp(-1, 1)
        s = x if b["down"] is None else _qconv64(x, b["down"], bits, b["stride"], 0)
        x = (_qconv64(h, b["c2"], bits, 1, 1) + s).clamp(-1, 1)
    return _head64(x, p["fc"])


def _wdense64(p, x):
    bits = p["bits_w"]
    f = _bn64(_conv64(x, _t64(p["stem"]["w"]), 1, 1), p["stem"]).clamp(-1, 1)
    for i, block in enumerate(p["blocks"]):
        for lay in block:
            h = _qconv64(f, lay["b"], bits, 1, 0).clamp(-1, 1)
            f = torch.cat([f, _qconv64(h, lay["c"], bits, 1, 1).clamp(-1, 1)], dim=1)
        if i < 2:
            f = F.avg_pool2d(_qconv64(f, p["trans"][i], bits, 1, 0).clamp(-1, 1), 2)
    return _head64(f, p["fc"])


def _head64(x, fc):
    y = x.mean(dim=(2, 3)) @ _t64(fc["w"]).t()
    return y * _t64(fc["scale"]) + _t64(fc["shift"])
