"""Workloads for timing the framework through its public entry points.

Every case is an operator graph that goes through rewriting and fusion planning once (`prepare`) and is then executed with
`Session.run()`, one call per pass, plain stream launches: what a program that serves a model does.  The kinds are those of
`paper_2108_13342_b200/workloads.py` with every size free; the graphs are written out here because the inputs are drawn on
the GPU and never exist on the host.

  swish        bias + scale + swish + NCHW -> NHWC transpose, fp32: the element-wise / Shuffle kernels
  softmax      scale + causal mask + row softmax, fp32: attention scores of a batch
  layernorm    residual add + LayerNorm + GELU, fp32
  ffn          GEMM + bias + GELU, GEMM + bias + residual, bf16: a transformer's feed-forward block
  mbconv       inverted-residual block, fp32 NHWC: expansion, depthwise 3x3, projection, residual
  stack        MobileNetV2-shaped network of nine inverted-residual blocks, pools, head and classifier, fp32 NHWC
  neck         feature-pyramid fragment: pools, SpaceToDepth / DepthToSpace, Resize, Concat, global-pool gate, fp32 NHWC
  style        decoder of a style-transfer network: InstanceNormalization, overlapping ConvTranspose, fp32 NHWC
  encoder      post-LayerNorm transformer encoder as primitive operators, bf16
  decoder      GPT-2 style pre-LayerNorm decoder as primitive operators, bf16
"""
import math

import torch

from paper_2108_13342_b200 import binding as B
from paper_2108_13342_b200 import workloads as W
from paper_2108_13342_b200.runtime import Session


# --------------------------------------------------------------------------------------------------
# Graphs: operators as plain data, external tensors with the distribution their values are drawn from
# --------------------------------------------------------------------------------------------------

class _Net:
    def __init__(self, name):
        self.g = W.GraphDesc(name)
        self.values = {}                                   # external tensor -> (distribution, a, b)

    def ext(self, shape, dist, dtype="f32", name=None):
        name = name or "p%d" % len(self.values)
        self.g.ext(name, shape, dtype, "weight" if name[0] == "p" else "input")
        self.values[name] = dist
        return name

    def add(self, op, *inputs, **kw):
        return self.g.add(op, list(inputs), **kw)

    def done(self, out):
        self.g.mark_output(out)
        return self

    # ---- fp32 NHWC pieces
    def bn(self, x, c):
        return self.add("ScaleShift", x, self.ext((c,), ("uniform", 0.5, 1.5)), self.ext((c,), ("uniform", -0.5, 0.5)), axis=-1)

    def relu6(self, x):
        return self.add("Clip", x, lo=0.0, hi=6.0)

    def conv(self, x, cin, cout, gain=2.0):
        return self.add("Conv1x1", x, self.ext((cin, cout), ("normal", 0.0, math.sqrt(gain / cin))))

    def dwconv(self, x, c):
        return self.add("DwConv3x3", x, self.ext((3, 3, c), ("normal", 0.0, math.sqrt(2.0 / 9.0))))

    def inverted_residual(self, x, cin, cout, t, gain=1.0):
        e = cin * t
        y = self.relu6(self.bn(self.conv(x, cin, e), e))
        y = self.relu6(self.bn(self.dwconv(y, e), e))
        y = self.bn(self.conv(y, e, cout, gain), cout)
        return self.add("Add", y, x) if cin == cout else y

    # ---- bf16 transformer pieces
    def vec(self, n, mean=0.0):
        return self.ext((n,), ("normal", mean, 0.02))

    def linear(self, x, k, n):
        y = self.add("MatMul", x, self.ext((k, n), ("normal", 0.0, 0.02), "bf16"))
        return self.add("Add", y, self.vec(n))

    def layernorm(self, x, n):
        mu = self.add("ReduceMean", x, axis=-1, keepdims=1)
        xc = self.add("Sub", x, mu)
        var = self.add("ReduceMean", self.add("Pow", xc, p=2.0), axis=-1, keepdims=1)
        xn = self.add("Div", xc, self.add("Sqrt", self.add("AddC", var, c=1e-5)))
        return self.add("Add", self.add("Mul", xn, self.vec(n, 1.0)), self.vec(n))

    def gelu_erf(self, x):
        t = self.add("AddC", self.add("Erf", self.add("MulC", x, c=1.0 / math.sqrt(2.0))), c=1.0)
        return self.add("MulC", self.add("Mul", x, t), c=0.5)

    def gelu_tanh(self, x):
        x3 = self.add("Mul", self.add("Mul", x, x), x)
        t = self.add("Add", x, self.add("MulC", x3, c=0.044715))
        t = self.add("AddC", self.add("Tanh", self.add("MulC", t, c=math.sqrt(2.0 / math.pi))), c=1.0)
        return self.add("MulC", self.add("Mul", x, t), c=0.5)

    def attention(self, x, batch, seq, heads, mask):
        hidden = 64 * heads
        qkv = self.add("Split", self.linear(x, hidden, 3 * hidden), n_out=3, axis=-1, sizes=(hidden,) * 3)
        q, k, v = (self.add("Transpose", self.add("Reshape", t, shape=(batch, seq, heads, 64)), perm=(0, 2, 1, 3)) for t in qkv)
        s = self.add("MatMul", q, self.add("Transpose", k, perm=(0, 1, 3, 2)))
        s = self.add("Add", self.add("MulC", s, c=0.125), mask)
        a = self.add("Transpose", self.add("MatMul", self.add("Softmax", s, axis=-1), v), perm=(0, 2, 1, 3))
        return self.linear(self.add("Reshape", a, shape=(batch, seq, hidden)), hidden, hidden)


def _swish(c):
    net = _Net("swish")
    t = net.add("Add", net.ext((c["n"], c["c"], c["h"], c["w"]), ("uniform", -1.0, 1.0), name="X"),
                net.ext((1, c["c"], 1, 1), ("uniform", -0.5, 0.5)))
    t = net.add("MulC", t, c=0.5)
    return net.done(net.add("Transpose", net.add("Mul", t, net.add("Sigmoid", t)), perm=(0, 2, 3, 1)))


def _softmax(c):
    net = _Net("softmax")
    s = net.ext((c["batch"], c["heads"], c["seq"], c["seq"]), ("normal", 0.0, 1.0), name="S")
    t = net.add("Add", net.add("MulC", s, c=0.125), net.ext((c["seq"], c["seq"]), ("causal", 0, 0)))
    return net.done(net.add("Softmax", t, axis=-1))


def _layernorm(c):
    net = _Net("layernorm")
    h, r = (net.ext((c["rows"], c["hidden"]), ("normal", 0.0, 1.0), name=n) for n in ("H", "R"))
    y = net.add("LayerNorm", net.add("Add", h, r), net.vec(c["hidden"], 1.0), net.vec(c["hidden"]), axis=-1, eps=1e-5)
    return net.done(net.add("Gelu", y, approx="erf"))


def _ffn(c):
    net = _Net("ffn")
    x = net.ext((c["rows"], c["hidden"]), ("normal", 0.0, 1.0), "bf16", name="A")
    t = net.add("Gelu", net.linear(x, c["hidden"], 4 * c["hidden"]), approx="tanh")
    return net.done(net.add("Add", net.linear(t, 4 * c["hidden"], c["hidden"]), x))


def _mbconv(c):
    net = _Net("mbconv")
    x = net.ext((c["n"], c["h"], c["w"], c["cin"]), ("uniform", 0.0, 1.0), name="X")
    return net.done(net.inverted_residual(x, c["cin"], c["cin"], c["t"], gain=2.0))


def _stack(c):
    net = _Net("stack")
    x = net.ext((c["n"], c["hw"], c["hw"], 16), ("uniform", 0.0, 1.0), name="X")
    hw = c["hw"]
    for cin, cout in ((16, 24), (24, 24), (0, 0), (24, 32), (32, 32), (32, 64), (0, 0), (64, 64), (64, 96), (96, 96), (96, 160)):
        if cin:
            x = net.inverted_residual(x, cin, cout, 6)
        else:
            x = net.add("MaxPool", x, kernel=3, stride=2, pad=1)
            hw = (hw + 1) // 2
    x = net.relu6(net.bn(net.conv(x, 160, 320), 320))
    x = net.add("AveragePool", x, kernel=hw, stride=1, pad=0)
    return net.done(net.add("Add", net.conv(x, 320, 100, 1.0), net.ext((100,), ("uniform", -0.1, 0.1))))


def _neck(c):
    net, n, hw, ch = _Net("neck"), c["n"], c["hw"], c["c"]
    x = net.ext((n, hw, hw, ch), ("uniform", 0.0, 1.0), name="X")

    def unit(y, cin, cout):
        return net.relu6(net.bn(net.conv(y, cin, cout), cout))

    stem = unit(x, ch, 2 * ch)
    low = net.add("MaxPool", stem, kernel=3, stride=2, pad=1)
    lateral = unit(net.add("SpaceToDepth", stem, block=2), 8 * ch, 2 * ch)
    dw = net.relu6(net.bn(net.dwconv(net.add("Concat", low, lateral, axis=3), 4 * ch), 4 * ch))
    gate = net.add("Sigmoid", net.conv(net.add("AveragePool", dw, kernel=hw // 2, stride=1, pad=0), 4 * ch, 4 * ch, 1.0))
    gated = net.add("Mul", dw, gate)
    up_a = net.add("DepthToSpace", gated, block=2)
    up_b = net.add("Resize", unit(gated, 4 * ch, ch), scale=2)
    return net.done(net.add("Add", unit(net.add("Concat", up_a, up_b, x, axis=3), 3 * ch, ch), x))


def _style(c):
    net, ch = _Net("style"), c["c"]

    def inorm(y, k):
        return net.add("InstanceNorm", y, net.ext((k,), ("uniform", 0.5, 1.5)), net.ext((k,), ("uniform", -0.5, 0.5)), eps=1e-5)

    x = net.ext((c["n"], c["hw"], c["hw"], ch), ("uniform", -1.0, 1.0), name="X")
    y = net.add("Relu", inorm(net.conv(x, ch, ch), ch))
    y = net.add("Add", inorm(net.dwconv(y, ch), ch), x)
    for _ in range(2):
        w = net.ext((ch, 4, 4, ch // 2), ("normal", 0.0, math.sqrt(2.0 / (4 * ch))))
        ch //= 2
        y = net.add("Relu", inorm(net.add("ConvTranspose", y, w, kernel=4, stride=2, pad=1), ch))
    y = net.add("Add", net.conv(y, ch, 4, 1.0), net.ext((4,), ("uniform", -0.1, 0.1)))
    return net.done(net.add("Tanh", y))


def _transformer(c):
    pre = c["kind"] == "decoder"
    net, hidden, dims = _Net(c["kind"]), 64 * c["heads"], (c["batch"], c["seq"], c["heads"])
    x = net.ext((c["batch"], c["seq"], hidden), ("normal", 0.0, 1.0), "bf16", name="X")
    mask = net.ext((c["seq"], c["seq"]), ("causal", 0, 0))
    for _ in range(c["layers"]):
        if pre:
            x = net.add("Add", x, net.attention(net.layernorm(x, hidden), *dims, mask))
            f = net.gelu_tanh(net.linear(net.layernorm(x, hidden), hidden, 4 * hidden))
            x = net.add("Add", x, net.linear(f, 4 * hidden, hidden))
        else:
            x = net.layernorm(net.add("Add", net.attention(x, *dims, mask), x), hidden)
            f = net.gelu_erf(net.linear(x, hidden, 4 * hidden))
            x = net.layernorm(net.add("Add", net.linear(f, 4 * hidden, hidden), x), hidden)
    return net.done(net.layernorm(x, hidden) if pre else x)


_BUILD = {"swish": _swish, "softmax": _softmax, "layernorm": _layernorm, "ffn": _ffn, "mbconv": _mbconv, "stack": _stack,
          "neck": _neck, "style": _style, "encoder": _transformer, "decoder": _transformer}


# --------------------------------------------------------------------------------------------------
# The cases
# --------------------------------------------------------------------------------------------------

def listed():
    return [
        # one activation map of a small image between two convolutions: a single launch, 1.6 MB
        {"name": "swish_one_image", "kind": "swish", "n": 1, "c": 64, "h": 56, "w": 56},
        # attention scores of a small batch at a sequence length that fits no vector width
        {"name": "softmax_seq_197", "kind": "softmax", "batch": 8, "heads": 12, "seq": 197},
        # the norm block of a large training-sized batch: pure memory streaming, 1.2 GB
        {"name": "layernorm_131072_rows", "kind": "layernorm", "rows": 131072, "hidden": 768},
        # feed-forward block of a base-sized transformer on 4096 tokens
        {"name": "ffn_4096_tokens", "kind": "ffn", "rows": 4096, "hidden": 768},
        # the same layer, wider, on a large ragged batch of packed sequences: the most arithmetic
        {"name": "ffn_12345_tokens", "kind": "ffn", "rows": 12345, "hidden": 1024},
        # an inverted-residual block of a mobile CNN on a batch of 32
        {"name": "mbconv_32_images", "kind": "mbconv", "n": 32, "h": 56, "w": 56, "cin": 24, "t": 6},
        # a whole mobile CNN on one image: latency, 32 small kernels
        {"name": "stack_one_image", "kind": "stack", "n": 1, "hw": 56},
        # the same network on a batch
        {"name": "stack_32_images", "kind": "stack", "n": 32, "hw": 56},
        # detection-style feature pyramid with the index operators and a global-pool gate
        {"name": "neck_8_images", "kind": "neck", "n": 8, "hw": 64, "c": 32},
        # image-to-image decoder, 64 x 64 features to 256 x 256 pixels
        {"name": "style_8_images", "kind": "style", "n": 8, "hw": 64, "c": 64},
        # a 12-layer encoder, 576 primitive operators, planned by the paper's rules
        {"name": "encoder_8x128", "kind": "encoder", "layers": 12, "batch": 8, "seq": 128, "heads": 12, "beyond": False},
        # a 12-layer decoder on one long prompt, with the single-kernel attention block
        {"name": "decoder_1x248", "kind": "decoder", "layers": 12, "batch": 1, "seq": 248, "heads": 12, "beyond": True},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def _any_case(rng):
    kind = rng.choice(sorted(_BUILD))
    if kind == "swish":
        c = {"n": _log(rng, 1, 256), "c": _log(rng, 8, 256), "h": _log(rng, 7, 112), "w": _log(rng, 7, 112)}
        size = c["n"] * c["c"] * c["h"] * c["w"]
    elif kind == "softmax":
        c = {"batch": _log(rng, 1, 64), "heads": rng.randint(1, 16), "seq": _log(rng, 16, 1024)}
        size = c["batch"] * c["heads"] * c["seq"] ** 2
    elif kind == "layernorm":
        c = {"rows": _log(rng, 1, 131072), "hidden": _log(rng, 64, 4096)}
        size = c["rows"] * c["hidden"]
    elif kind == "ffn":
        c = {"rows": _log(rng, 1, 12345), "hidden": 64 * rng.randint(2, 16)}
        size = 0
    elif kind == "mbconv":
        c = {"n": _log(rng, 1, 64), "h": _log(rng, 7, 112), "w": _log(rng, 7, 112), "cin": 8 * rng.randint(2, 12), "t": rng.choice((3, 4, 6))}
        size = 6 * c["n"] * c["h"] * c["w"] * c["cin"] * c["t"]
    elif kind == "stack":
        c = {"n": _log(rng, 1, 32), "hw": _log(rng, 28, 112)}
        size = 1000 * c["n"] * c["hw"] ** 2
    elif kind == "neck":
        c = {"n": _log(rng, 1, 32), "hw": 2 * rng.randint(8, 48), "c": 8 * rng.randint(1, 8)}
        size = 25 * c["n"] * c["hw"] ** 2 * c["c"]
    elif kind == "style":
        c = {"n": _log(rng, 1, 16), "hw": _log(rng, 16, 96), "c": 16 * rng.randint(1, 8)}
        size = 45 * c["n"] * c["hw"] ** 2 * c["c"]
    else:
        c = {"layers": rng.randint(1, 12), "batch": _log(rng, 1, 16), "seq": _log(rng, 16, 256), "heads": rng.randint(2, 12),
             "beyond": rng.random() < 0.5}
        size = 100000 * c["batch"] * c["seq"]
    return dict(c, kind=kind), size


def draw(rng):
    """A case of any kind; sizes whose pass would take longer than the largest listed ones are drawn again."""
    while True:
        c, size = _any_case(rng)
        if size <= 103_000_000:
            return c


def prepare(case, seed):
    net = _BUILD[case["kind"]](case)
    transformer = case["kind"] in ("encoder", "decoder")
    sess = Session(W.Workload(net.g, {}), plan_flags=B.PLAN_BEYOND_TABLE3 if case.get("beyond") else B.PLAN_FUSED,
                   rewrite_flags=B.REWRITE_CANON_MACRO if transformer else B.REWRITE_DEFAULT, upload=False)
    gen = torch.Generator(device=sess.device).manual_seed(seed)
    for name, (dist, a, b) in net.values.items():
        t = net.g.tensors[name]
        x = torch.empty(t.shape, dtype=torch.float32, device=sess.device)
        if dist == "causal":
            x = x.fill_(-1e9).triu_(1)
        elif dist == "normal":
            x.normal_(a, b, generator=gen)
        else:
            x.uniform_(a, b, generator=gen)
        sess.buffers[name] = x.to(torch.bfloat16) if t.dtype == "bf16" else x
        sess.g.bind(sess.ids[name], sess.buffers[name].data_ptr())
    return sess


def run(sess):
    sess.run()
    return [sess.buffers[name] for name in sess.desc.outputs]


def work(case):
    """Inputs and weights read once, outputs written once; multiply-adds of the contractions and depthwise filters."""
    net = _BUILD[case["kind"]](case)
    g = net.g
    nbytes = sum(math.prod(t.shape) * (2 if t.dtype == "bf16" else 4) for t in g.tensors.values())
    c, k = case, case["kind"]
    flops = 0
    if k in ("swish", "softmax", "layernorm"):
        x = {"swish": "X", "softmax": "S", "layernorm": "H"}[k]
        nbytes += 4 * math.prod(g.tensors[x].shape)
    elif k == "ffn":
        nbytes += 2 * c["rows"] * c["hidden"]
        flops = 16 * c["rows"] * c["hidden"] ** 2
    elif k == "mbconv":
        px, e = c["n"] * c["h"] * c["w"], c["cin"] * c["t"]
        nbytes += 4 * px * c["cin"]
        flops = px * e * (4 * c["cin"] + 18)
    elif k in ("encoder", "decoder"):
        tokens, hidden = c["batch"] * c["seq"], 64 * c["heads"]
        nbytes += 2 * tokens * hidden
        flops = c["layers"] * tokens * (24 * hidden ** 2 + 4 * c["seq"] * hidden)
    elif k == "stack":
        hw, px = c["hw"], c["n"] * c["hw"] ** 2
        for cin, cout in ((16, 24), (24, 24), (0, 0), (24, 32), (32, 32), (32, 64), (0, 0), (64, 64), (64, 96), (96, 96), (96, 160)):
            if cin:
                flops += px * 6 * cin * (2 * cin + 18 + 2 * cout)
            else:
                hw = (hw + 1) // 2
                px = c["n"] * hw ** 2
        nbytes += 4 * c["n"] * 100
        flops += px * 2 * 160 * 320 + c["n"] * 2 * 320 * 100
    elif k == "neck":
        px, ch = c["n"] * c["hw"] ** 2, c["c"]
        nbytes += 4 * px * ch
        flops = px * (2 * ch * 2 * ch + 2 * 3 * ch * ch) + px // 4 * (2 * 8 * ch * 2 * ch + 18 * 4 * ch + 2 * 4 * ch * ch) + c["n"] * 2 * (4 * ch) ** 2
    else:
        px, ch = c["n"] * c["hw"] ** 2, c["c"]
        nbytes += 4 * px * 16 * 4
        flops = px * (2 * ch * ch + 18 * ch + 2 * ch * 8 * ch + 4 * 2 * (ch // 2) * 4 * ch + 16 * 2 * (ch // 4) * 4)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times what was measured between two correct ways of computing the same case."""
    kind = case["kind"]
    if kind in ("swish", "softmax", "layernorm"):
        return {"rel": 5e-7, "max": 3e-6}       # fp32 against fp64: 1.3e-7, 5.7e-7
    if kind in ("mbconv", "stack", "neck", "style"):
        return {"rel": 1e-5, "max": 4e-5}       # split-TF32 tensor cores against fp32 multiply-adds: 2.4e-6, 7.4e-6
    if kind == "ffn":
        return {"rel": 2e-3, "max": 3e-2}       # bf16 results against fp64 with the hidden values in bf16: 3.3e-4, 7.8e-3
    return {"rel": 0.03, "max": 0.3}            # 12 layers of bf16 activations, other sums and roundings: 1.4e-2, 9.4e-2
