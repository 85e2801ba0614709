"""The work whose speed is tracked: what a program that fine-tunes or serves a BCQ model has this
library do, through the public functions of the package.

Kinds of pass (a case's "kind"):
  train     one optimiser step's share of one layer: the forward of its linears, then for each of
            them, last first, the scale gradient and the input gradient
  prefill   the forward of a layer's linears over a long prompt
  decode    one token (or a small batch of tokens) through a layer's linears, from decode packs
  planes    the same from the canonical planes: a model whose scales are still being trained
  quantize  post-training quantization of a layer's linears, greedy or alternating
  update    AdamW on the trained scales of a whole model, and the checkpoint of them
"shape" says which linears: "block" are the four quantized linears of a Transformer block of width
d_in with a feed-forward width of d_out (qkv, attention output, FFN up, FFN down); "single" is one
linear d_in -> d_out.  g = 0 stands for row-wise scales (g = d_in of each linear).
"""
import math

import torch

import paper_2210_03858_b200 as bcq
from paper_2210_03858_b200.dist import AlphaBucket


def _linears(c):
    if c["shape"] == "single":
        return [(c["d_in"], c["d_out"])]
    h, f = c["d_in"], c["d_out"]
    return [(h, 3 * h), (h, h), (h, f), (f, h)]


def _g(c, d_in):
    return c["g"] or d_in


def listed():
    return [
        # The update of a GPT-2-medium run that trains alpha_1 of its 96 linears (row-wise, q = 3):
        # the smallest call, once per step.
        dict(name="update_gpt2_medium", kind="update", shape="block", d_in=1024, d_out=4096, q=3, g=0, layers=24),
        # One token through a GPT-2-medium layer: weights of 1 to 4 MB, so latency is what counts.
        dict(name="decode_gpt2_medium_q3_n1", kind="decode", shape="block", d_in=1024, d_out=4096, q=3, g=0, n=1,
             bf16=True, bias=True),
        # Serving one stream of OPT-6.7B at four bits: 126 MB of packed weights per layer.
        dict(name="decode_opt_6.7b_q4_n1", kind="decode", shape="block", d_in=4096, d_out=16384, q=4, g=128, n=1,
             bf16=False, bias=False),
        # Serving a full batch of the decode regime at three bits.
        dict(name="decode_opt_6.7b_q3_n16", kind="decode", shape="block", d_in=4096, d_out=16384, q=3, g=128, n=16,
             bf16=True, bias=False),
        # Generating during fine-tuning: the scales still change, so there is no pack.
        dict(name="decode_planes_gpt2_xl_q4_n4", kind="planes", shape="block", d_in=1600, d_out=6400, q=4, g=128, n=4,
             bf16=True, bias=True),
        # Fine-tuning as the paper does it: row-wise scales, q = 3, only alpha_1 gets a gradient.
        dict(name="train_gpt2_medium_q3", kind="train", shape="block", d_in=1024, d_out=4096, q=3, g=0, n=2048,
             bf16=True, bias=False, prepared=True, planes=1),
        # Group-wise scales, four planes, every plane trained, a long batch.
        dict(name="train_gpt2_xl_q4_g128", kind="train", shape="block", d_in=1600, d_out=6400, q=4, g=128, n=4096,
             bf16=True, bias=False, prepared=True, planes=15),
        # A short, ragged batch on one odd-sized linear straight from the canonical planes, with
        # fp32 results: nothing divides a tile.
        dict(name="train_ragged_q2_g64", kind="train", shape="single", d_in=1000, d_out=1528, q=2, g=64, n=777,
             bf16=False, bias=True, prepared=False, planes=3),
        # A prompt of 2048 tokens through an OPT-13B layer: the largest forward.
        dict(name="prefill_opt_13b_q2", kind="prefill", shape="block", d_in=5120, d_out=20480, q=2, g=128, n=2048,
             bf16=True, bias=False, prepared=True),
        # Greedy quantization of a GPT-2-XL layer, group-wise.
        dict(name="quantize_gpt2_xl_greedy_q4", kind="quantize", shape="block", d_in=1600, d_out=6400, q=4, g=128,
             iters=0, outliers=0.0),
        # Greedy quantization with one scale per row and plane.
        dict(name="quantize_gpt2_medium_row_q3", kind="quantize", shape="block", d_in=1024, d_out=4096, q=3, g=0,
             iters=0, outliers=0.0),
        # Alternating quantization of one OPT-13B linear with outliers.
        dict(name="quantize_opt_13b_alt5_q3", kind="quantize", shape="single", d_in=5120, d_out=5120, q=3, g=128,
             iters=5, outliers=1e-3),
    ]


def _log(rng, lo, hi, step):
    """A multiple of `step` in [lo, hi], spread evenly over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    kind = rng.choice(["update", "decode", "decode", "decode", "planes", "train", "train", "train", "prefill",
                       "quantize", "quantize", "quantize"])
    q = rng.choice([2, 3, 4])
    g = rng.choice([0, 64, 128, 128, 256])
    c = dict(kind=kind, q=q, g=g)
    if kind == "update":
        h = _log(rng, 768, 2048, 64)
        c.update(shape="block", d_in=h, d_out=4 * h, layers=rng.randint(12, 48))
    elif kind in ("decode", "planes"):
        n = rng.choice([1, 1, 2, 4, 8, 16, rng.randint(1, 16)])
        c.update(n=n, bf16=rng.random() < 0.5, bias=rng.random() < 0.5)
        if rng.random() < 0.5:
            h = _log(rng, 768, 5120 if kind == "decode" else 2560, 64)
            c.update(shape="block", d_in=h, d_out=4 * h)
        else:
            c.update(shape="single", d_in=_log(rng, 512, 16384, 8), d_out=_log(rng, 512, 16384, 1))
    elif kind == "train":
        c.update(n=_log(rng, 128, 4096, 1), bf16=rng.random() < 0.75, bias=rng.random() < 0.5,
                 prepared=rng.random() < 0.75, planes=rng.choice([1, (1 << q) - 1]))
        if rng.random() < 0.5:
            h = _log(rng, 768, 1600, 32)
            c.update(shape="block", d_in=h, d_out=4 * h)
        else:
            c.update(shape="single", d_in=_log(rng, 512, 6400, 8), d_out=_log(rng, 512, 6400, 8))
    elif kind == "prefill":
        c.update(n=_log(rng, 32, 2048, 1), bf16=rng.random() < 0.75, bias=rng.random() < 0.5, prepared=True)
        if rng.random() < 0.5:
            h = _log(rng, 1024, 5120, 64)
            c.update(shape="block", d_in=h, d_out=4 * h)
        else:
            c.update(shape="single", d_in=_log(rng, 1024, 16384, 8), d_out=_log(rng, 1024, 16384, 1))
    else:
        iters = rng.choice([0, 0, 5, 15])
        c.update(shape="single", d_in=_log(rng, 512, 8192, 1), d_out=_log(rng, 512, 3200 if iters else 8192, 1),
                 iters=iters, outliers=rng.choice([0.0, 1e-3]))
    return c


def _weights(c, d_out, d_in, gen):
    W = torch.randn((d_out, d_in), generator=gen, device="cuda") * 0.02
    if c.get("outliers"):
        W = torch.where(torch.rand((d_out, d_in), generator=gen, device="cuda") < c["outliers"], W * 20.0, W)
    return W


def _ws(op, d_out, d_in, q, g, n):
    return torch.empty(max(16, bcq.workspace_bytes(op, d_out, d_in, q, g, n)), dtype=torch.uint8, device="cuda")


def _bf16(shape, gen):
    return torch.randn(shape, generator=gen, device="cuda").bfloat16()


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind, q = c["kind"], c["q"]
    st = dict(case=c, lin=[])
    if kind == "update":
        shapes = [(q, do, bcq.num_groups(di, _g(c, di))) for di, do in _linears(c)] * c["layers"]
        flat = [AlphaBucket(shapes, "cuda") for _ in range(4)]  # alpha, its gradient, the two moments
        alpha, grad, m, v = (b.flat for b in flat)
        alpha.copy_(torch.rand(alpha.shape, generator=gen, device="cuda") * 0.02)
        grad.copy_(torch.randn(grad.shape, generator=gen, device="cuda"))
        scales = [1.0 / _g(c, di) for di, _ in _linears(c)] * c["layers"]
        seg = bcq.Segments(flat[0].plane_segments(1), "cuda", scales)
        return dict(case=c, alpha=alpha, grad=grad, m=m, v=v, seg=seg, step=0)
    for d_in, d_out in _linears(c):
        g = _g(c, d_in)
        W = _weights(c, d_out, d_in, gen)
        if kind == "quantize":
            st["lin"].append(dict(W=W, g=g))
            continue
        n, dt = c["n"], torch.bfloat16 if c["bf16"] else torch.float32
        bits, alpha, _ = bcq.quantize(W, q, g)
        l = dict(d_in=d_in, d_out=d_out, g=g, bits=bits, alpha=alpha, X=_bf16((n, d_in), gen),
                 Y=torch.empty((n, d_out), dtype=dt, device="cuda"),
                 bias=torch.randn(d_out, generator=gen, device="cuda") * 0.02 if c["bias"] else None)
        if kind == "decode":
            l.update(pack=bcq.decode_pack(bits, alpha, d_in, g), ws=_ws(bcq.OP_DECODE_PACKED, d_out, d_in, q, g, n))
        elif kind == "planes":
            l.update(ws=_ws(bcq.OP_DECODE, d_out, d_in, q, g, n))
        else:
            l.update(fwd=bcq.prepare_planes(bcq.OP_FWD, bits, d_in, g) if c["prepared"] else bits,
                     ws=_ws(bcq.OP_FWD, d_out, d_in, q, g, n))
        if kind == "train":
            l.update(dY=_bf16((n, d_out), gen), dX=torch.empty((n, d_in), dtype=dt, device="cuda"),
                     dA=torch.zeros_like(alpha), bwd=bcq.prepare_planes(bcq.OP_BWD_X, bits, d_in, g) if c["prepared"] else bits,
                     ws_dA=_ws(bcq.OP_BWD_ALPHA, d_out, d_in, q, g, n), ws_dX=_ws(bcq.OP_BWD_X, d_out, d_in, q, g, n))
        st["lin"].append(l)
    return st


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "update":
        s = state
        s["step"] += 1
        lr = bcq.lr_linear_decay(1e-3, s["step"] - 1, 0, 10 ** 9)
        bcq.alpha_adamw(s["alpha"], s["grad"], s["m"], s["v"], s["step"], lr, weight_decay=0.01, segments=s["seg"])
        return s["alpha"], s["m"], s["v"], bcq.alpha_pack(s["alpha"], s["seg"])
    if kind == "quantize":
        return [bcq.quantize(l["W"], c["q"], l["g"], c["iters"])[:2] for l in state["lin"]]
    if kind == "decode":
        return [bcq.linear_decode_packed(l["X"], l["pack"], l["d_out"], l["d_in"], c["q"], l["g"], bias=l["bias"],
                                         out=l["Y"], ws=l["ws"]) for l in state["lin"]]
    if kind == "planes":
        return [bcq.linear_decode(l["X"], l["bits"], l["alpha"], l["d_in"], l["g"], bias=l["bias"], out=l["Y"],
                                  ws=l["ws"]) for l in state["lin"]]
    out = [bcq.linear_fwd(l["X"], l["fwd"], l["alpha"], l["d_in"], l["g"], bias=l["bias"], out=l["Y"], ws=l["ws"])
           for l in state["lin"]]
    if kind == "train":
        for l in reversed(state["lin"]):
            out.append(bcq.linear_bwd_alpha(l["dY"], l["X"], l["bits"], l["d_in"], l["g"], plane_mask=c["planes"],
                                            scale=1.0 / l["g"], out=l["dA"], ws=l["ws_dA"]))
            out.append(bcq.linear_bwd_x(l["dY"], l["bwd"], l["alpha"], l["d_in"], l["g"], out=l["dX"], ws=l["ws_dX"]))
    return out


def work(case):
    c = case
    kind, q = c["kind"], c["q"]
    by, fl = 0.0, 0.0
    for d_in, d_out in _linears(c):
        g = _g(c, d_in)
        w, na = d_in * d_out, d_out * -(-d_in // g)  # weights; scales of one plane
        if kind == "update":
            # alpha, gradient and moments of plane 1 read, three of them written, the checkpoint written
            by += c["layers"] * na * 4 * (4 + 3 + 1)
            fl += c["layers"] * na * 15
        elif kind == "quantize":
            # per weight and plane: into the mean, and off the residual; per round: q sums and the
            # choice among 2^q levels (q comparisons)
            by += 4 * w + q * w / 8 + 4 * q * na
            fl += w * (2 * q + (q + c["iters"] * 2 * q if c["iters"] else 0))
        else:
            n, e = c["n"], 2 if c["bf16"] else 4
            planes = q * w / 8 + 4 * q * na
            by += planes + 2 * n * d_in + e * n * d_out + (4 * d_out if c["bias"] else 0)
            fl += 2.0 * n * w
            if kind == "train":
                trained = bin(c["planes"]).count("1")
                by += 2 * (2 * n * d_out) + 2 * n * d_in + planes + trained * (w / 8 + 4 * na) + e * n * d_in
                fl += 4.0 * n * w
    return {"bytes": by, "flops": fl}


def tolerance(case):
    c = case
    if c["kind"] == "update":
        return {"rel": 1e-6, "max": 1e-5}  # fp32 element by element
    if c["kind"] == "quantize":
        # bits equal but for ties that the order of a 64-bit sum decides; scales are 32-bit
        return {"rel": 1e-6, "max": 1e-5, "differ": 1e-6}
    # Weights go into the products as fp16 (relative rounding error up to 2^-11, 2e-4 over a result);
    # a bf16 result adds its own rounding (1.7e-3).
    return {"rel": 6e-3, "max": 4e-2} if c["bf16"] else {"rel": 1e-3, "max": 1e-2}
