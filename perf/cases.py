"""The work whose time counts: training steps of quantised layers and of a layer stack, their products, their
normalisation and their quantisers, each through the public entry points a training program calls.

Kinds, with the ranges that `listed` samples and `draw` covers:

  conv     forward + backward of one convolution layer (3x3 or 1x1, stride 1): 1 to 256 images of 5x5 to 56x56 positions,
           32 to 512 channels, the channel counts of residual networks (64 ... 512) and odd multiples of 32
  linear   forward + backward of one linear layer: batch 16 to 4096, 16 to 4096 features, multiples of 16
  stack    one training step of a bottleneck of three convolutions (chained codes, weight update), 2 to 256 images
  infer    the forward of such a bottleneck alone: inner layers hand on 8-bit codes and keep no fp32 product
  gemm     the 8-bit product on codes in hand, each operand either way round: 128 to 8192 in each direction
  wgrad    the 16-bit x 8-bit weight-gradient product, dense: 128 to 8192 in each direction
  rangebn  Range BN forward + backward on its own, with and without the rectifier: 1 K to 800 K rows, 16 to 2048 channels
  quantize the quantisers on their own: nearest or stochastic, per tensor or per channel, 8 or 16 bits, both copies of
           a gradient; also row lengths that are no multiple of 4
  ternary  forward + backward of the low-bit layer (Appendix C): 1-bit operands, ternary gradients, 1 to 8 samples

Values as in paper_1805_11046_b200/synth.py: rectified N(0,1) activations, Kaiming filters, N(0, 0.1) gradients,
per-channel shifted Gaussians for Range BN on its own."""
from __future__ import annotations

import math

import torch

from paper_1805_11046_b200 import binding as B
from paper_1805_11046_b200 import layer


def listed():
    return [
        # the smallest layer of the tests and of the benchmark: all latency and launches
        dict(name="linear_64", kind="linear", batch=64, cin=256, cout=128),
        # a classifier or embedding layer in training: wide, one ragged extent
        dict(name="linear_1024", kind="linear", batch=1024, cin=2048, cout=1008),
        # the first stage of a residual network at a full minibatch: the benchmark's layer, bound by memory
        dict(name="conv_56x64", kind="conv", n=256, hw=56, c=64, k=64, r=3),
        # a late stage of the same network: fewer positions, more channels, bound by the products
        dict(name="conv_14x256", kind="conv", n=256, hw=14, c=256, k=256, r=3),
        # a small minibatch of odd images between unequal, odd channel counts
        dict(name="conv_19_odd", kind="conv", n=20, hw=19, c=96, k=160, r=3),
        # the training step of the benchmark's bottleneck stack
        dict(name="stack_256", kind="stack", n=256, hw=28, c=256, mid=128, k=512),
        # serving the same stack to a few images
        dict(name="infer_8", kind="infer", n=8, hw=28, c=256, mid=128, k=512),
        # the dense product of the benchmark's sweep: bound by the tensor cores
        dict(name="gemm_8192", kind="gemm", m=8192, n=8192, k=8192, ta=False, tb=False),
        # the weight gradient of a wide linear layer over a long minibatch
        dict(name="wgrad_4096", kind="wgrad", m=8192, n=2048, k=4096),
        # Range BN on its own, a middle shape of the benchmark's sweep
        dict(name="rangebn_14x256", kind="rangebn", rows=256 * 14 * 14, c=256, relu=True),
        # both copies of a gradient as another framework's backward hands it over
        dict(name="bifurcate_28x128", kind="quantize", rows=256 * 28 * 28, cols=128, what="bifurcate", per_channel=False),
        # the low-bit layer in training
        dict(name="ternary_28x128", kind="ternary", n=64, hw=28, c=128, k=128, r=3, samples=6),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _mult(rng, lo, hi, step):
    """A multiple of `step` between lo and hi, its logarithm spread evenly."""
    return int(min(hi, max(lo, step * round(_log(rng, lo, hi) / step))))


_POSITIONS = 256 * 56 * 56          # of the largest listed layer


def draw(rng):
    kind = rng.choice(("conv", "conv", "conv", "linear", "linear", "stack", "infer", "gemm", "wgrad", "rangebn", "quantize", "ternary"))
    if kind in ("conv", "ternary"):
        while True:
            c, k = (rng.choice((64, 128, 256, 512)) if rng.random() < 0.5 else _mult(rng, 32, 512, 32) for _ in range(2))
            hw, n, r = int(_log(rng, 5, 56.9)), int(_log(rng, 1, 256.9)), rng.choice((1, 3, 3))
            # at most the memory and the arithmetic of the listed layers of the kind
            cost = n * hw * hw * max(c, k) / (_POSITIONS * 64) + n * hw * hw * c * k * r * r / (4 * _POSITIONS * 64 * 64 * 9)
            if n * hw * hw >= 25 and cost <= (0.25 if kind == "ternary" else 1.0):
                break
        case = dict(kind=kind, n=n, hw=hw, c=c, k=k, r=r)
        return dict(case, samples=rng.randint(1, 8)) if kind == "ternary" else case
    if kind == "linear":
        return dict(kind=kind, batch=_mult(rng, 16, 4096, 16), cin=_mult(rng, 16, 4096, 16), cout=_mult(rng, 16, 4096, 16))
    if kind in ("stack", "infer"):
        mid = rng.choice((64, 96, 128))
        return dict(kind=kind, n=int(_log(rng, 2, 256.9 if kind == "stack" else 64.9)), hw=rng.randint(7, 28), c=rng.choice((128, 256)), mid=mid, k=4 * mid)
    if kind == "gemm":
        return dict(kind=kind, m=_mult(rng, 128, 8192, 16), n=_mult(rng, 128, 8192, 16), k=_mult(rng, 128, 8192, 16),
                    ta=rng.random() < 0.25, tb=rng.random() < 0.5)
    if kind == "wgrad":
        return dict(kind=kind, m=_mult(rng, 128, 8192, 16), n=_mult(rng, 128, 4096, 16), k=_mult(rng, 128, 4096, 16))
    if kind == "rangebn":
        c = rng.choice((64, 128, 256, 512, 2048, _mult(rng, 16, 2048, 4)))
        return dict(kind=kind, rows=int(_log(rng, 1000, min(_POSITIONS, _POSITIONS * 64 // c))), c=c, relu=rng.random() < 0.5)
    what = rng.choice(("nearest8", "stochastic8", "stochastic16", "bifurcate"))
    cols = rng.choice((64, 128, 256, 512, _mult(rng, 16, 2048, 4), rng.randint(16, 2048)))
    return dict(kind="quantize", rows=int(_log(rng, 64, _POSITIONS * 64 // cols)), cols=cols, what=what,
                per_channel=what != "bifurcate" and rng.random() < 0.4)


# ------------------------------------------------------------------ inputs
class _Inputs:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def normal(self, *shape, std=1.0):
        return torch.randn(shape, generator=self.g, device="cuda") * std

    def relu(self, *shape):
        return torch.randn(shape, generator=self.g, device="cuda").clamp_(min=0.0)

    def uniform(self, *shape, lo, hi):
        return torch.rand(shape, generator=self.g, device="cuda") * (hi - lo) + lo

    def filter(self, k, r, c):
        return self.normal(k, r, r, c, std=math.sqrt(2.0 / (r * r * c)))

    def affine(self, c):
        """gamma and beta of a Range BN some way into training."""
        return self.uniform(c, lo=0.5, hi=1.5), self.normal(c, std=0.1)

    def channels(self, rows, c):
        """Per-channel N(mu, sigma^2), mu ~ U(-1, 1), sigma ~ U(0.5, 2)."""
        mu, sigma = self.uniform(c, lo=-1.0, hi=1.0), self.uniform(c, lo=0.5, hi=2.0)
        return self.normal(rows, c).mul_(sigma).add_(mu)


def _conv(n, hw, c, k, r):
    return B.conv_desc(n, hw, hw, c, k, r, r, 1, (r - 1) // 2)


def _stack_convs(case):
    n, hw, c, mid, k = (case[f] for f in ("n", "hw", "c", "mid", "k"))
    return [_conv(n, hw, c, mid, 1), _conv(n, hw, mid, mid, 3), _conv(n, hw, mid, k, 1)]


def prepare(case, seed):
    i, kind, s = _Inputs(seed), case["kind"], dict(case=case)
    if kind == "conv":
        n, hw, c, k, r = (case[f] for f in ("n", "hw", "c", "k", "r"))
        s["layer"] = layer.QuantizedLayer(conv=_conv(n, hw, c, k, r), relu=True, seed=seed, tensor_id8=1, tensor_id16=1, keep_g=False)
        s.update(x=i.relu(n, hw, hw, c), w=i.filter(k, r, c), affine=i.affine(k), dy=i.normal(n, hw, hw, k, std=0.1))
    elif kind == "linear":
        b, cin, cout = case["batch"], case["cin"], case["cout"]
        s["layer"] = layer.QuantizedLayer(batch=b, in_features=cin, out_features=cout, relu=True, seed=seed, tensor_id8=1, tensor_id16=1, keep_g=False)
        bound = math.sqrt(6.0 / cin)
        s.update(x=i.normal(b, cin), w=i.uniform(cin, cout, lo=-bound, hi=bound), affine=i.affine(cout), dy=i.normal(b, cout, std=0.1))
    elif kind == "stack":
        n, hw, c, mid, k = (case[f] for f in ("n", "hw", "c", "mid", "k"))
        w = [i.filter(mid, 1, c), i.filter(mid, 3, mid), i.filter(k, 1, mid)]
        # (the gradient is a sum over the minibatch, not a mean: hence the small rate)
        s["stack"] = layer.QuantizedStack(_stack_convs(case), w, seed=seed, lr=1e-6)
        s.update(x=i.normal(n, hw, hw, c), dy=i.normal(n, hw, hw, k, std=0.1))
    elif kind == "infer":
        convs, prev, s["layers"] = _stack_convs(case), None, []
        for j, conv in enumerate(convs):
            last = j == len(convs) - 1
            prev = layer.QuantizedLayer(conv=conv, relu=True, input_from=prev, emit_codes=not last, keep_y=last, keep_z=last, keep_g=False)
            s["layers"].append(prev)
        s.update(x=i.normal(case["n"], case["hw"], case["hw"], case["c"]),
                 w=[i.filter(d.K, d.R, d.C) for d in convs], affine=[i.affine(d.K) for d in convs])
    elif kind == "gemm":
        m, n, k, ta, tb = (case[f] for f in ("m", "n", "k", "ta", "tb"))
        s["a"] = B.qbp_quantize_s8(i.normal(*((k, m) if ta else (m, k))))
        s["b"] = B.qbp_quantize_s8(i.normal(*((n, k) if tb else (k, n))))
        s["out"] = torch.empty((m, n), dtype=torch.float32, device="cuda")
    elif kind == "wgrad":
        m, n, k = case["m"], case["n"], case["k"]
        s["x"] = B.qbp_quantize_s8(i.normal(m, k))
        s["g"] = B.qbp_quantize_s16(i.normal(m, n, std=0.1), rounding=B.QBP_ROUND_STOCHASTIC, seed=seed, tensor_id=1, want=("hi", "lo"))[1:]
        s["dw"] = torch.empty((k, n), dtype=torch.float32, device="cuda")
    elif kind == "rangebn":
        rows, c = case["rows"], case["c"]
        s.update(x=i.channels(rows, c), affine=i.affine(c), dy=i.normal(rows, c, std=0.1))
        s.update(y=torch.empty_like(s["x"]), dx=torch.empty_like(s["x"]))
    elif kind == "quantize":
        rows, cols, what = case["rows"], case["cols"], case["what"]
        s.update(x=i.relu(rows, cols) if what == "nearest8" else i.normal(rows, cols, std=0.1), seed=seed)
    elif kind == "ternary":
        n, hw, c, k, r = (case[f] for f in ("n", "hw", "c", "k", "r"))
        s["layer"] = layer.TernarizedLayer(conv=_conv(n, hw, c, k, r), relu=True, seed=seed, samples=case["samples"])
        s.update(x=i.normal(n, hw, hw, c), w=i.filter(k, r, c), affine=i.affine(k), dy=i.normal(n, hw, hw, k, std=0.1))
    else:
        raise ValueError(kind)
    return s


# -------------------------------------------------------------------- a pass
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("conv", "linear", "ternary"):
        y = s["layer"].forward(s["x"], s["w"], *s["affine"])
        return (y, *s["layer"].backward(s["dy"]))
    if kind == "stack":
        t = s["stack"]
        dx = t.train_step(s["x"], s["dy"])
        return dict(y=t.layers[-1].y, dx=dx, w=t.w, gamma=t.gamma, beta=t.beta, vw=t.vw, vg=t.vg, vb=t.vb)
    if kind == "infer":
        a = s["x"]
        for q, w, (gamma, beta) in zip(s["layers"], s["w"], s["affine"]):
            a = q.forward(a if q.rq_in is None else None, w, gamma, beta)
        return a
    if kind == "gemm":
        return B.qbp_gemm_s8(*s["a"], *s["b"], transA=case["ta"], transB=case["tb"], out=s["out"])[1]
    if kind == "wgrad":
        hi, lo, qp = s["g"]
        return B.qbp_wgrad_s16(*s["x"], hi, lo, qp, dW=s["dw"])[1]
    if kind == "rangebn":
        gamma, beta = s["affine"]
        y, mean, vmin, vmax, _ = B.qbp_rangebn_fwd(s["x"], gamma, beta, relu=case["relu"], y=s["y"])
        return (y, *B.qbp_rangebn_bwd(s["dy"], s["x"], mean, vmin, vmax, gamma, beta, relu=case["relu"], dx=s["dx"]))
    what, x = case["what"], s["x"]
    if what == "bifurcate":
        return B.qbp_bifurcate(x, s["seed"], 1, 1)
    rounding = B.QBP_ROUND_NEAREST if what == "nearest8" else B.QBP_ROUND_STOCHASTIC
    if what == "stochastic16":
        return B.qbp_quantize_s16(x, granularity=int(case["per_channel"]), rounding=rounding, seed=s["seed"], tensor_id=1, want=("hi", "lo"))
    return B.qbp_quantize_s8(x, granularity=int(case["per_channel"]), rounding=rounding, seed=s["seed"], tensor_id=1)


# ------------------------------------------------------- what a pass cannot do without
def _layer_work(rows, cin, cout, taps):
    """x, w, dy read; y, dx, dw written (fp32).  Three products; the 16-bit operand of the third counts as two 8-bit ones."""
    macs = rows * cin * cout * taps
    return dict(bytes=8.0 * (rows * (cin + cout) + taps * cin * cout), flops=8.0 * macs)


def work(case):
    kind = case["kind"]
    if kind in ("conv", "ternary"):
        return _layer_work(case["n"] * case["hw"] ** 2, case["c"], case["k"], case["r"] ** 2)
    if kind == "linear":
        return _layer_work(case["batch"], case["cin"], case["cout"], 1)
    if kind in ("stack", "infer"):
        rows, c, mid, k = case["n"] * case["hw"] ** 2, case["c"], case["mid"], case["k"]
        weights = c * mid + 9 * mid * mid + mid * k
        if kind == "infer":
            return dict(bytes=4.0 * (rows * (c + k) + weights), flops=2.0 * rows * weights)
        # the step also reads and writes the weights and their momentum
        return dict(bytes=4.0 * (2 * rows * (c + k) + 4 * weights), flops=8.0 * rows * weights)
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return dict(bytes=float(m * k + k * n + 4 * m * n), flops=2.0 * m * n * k)
    if kind == "wgrad":
        m, n, k = case["m"], case["n"], case["k"]
        return dict(bytes=float(m * k + 2 * m * n + 4 * k * n), flops=4.0 * m * n * k)
    if kind == "rangebn":
        return dict(bytes=16.0 * case["rows"] * case["c"], flops=0.0)          # x, dy read; y, dx written
    out = dict(nearest8=1, stochastic8=1, stochastic16=2, bifurcate=3)[case["what"]]
    return dict(bytes=float((4 + out) * case["rows"] * case["cols"]), flops=0.0)


def tolerance(case):
    """Measured against the same path with Range BN in 64 bits (statistics and element formula) and the codes made from its
    result, over the listed cases and some fifty drawn ones; about four times the largest difference seen.

    Where a value that differs in its last bit is quantised, a few codes in a million land on the next one (a ternary code
    on the next of three), and what is computed from them moves by that step: hence the figures of the layers."""
    kind = case["kind"]
    if kind == "quantize":
        return "exact"                                   # codes and their parameters, bit for bit
    if kind in ("gemm", "wgrad"):
        return {"rel": 5e-7, "max": 1e-6}                # an exact integer times one fp32 scale
    if kind == "rangebn":
        return {"rel": 4e-7, "max": 3e-5}                # seen: 1e-7, 7e-6 (dx next to zero)
    if kind in ("conv", "linear"):
        return {"rel": 1.6e-3, "max": 0.75}              # seen: 4e-4, 0.19 (a layer gradient's element, one code apart); without a step 1e-7
    if kind == "ternary":
        return {"rel": 1e-3, "max": 0.5}                 # seen: 1e-7 and no step; one step in 10^5 elements is 1e-3
    if kind == "infer":
        return {"rel": 1e-3, "max": 0.15}                # seen: 2.5e-4, 0.04
    # stack: three layers of such steps forwards, and backwards every position at a channel's extreme carries the whole
    # channel's sum, so a step there moves many: seen up to 0.1 in the last layer's gradient, 0.004 in the first's.
    # Stated is the most that still tells a wrong gradient from a right one.
    return {"rel": 0.03, "max": 0.99}
