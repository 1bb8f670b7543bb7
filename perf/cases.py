"""Timed cases of the library: what flow-model programs ask of the inverse convolution and its neighbours.

A case is one operation on one shape, called through `paper_2410_14634_b200.binding`:

  forward   x = f^-1(y)                                            density evaluation, no gradients
  sample    y = f(x)                                               drawing images (the masked convolution)
  layer     forward, then backward with both gradients             the layer alone in a training step
  train     the same two calls with the log-determinant folded in  the layer in a likelihood's training step
  flow      the layer with Actnorm and the 1x1 convolution, both directions
  bf16      forward and backward with bfloat16 activations

Ranges (listed() picks points of them, draw() spreads over them):

  images of 1 to 4 channels, sides 16 to 256: MNIST, CIFAR, ImageNet crops before any squeeze, and the image-side axis of
    the method's ablation; kernels 2, 3, 5 and, up to 64 pixels a side, the kernel-size axis's 7, 9, 11
  squeezed levels of 5 to 96 channels, sides 4 to 64, at most 16384 values an image: the levels a multi-scale flow on images
    of up to 64x64 pixels runs (12x32x32, 24x16x16, 48x16x16, 96x8x8 ...); kernels 2, 3, 5
  batches of 1 (one sample, one request) to 256 (training)
"""
import math

import torch

from paper_2410_14634_b200 import binding

OPS = ("forward", "sample", "layer", "train", "flow", "bf16")


def _case(name, op, B, C, H, W, k):
    return {"name": name, "op": op, "B": B, "C": C, "H": H, "W": W, "k": k}


def listed():
    return [
        # one CIFAR-sized image drawn through one layer: the latency of a single small call
        _case("sample_one_image", "sample", 1, 3, 32, 32, 3),
        # an MNIST training batch
        _case("mnist_train", "train", 256, 1, 28, 28, 3),
        # one step of a flow on CIFAR images at the batch size the method's model tables use
        _case("cifar_flow_step", "flow", 100, 3, 32, 32, 3),
        # CIFAR activations kept in bfloat16, a large training batch
        _case("cifar_bf16", "bf16", 256, 3, 32, 32, 3),
        # the first squeezed level of a CIFAR flow, training
        _case("squeezed12_train", "train", 256, 12, 16, 16, 3),
        # density evaluation of a small batch at an odd size and channel count (cropped images, a split level)
        _case("ragged6_forward", "forward", 37, 6, 45, 51, 3),
        # many channels, a large kernel, a large batch: the heaviest arithmetic
        _case("wide48_layer", "layer", 128, 48, 16, 16, 5),
        # the deepest level of a 64-pixel flow
        _case("wide96_train", "train", 64, 96, 8, 8, 3),
        # drawing a batch of images, a many-channel level
        _case("wide48_sample", "sample", 128, 48, 16, 16, 3),
        # 64-pixel images with the wider kernel
        _case("image64_layer", "layer", 16, 3, 64, 64, 5),
        # the largest images of the image-side axis
        _case("image256_layer", "layer", 32, 3, 256, 256, 3),
        # the kernel-size axis
        _case("kernel7_layer", "layer", 32, 3, 32, 32, 7),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(c):
    w = work(c)
    return w["bytes"] / 6.5e12 + w["flops"] / 50e12


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        op = rng.choice(OPS)
        if rng.random() < 0.4:
            C = rng.choice((1, 2, 3, 3, 4))
            k = rng.choice((2, 3, 3, 3, 3, 5, 5, 7, 9, 11))
            largest = 256 if k <= 5 else 64
            H = _log_uniform(rng, 16, largest)
        else:
            C = rng.choice((6, 8, 12, 12, 16, 24, 24, 32, 48, 48, 64, 96, 2 * rng.randint(3, 48)))
            k = rng.choice((2, 3, 3, 3, 3, 5))
            largest = min(64, int(math.sqrt(16384 / C)))
            H = _log_uniform(rng, 4, largest)
        # square images mostly, as datasets have them; crops and odd sides otherwise
        W = H if rng.random() < 0.6 else min(largest, max(4, _log_uniform(rng, H / 2, H * 2)))
        B = _log_uniform(rng, 1, 256)
        case = {"op": op, "B": B, "C": C, "H": H, "W": W, "k": k}
        if _cost(case) <= most and B * C * H * W <= 32 * 3 * 256 * 256:
            return case


def prepare(case, seed):
    """Standard-normal activations, and a kernel whose recursion is stable as a trained layer's is: small off-centre taps,
    the channel diagonal of the tap on the pixel itself near one."""
    B, C, H, W, k = (case[n] for n in ("B", "C", "H", "W", "k"))
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32)

    w = normal(C, C, k, k) * (0.15 / math.sqrt(C * k * k))
    centre = torch.tril(w[:, :, k - 1, k - 1], -1)
    w[:, :, k - 1, k - 1] = centre + torch.diag(0.8 + 0.4 * torch.rand(C, generator=g, device="cuda"))
    state = {"op": case["op"], "w": w}
    store = torch.bfloat16 if case["op"] == "bf16" else torch.float32
    state["in"] = normal(B, C, H, W).to(store)
    if case["op"] in ("layer", "train", "flow", "bf16"):
        state["grad"] = normal(B, C, H, W).to(store)
    if case["op"] == "train":
        state["grad_logdet"] = torch.full((1,), -0.25, device="cuda")
    if case["op"] == "flow":
        state["s"] = 0.8 + 0.4 * torch.rand(C, generator=g, device="cuda")
        state["b"] = 0.1 * normal(C)
        # 1x1 convolutions start as random rotations
        state["V"] = torch.linalg.qr(normal(C, C))[0].contiguous()
    return state


def run(state):
    op, w, t = state["op"], state["w"], state["in"]
    if op == "forward":
        return binding.invconv_forward(t, w)
    if op == "sample":
        return binding.masked_conv_forward(t, w)
    if op == "layer":
        x = binding.invconv_forward(t, w)
        grad_y, grad_w = binding.invconv_backward(state["grad"], x, w)
        return x, grad_y, grad_w
    if op == "train":
        x, logdet = binding.invconv_forward_logdet(t, w)
        grad_y, grad_w = binding.invconv_backward_logdet(state["grad"], x, w, state["grad_logdet"])
        return x, logdet, grad_y, grad_w
    if op == "flow":
        s, b, V = state["s"], state["b"], state["V"]
        x, u, logdet = binding.invconv_flow_step_forward(t, w, s, b, V)
        return x, u, logdet, binding.invconv_flow_step_backward(state["grad"], x, w, s, b, V)
    x = binding.invconv_forward_bf16(t, w)
    grad_y, grad_w = binding.invconv_backward_bf16(state["grad"], x, w)
    return x, grad_y, grad_w


def work(case):
    """Each input read once and each output written once; two operations a multiply-add of the taps."""
    op, C, k = case["op"], case["C"], case["k"]
    n = case["B"] * C * case["H"] * case["W"]
    weights = 4 * C * C * k * k
    taps = 2 * n * C * k * k
    if op in ("forward", "sample"):
        return {"bytes": 8 * n + weights, "flops": taps}
    # one solve forward; one solve and one correlation backward, which reads the gradient and x and writes a gradient
    value = 2 if op == "bf16" else 4
    byts, flops = 5 * value * n + 3 * weights, 3 * taps
    if op == "flow":
        # u is written beside x; the channel mix runs forward, transposed, and in its own gradient
        byts, flops = byts + value * n + 12 * C * C, flops + 6 * n * C
    return {"bytes": byts, "flops": flops}


def tolerance(case):
    if case["op"] in ("forward", "sample"):
        return {"rel": 1e-5}
    if case["op"] == "bf16":
        return {"rel": 1e-2}
    # from 8 channels on grad_w may take its two operands rounded to tf32 (see the header); below, the sums over batch and
    # pixels are 32-bit sums of up to millions of terms that cancel
    return {"rel": 1e-3 if case["C"] >= 8 else 1e-4}
