"""The measured workloads: what a training program has this library do with the activation maps that it saves.

A pass of a "map", "planes", "line" or "volume" case is what happens to one saved map in one training step: it is
compressed in the forward pass and rebuilt in the backward pass, through the calls a program makes (`binding.Codec`,
`binding.PlaneGroupCodec`, and the C ABI's 3-D calls, which have no buffer-owning class).  A pass of a "step" case is a
whole forward and backward pass of a small convolutional network under `autograd.DivisionCache` with mask-caching ReLUs.

Maps are post-ReLU-like (half the values exactly zero, a smooth component of a few pixels, 10 % noise) or
post-normalisation-like (smooth component plus N(0, 1)); tokens of 1-D maps are normal with a scale per token.
"""
import math

import torch
import torch.nn.functional as F

from paper_2208_04187_b200 import autograd as dv
from paper_2208_04187_b200 import binding

# sides of the planes that convolutional networks produce from 32, 64 and 224 pixel inputs
USUAL_SIDES = (4, 7, 8, 14, 16, 28, 32, 56, 64, 112)
MAX_ELEMENTS = 64 * 64 * 112 * 112          # the largest listed map
BYTES = {"f32": 4, "bf16": 2}


def listed():
    return [
        # the smallest map of the configurations: what a call costs
        dict(name="small_32x32", kind="map", n=8, c=64, h=32, w=32, block=8, qbits=2, x="f32", lfc="f32", relu=True),
        # first stage of a CIFAR network, batch 128
        dict(name="cifar_32x32", kind="map", n=128, c=64, h=32, w=32, block=8, qbits=2, x="f32", lfc="f32", relu=False),
        # the five resolutions of an ImageNet network, batch 64: the stem (largest map of all), then stages 2 to 4;
        # the 7 x 7 planes have odd rows
        dict(name="stem_112x112", kind="map", n=64, c=64, h=112, w=112, block=8, qbits=2, x="f32", lfc="f32", relu=True),
        dict(name="stage_28x28", kind="map", n=64, c=512, h=28, w=28, block=8, qbits=2, x="f32", lfc="f32", relu=True),
        dict(name="stage_14x14", kind="map", n=64, c=1024, h=14, w=14, block=8, qbits=2, x="f32", lfc="f32", relu=True),
        dict(name="stage_7x7", kind="map", n=64, c=2048, h=7, w=7, block=8, qbits=2, x="f32", lfc="f32", relu=True),
        # a wide residual network in mixed precision: bfloat16 maps, 4-bit codes
        dict(name="wide_bf16_32x32", kind="map", n=128, c=160, h=32, w=32, block=4, qbits=4, x="bf16", lfc="bf16", relu=True),
        # inputs whose sides are no power of two leave odd planes wider than a warp (600 pixels / 8)
        dict(name="odd_75x75", kind="map", n=32, c=64, h=75, w=75, block=8, qbits=2, x="f32", lfc="bf16", relu=True),
        # one bfloat16 pair of parameters per plane, the grouping of the paper's byte count
        dict(name="planes_56x56", kind="planes", n=64, c=256, h=56, w=56, block=8, qbits=2, x="f32", lfc="f32", relu=True),
        # transformer tokens: batch 32, 512 tokens of 768 numbers
        dict(name="tokens_768", kind="line", n=32, c=512, w=768, block=8, qbits=4, x="f32", lfc="f32"),
        # a video or volume network: 16 frames
        dict(name="volume_16x56x56", kind="volume", n=8, c=64, d=16, h=56, w=56, block=8, qbits=2, x="f32", lfc="f32", relu=True),
        # one training step of a small network: convolution, batch norm and ReLU, four times over
        dict(name="step_conv_net", kind="step", n=32, c=64, h=56, w=56, layers=4, block=8, qbits=2),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _types(rng):
    x = rng.choice(("f32", "f32", "bf16"))
    return x, rng.choice((x, x, "bf16"))


def draw(rng):
    kind = rng.choices(("map", "planes", "line", "volume", "step"), (14, 3, 3, 2, 1))[0]
    if kind == "step":
        return dict(kind="step", n=rng.choice((8, 16, 24, 32)), c=rng.choice((32, 48, 64)), h=rng.randint(20, 56), w=rng.randint(20, 56),
                    layers=rng.randint(2, 4), block=8, qbits=rng.choice((2, 2, 4)))
    x, lfc = _types(rng)
    block, qbits = rng.choice((8, 8, 8, 4, 16)), rng.choice((2, 2, 4, 8))
    size = _log_uniform(rng, 1 << 19, MAX_ELEMENTS)             # elements of the map, about
    if kind == "line":
        c, w = rng.choice((64, 128, 196, 197, 256, 384, 512, 577)), rng.choice((96, 192, 384, 512, 768, 1000, 1024))
        block = rng.choice((8, 8, 16, 64))
        return dict(kind="line", n=max(1, min(64, size // (c * w))), c=c, w=w, block=block, qbits=qbits, x=x, lfc=lfc)
    if kind == "volume":
        d, side = rng.choice((4, 8, 13, 16, 32)), rng.choice((7, 14, 28, 56, rng.randint(7, 56)))
        c = 8 * _log_uniform(rng, 1, 16)
        return dict(kind="volume", n=max(1, min(16, size // (c * d * side * side))), c=c, d=d, h=side, w=side, block=rng.choice((4, 8)),
                    qbits=qbits, x=x, lfc=lfc, relu=rng.random() < 0.7)
    h = rng.choice(USUAL_SIDES) if rng.random() < 0.6 else _log_uniform(rng, 5, 112)
    w = h if rng.random() < 0.8 else _log_uniform(rng, 5, 112)
    n = rng.choice((8, 16, 24, 32, 50, 64, 96, 128))
    c = min(2048, max(8, size // (n * h * w) // 8 * 8))
    while n > 1 and n * c * h * w > MAX_ELEMENTS:
        n -= 1
    return dict(kind=kind, n=n, c=c, h=h, w=w, block=block, qbits=qbits, x=x, lfc=lfc, relu=rng.random() < 0.7)


def _activation(gen, planes, h, w, relu):
    """planes x h x w values with the statistics named at the top."""
    lattice = torch.randn(planes, 1, -(-h // 4) + 1, -(-w // 4) + 1, device="cuda", generator=gen)
    g = F.interpolate(lattice, size=(h, w), mode="bilinear", align_corners=False).view(planes, h, w)
    noise = torch.randn(planes, h, w, device="cuda", generator=gen)
    if not relu:
        return g + noise
    keep = torch.randint(0, 2, (planes, h, w), device="cuda", generator=gen, dtype=torch.uint8)
    return g.add_(noise, alpha=0.1).abs_().mul_(keep)


class _ConvNet(torch.nn.Module):
    def __init__(self, c, layers):
        super().__init__()
        body = []
        for i in range(layers):
            body += [torch.nn.Conv2d(3 if i == 0 else c, c, 3, padding=1, bias=False), torch.nn.BatchNorm2d(c), torch.nn.ReLU()]
        self.body = torch.nn.Sequential(*body)

    def forward(self, x):
        return self.body(x)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind, n, c, w = case["kind"], case["n"], case["c"], case["w"]
    if kind == "step":
        torch.manual_seed(seed)
        model = dv.to_division_modules(_ConvNet(c, case["layers"])).cuda().train()
        images = torch.randn(n, 3, case["h"], w, device="cuda", generator=gen)
        return dict(kind=kind, model=model, images=images, block=case["block"], qbits=case["qbits"], seed=seed,
                    weight=torch.randn(n, c, case["h"], w, device="cuda", generator=gen) / (n * case["h"] * w))
    dtype = binding.torch_dtype(case["x"])
    types = (case["x"], case["lfc"])
    if kind == "line":
        scale = 1 + torch.rand(n, c, 1, 1, device="cuda", generator=gen)
        x = (torch.randn(n, c, 1, w, device="cuda", generator=gen) * scale).to(dtype)
        return dict(kind=kind, x=x, seed=seed, codec=binding.Codec(n, c, 1, w, case["block"], case["qbits"], *types))
    h = case["h"]
    if kind == "volume":
        d = case["d"]
        x = _activation(gen, n * c * d, h, w, case["relu"]).view(n, c, d, h, w).to(dtype)
        desc = binding.make_desc_3d(n, c, d, h, w, case["block"], case["qbits"], *types)
        layout = binding.div_compressed_bytes_3d(desc)
        return dict(kind=kind, x=x, seed=seed, desc=desc, blob=torch.zeros(int(layout.total_bytes), dtype=torch.uint8, device="cuda"),
                    workspace=torch.zeros(int(layout.workspace_bytes), dtype=torch.uint8, device="cuda"))
    x = _activation(gen, n * c, h, w, case["relu"]).view(n, c, h, w).to(dtype)
    codec = binding.Codec if kind == "map" else binding.PlaneGroupCodec
    return dict(kind=kind, x=x, seed=seed, codec=codec(n, c, h, w, case["block"], case["qbits"], *types))


def run(state):
    kind = state["kind"]
    if kind == "step":
        model = state["model"]
        model.zero_grad(set_to_none=True)
        with dv.DivisionCache(block=state["block"], qbits=state["qbits"], seed=state["seed"]):
            out = model(state["images"])
        (out * state["weight"]).sum().backward()
        return [out.detach()] + [p.grad for p in model.parameters()]
    if kind == "volume":
        x, blob, ws = state["x"], state["blob"], state["workspace"]
        stream = binding.current_stream_handle()
        binding.div_compress_3d(state["desc"], x.data_ptr(), blob.data_ptr(), blob.numel(), ws.data_ptr(), ws.numel(), state["seed"], stream)
        rebuilt = torch.empty_like(x)
        binding.div_decompress_3d(state["desc"], blob.data_ptr(), blob.numel(), rebuilt.data_ptr(), stream)
        return blob, rebuilt
    codec = state["codec"]
    blob = codec.compress(state["x"], seed=state["seed"])
    return blob, codec.decompress()


def _sides(case):
    """Elements of the map, low-frequency values, and pairs of parameters (with the bytes of a pair)."""
    up = lambda a: -(-a // case["block"])  # noqa: E731
    n, c = case["n"], case["c"]
    dims = [case[k] for k in ("d", "h", "w") if k in case]
    pairs = (n * c, 4) if case["kind"] == "planes" else (n, 8)
    return n * c * math.prod(dims), n * c * math.prod(up(a) for a in dims), pairs


def work(case):
    if case["kind"] == "step":
        # three convolutions' worth of arithmetic a layer; per layer the forward pass reads a map and writes three
        # (convolution, normalisation, ReLU), two of them compressed, the backward pass reads as many and their gradients
        maps = case["n"] * case["h"] * case["w"] * case["c"]
        flops = sum(2 * 9 * maps * (3 * 2 if i == 0 else case["c"] * 3) for i in range(case["layers"]))
        return dict(bytes=case["layers"] * maps * 4 * 12, flops=flops)
    elements, tiles, (pairs, pair_bytes) = _sides(case)
    blob = tiles * BYTES[case["lfc"]] + -(-elements * case["qbits"] // 32) * 4 + pairs * pair_bytes
    # per element: block sum, residual, two extremes, four operations of the quantiser; three to rebuild
    return dict(bytes=2 * (elements * BYTES[case["x"]] + blob), flops=11 * elements)


def tolerance(case):
    # the network around the maps is cuDNN's, whose weight gradients add up in no fixed order (3e-7 between two runs)
    if case["kind"] == "step":
        return {"rel": 1e-5}
    # the output format fixes every rounding and the order of every sum (see include/division.h): bytes and floats
    # are the same for every correct implementation
    return "exact"
