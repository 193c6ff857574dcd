"""The work that a user of the integer-only ViT library has it do, as cases that can be timed.

A case names an entry point (`kind`) and its sizes.  The kinds, and what each stands for in real use:

  vit        one forward of a ViT-family model on images that are on the device: batch inference
  vit_host   the same from host memory to host memory: a server answering requests
  swin       one forward of the Swin-shaped model (windows of 49 tokens, patch merging)
  block      one encoder block on its own: a user who composes a model of their own
  linear     a Dense layer with requantisation, residual port and int32 output: heads, adapters, other MLPs
  matmul     the batched products Q K^T and P V
  shiftmax, shiftgelu, layernorm   the row operators, on int8 or int32 rows

Everything is integer arithmetic, so every output is compared exactly.  The library computes forward passes only.
"""
import math

import numpy as np
import torch

from ivit_inputs import ExpParams, Scale
from ivit_inputs.gen import dyadic, make_block_input, make_image, make_swin, make_vit
from paper_2207_01405_b200 import binding

# (embedding width, heads, MLP width) of the repository's model shapes: DeiT-T, DeiT-S, ViT-B, ViT-L
WIDTHS = ((192, 3, 768), (384, 6, 1536), (768, 12, 3072), (1024, 16, 4096))
PATCH = 16
SWIN = dict(dims=(96, 192, 384, 768), depths=(2, 2, 6, 2), res=56, window=7, patch=4)


def listed():
    return [
        # one DeiT-T block on one image: the smallest call, all latency (the repository's configuration 0)
        dict(name="block_tiny_b1", kind="block", B=1, T=197, width=0, bias=False),
        # a whole DeiT-T forward of one image: interactive use, where launches count
        dict(name="vit_tiny_b1", kind="vit", B=1, img=224, width=0, depth=12, classes=1000, tokens=False),
        # DeiT-S from host memory to host memory at the batch size of the paper's latency table
        dict(name="vit_small_host_b8", kind="vit_host", B=8, img=224, width=1, depth=12, classes=1000),
        # an odd batch of odd-sized images (13 x 13 patches, 170 tokens), with the encoder's tokens as features
        dict(name="vit_small_208_b27_tokens", kind="vit", B=27, img=208, width=1, depth=12, classes=100, tokens=True),
        # DeiT-S at batch 64: the headline workload (configuration 1)
        dict(name="vit_small_b64", kind="vit", B=64, img=224, width=1, depth=12, classes=1000, tokens=False),
        # ViT-B at batch 128: throughput (configuration 2)
        dict(name="vit_base_b128", kind="vit", B=128, img=224, width=2, depth=12, classes=1000, tokens=False),
        # ViT-L at 384 x 384, batch 32, 577 tokens: long rows, the largest products (configuration 4, half of its
        # 24 equal blocks)
        dict(name="vit_large_384_b32", kind="vit", B=32, img=384, width=3, depth=12, classes=1000, tokens=False),
        # Swin-T at batch 64 with shifted windows (configuration 3): window attention with relative-position bias
        dict(name="swin_tiny_b64", kind="swin", B=64, shifted=True),
        # a Dense layer of its own: ragged rows, residual port
        dict(name="linear_12345x1536x768", kind="linear", M=12345, N=1536, K=768, res=True, i32=False),
        # Shiftmax straight on int32 accumulators of long rows
        dict(name="shiftmax_i32_18464x577", kind="shiftmax", rows=18464, d=577, i32=True),
        # ShiftGELU and I-LayerNorm on int8 rows, at the sizes of DeiT-S at batch 64 and ViT-B at batch 128
        dict(name="shiftgelu_12608x1536", kind="shiftgelu", rows=12608, cols=1536),
        dict(name="layernorm_25216x768", kind="layernorm", rows=25216, C=768, i32=False),
    ]


# ---- sizes drawn from the same ranges ----

def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["vit", "vit", "vit", "vit_host", "swin", "block", "block", "linear", "matmul", "shiftmax",
                       "shiftgelu", "layernorm"])
    biggest = max(work(c)["flops"] for c in listed())
    while True:
        if kind in ("vit", "vit_host"):
            c = dict(kind=kind, B=_log_int(rng, 1, 128), img=PATCH * rng.randint(8, 24), width=rng.randrange(4),
                     depth=rng.randint(4, 12), classes=4 * rng.randint(2, 250))
            if kind == "vit":
                c["tokens"] = rng.random() < 0.3
        elif kind == "swin":
            c = dict(kind=kind, B=_log_int(rng, 1, 64), shifted=rng.random() < 0.5)
        elif kind == "block":
            c = dict(kind=kind, B=_log_int(rng, 1, 512), T=_log_int(rng, 9, 600), width=rng.randrange(4),
                     bias=rng.random() < 0.3)
            if c["B"] * c["T"] > 40000:
                continue
        elif kind == "linear":
            c = dict(kind=kind, M=_log_int(rng, 1, 40000), N=16 * rng.randint(4, 256), K=16 * rng.randint(4, 256),
                     res=rng.random() < 0.4, i32=rng.random() < 0.2)
            c["res"] = c["res"] and not c["i32"]
        elif kind == "matmul":
            T, d = _log_int(rng, 9, 600), rng.choice([32, 64, 128])
            c = dict(kind=kind, nb=_log_int(rng, 3, 768), T=T, d=d, transB=rng.random() < 0.5)
        elif kind == "shiftmax":
            c = dict(kind=kind, rows=_log_int(rng, 64, 80000), d=_log_int(rng, 9, 1200), i32=rng.random() < 0.5)
        elif kind == "shiftgelu":
            c = dict(kind=kind, rows=_log_int(rng, 64, 40000), cols=16 * rng.randint(12, 320))
        else:
            c = dict(kind=kind, rows=_log_int(rng, 64, 40000), C=4 * rng.randint(12, 512), i32=rng.random() < 0.3)
        if work(c)["flops"] <= biggest and work(c)["bytes"] < 2e9:
            return c


# ---- inputs ----

def _up16(n):
    return (n + 15) // 16 * 16


class _Make:
    """Device tensors made from the seed alone."""

    def __init__(self, seed):
        self.dev = torch.device("cuda", torch.cuda.current_device())
        self.g = torch.Generator(device=self.dev)
        self.g.manual_seed(seed)

    def normal(self, *shape):
        return torch.randn(*shape, generator=self.g, device=self.dev)

    def i8(self, std, *shape):
        """int8 values of the given standard deviation; rows padded to a multiple of 16 bytes."""
        ld = _up16(shape[-1])
        x = self.normal(*shape[:-1], ld).mul_(std).round_().clamp_(-128, 127).to(torch.int8)
        return x[..., :shape[-1]]

    def i32(self, std, *shape):
        ld = (shape[-1] + 3) // 4 * 4
        return self.normal(*shape[:-1], ld).mul_(std).round_().to(torch.int32)[..., :shape[-1]]

    def channel_scale(self, n, ratio):
        """One requantisation ratio per channel, spread by a tenth around `ratio`."""
        r = (1.0 + 0.1 * self.normal(n).clamp_(-4, 4).double().cpu().numpy()) * ratio
        ms = [dyadic(x) for x in r]
        return binding.DevScale(Scale(np.array([m for m, _ in ms], np.int32), np.array([s for _, s in ms], np.uint8)),
                                self.dev)

    def tensor_scale(self, ratio):
        return binding.DevScale(Scale(*dyadic(ratio)), self.dev)


def prepare(case, seed):
    seed = int(seed) % (1 << 31)
    kind = case["kind"]
    dev = torch.device("cuda", torch.cuda.current_device())
    st = {"case": case}
    if kind in ("vit", "vit_host"):
        D, heads, H = WIDTHS[case["width"]]
        model = make_vit(seed, case["B"], case["img"], D, heads, H, case["depth"], patch=PATCH, classes=case["classes"])
        image = torch.from_numpy(make_image(seed, case["B"], case["img"]))
        st["model"] = binding.DeviceVit(model, dev)
        if kind == "vit":
            st["ctx"] = binding.Context(dev.index)
            st["ws"] = st["model"].workspace()
            st["image"] = image.to(dev)
            if case["tokens"]:
                st["tokens"] = torch.empty((case["B"] * model.T, D), dtype=torch.int8, device=dev)
        else:
            # a server: its own stream, pinned buffers, the entry point's graph replay switched on
            stream = torch.cuda.Stream(device=dev)
            st["ctx"] = binding.Context(dev.index, stream)
            st["ctx"].set_host_graph(True)
            st["ws"] = st["model"].host_workspace()
            st["image"] = image.pin_memory()
            st["logits"] = torch.empty((case["B"], case["classes"]), dtype=torch.int32).pin_memory()
            torch.cuda.current_stream(dev).synchronize()   # the weights are uploaded on the current stream
        return st
    st["ctx"] = binding.Context(dev.index)
    if kind == "swin":
        st["model"] = binding.DeviceSwin(make_swin(seed, case["B"], shifted=case["shifted"]), dev)
        st["image"] = torch.from_numpy(make_image(seed, case["B"], 224)).to(dev)
        st["ws"] = st["model"].workspace()
        return st
    if kind == "block":
        D, heads, H = WIDTHS[case["width"]]
        T = case["T"]
        blk = make_vit(seed, case["B"], 32, D, heads, H, 1, patch=PATCH, classes=16).blocks[0]
        blk.B, blk.T = case["B"], T
        if case["bias"]:   # relative-position bias, one matrix per head, a quarter of the scores' own deviation
            rng = np.random.default_rng(seed)
            std = 0.25 * math.sqrt(D // heads) * 32.0 * 32.0
            blk.attn_bias = np.rint(std * rng.standard_normal((heads, T, T), dtype=np.float32)).astype(np.int32)
        st["block"] = binding.DeviceBlock(blk, dev)
        st["x"] = torch.from_numpy(make_block_input(seed, case["B"], T, D)).to(dev)
        st["ws"] = st["block"].workspace()
        return st
    mk = _Make(seed)
    if kind == "linear":
        M, N, K = case["M"], case["N"], case["K"]
        acc_std = math.sqrt(K) * 32.0 * 33.0
        st["a"], st["w"] = mk.i8(32.0, M, K), mk.i8(33.0, N, K)
        st["bias"] = mk.i32(0.1 * acc_std, N)
        st["scale"] = mk.channel_scale(N, (2000.0 if case["i32"] else 32.0) / acc_std)
        if case["res"]:
            st["res"], st["res_scale"] = mk.i8(20.0, M, N), mk.tensor_scale(0.9)
    elif kind == "matmul":
        nb, T, d = case["nb"], case["T"], case["d"]
        if case["transB"]:
            st["a"], st["b"] = mk.i8(32.0, nb, T, d), mk.i8(32.0, nb, T, d)
            st["scale"] = mk.tensor_scale(30.0 / (math.sqrt(d) * 32.0 * 32.0))
        else:   # probabilities (non-negative, rows that sum to about 128) times values
            p = mk.normal(nb, T, _up16(T)).mul_(2.5)[..., :T].softmax(-1).mul_(128.0).clamp_(0, 127)
            st["a"] = torch.zeros((nb, T, _up16(T)), dtype=torch.int8, device=mk.dev)[..., :T]
            st["a"].copy_(p.round_().to(torch.int8))
            st["b"] = mk.i8(32.0, nb, T, d)
            st["scale"] = mk.tensor_scale(1.0 / (128.0 * 0.45))
    elif kind == "shiftmax":
        rows, d = case["rows"], case["d"]
        st["p"] = ExpParams(17, 15)
        if case["i32"]:
            st["x"] = mk.i32(8192.0, rows, d)
            st["pre"] = mk.tensor_scale(30.0 / 8192.0)
        else:
            st["x"] = mk.i8(30.0, rows, d)
    elif kind == "shiftgelu":
        st["x"] = mk.i8(33.0, case["rows"], case["cols"])
        st["p"], st["post"] = ExpParams(33, 23), mk.tensor_scale(1.0 / (128.0 * 0.9))
    elif kind == "layernorm":
        rows, C = case["rows"], case["C"]
        st["x"] = mk.i32(3000.0, rows, C) if case["i32"] else mk.i8(21.0, rows, C)
        st["gamma"] = mk.channel_scale(C, 32.0 * math.sqrt(C) / 2.0 ** 20)
        st["beta"] = mk.i32(3.2, C)
    else:
        raise ValueError(kind)
    return st


def run(state):
    c, ctx = state["case"], state["ctx"]
    kind = c["kind"]
    if kind == "vit":
        logits = ctx.vit_forward(state["model"], state["image"], workspace=state["ws"], tokens=state.get("tokens"))
        return (logits, state["tokens"]) if c["tokens"] else logits
    if kind == "vit_host":
        binding.vit_forward_host(ctx, state["model"], state["image"], state["logits"], state["ws"])
        ctx.stream.synchronize()   # the caller reads the logits next
        return state["logits"]
    if kind == "swin":
        return binding.swin_forward(ctx, state["model"], state["image"], workspace=state["ws"])
    if kind == "block":
        return ctx.block_forward(state["block"], state["x"], workspace=state["ws"])
    if kind == "linear":
        return ctx.linear(state["a"], state["w"], state["bias"], state["scale"], res=state.get("res"),
                          res_scale=state.get("res_scale"), out_dtype=binding.I32 if c["i32"] else binding.I8)
    if kind == "matmul":
        return ctx.matmul(state["a"], state["b"], c["transB"], state["scale"])
    if kind == "shiftmax":
        return ctx.shiftmax(state["x"], state["p"], pre=state.get("pre"))
    if kind == "shiftgelu":
        return ctx.shiftgelu(state["x"], state["p"], state["post"])
    return ctx.layernorm(state["x"], state["gamma"], state["beta"])


# ---- what a pass cannot do without ----

def _block_work(B, T, D, heads, H):
    """int8 operations (2 per multiply-accumulate) and weight bytes of one encoder block."""
    M = B * T
    ops = 2 * M * D * 3 * D + 4 * B * T * T * D + 2 * M * D * D + 4 * M * D * H
    weights = 4 * D * D + 2 * D * H
    return ops, weights


def work(case):
    kind = case["kind"]
    if kind in ("vit", "vit_host"):
        D, heads, H = WIDTHS[case["width"]]
        B, img, classes = case["B"], case["img"], case["classes"]
        np_ = (img // PATCH) ** 2
        ops, weights = _block_work(B, np_ + 1, D, heads, H)
        kpe = 3 * PATCH * PATCH
        flops = case["depth"] * ops + 2 * B * np_ * kpe * D + 2 * B * D * classes
        nbytes = case["depth"] * weights + kpe * D + np_ * D + D * classes + B * 3 * img * img + 4 * B * classes
        if case.get("tokens"):
            nbytes += B * (np_ + 1) * D
    elif kind == "swin":
        B, res, flops, nbytes = case["B"], SWIN["res"], 0, 0
        C0, kpe = SWIN["dims"][0], 3 * SWIN["patch"] ** 2
        flops += 2 * B * res * res * kpe * C0
        nbytes += B * 3 * 224 * 224 + kpe * C0 + 4 * B * 1000 + 1000 * SWIN["dims"][-1]
        for s, (C, depth) in enumerate(zip(SWIN["dims"], SWIN["depths"])):
            r = res >> s
            T = SWIN["window"] ** 2
            ops, weights = _block_work(B * r * r // T, T, C, C // 32, 4 * C)
            flops += depth * ops
            nbytes += depth * weights
            if s + 1 < len(SWIN["dims"]):
                flops += 2 * B * (r // 2) ** 2 * 4 * C * 2 * C
                nbytes += 8 * C * C
        flops += 2 * B * SWIN["dims"][-1] * 1000
    elif kind == "block":
        D, heads, H = WIDTHS[case["width"]]
        flops, weights = _block_work(case["B"], case["T"], D, heads, H)
        nbytes = weights + 2 * case["B"] * case["T"] * D + (4 * heads * case["T"] ** 2 if case["bias"] else 0)
    elif kind == "linear":
        M, N, K = case["M"], case["N"], case["K"]
        flops = 2 * M * N * K
        nbytes = M * K + N * K + 9 * N + M * N * (4 if case["i32"] else 1) + (M * N if case["res"] else 0)
    elif kind == "matmul":
        nb, T, d = case["nb"], case["T"], case["d"]
        flops = 2 * nb * T * T * d
        nbytes = nb * (2 * T * d + T * T)
    elif kind == "shiftmax":
        flops = 10 * case["rows"] * case["d"]
        nbytes = case["rows"] * case["d"] * (5 if case["i32"] else 2)
    elif kind == "shiftgelu":
        flops = 3 * case["rows"] * case["cols"]
        nbytes = 2 * case["rows"] * case["cols"]
    else:
        flops = 8 * case["rows"] * case["C"]
        nbytes = case["rows"] * case["C"] * (5 if case["i32"] else 2) + 9 * case["C"]
    return {"bytes": float(nbytes), "flops": float(flops)}


def tolerance(case):
    return "exact"   # integer arithmetic: there is one correct output
