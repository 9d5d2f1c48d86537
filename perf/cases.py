"""The work that users of this package have it do, as cases that can be timed.

Each case is one call, or one training step, through the package's public
Python entry points.  ``listed()`` names twelve of them; ``draw(rng)`` gives
others from the same ranges.  The kinds, and what each stands for:

  fwd     ``conv2d_fwd``: filtering images that are in hand (smoothing,
          sharpening, feature extraction); one image or a batch, FP32 or BF16.
  train   ``conv2d`` under autograd: the forward pass and both gradients of a
          learnable depthwise filter, one training step's share of this layer.
  ragged  ``BatchedPlan``: forward and both gradients of a list of images of
          different sizes, each with its own filter, in one launch; the plan is
          made and uploaded once, as a program that keeps its images would.
  up      ``upsample_conv2d``: enlarge an image and filter it in one pass.
  updb    ``UpsampleBatchedPlan``: the same over a list of images, each with
          its own scale and filter.
  sep     ``conv2d_separable``: a Gaussian blur with its two 1-D factors.
  gray    ``gray_conv2d``: RGB to grayscale, then the filter.
  dense   the dense 64 -> 64 channel 3 x 3 filter: forward, input gradient and
          filter gradient, one training step's share of this layer.

Pixels are uniform [0, 1), upstream gradients normal(0, 1), depthwise filters
normal(0, 0.1), dense filters normal(0, 0.05), as in ``workloads.py``.
"""
import math
import random

import torch

import paper_2504_01266_gb300 as giga

DEVICE = "cuda"
OPS_ALL = 7  # forward | input gradient | filter gradient
LAPLACIAN = ((-1.0, -1.0, -1.0), (-1.0, 8.0, -1.0), (-1.0, -1.0, -1.0))
GRAY = (0.299, 0.587, 0.114)

# Upper ends of the drawn sizes: none costs more than the largest listed case.
MAX_PIXELS = 8 * 3 * 4096 * 4096
MAX_TAPS = 8 * 3 * 4096 * 4096 * 225


def listed():
    return [
        # one small grayscale photo, the 5 x 5 Gaussian: latency and launches
        dict(name="fwd_512_k5", kind="fwd", N=1, C=1, H=512, W=512, K=5, border="zero",
             dtype="float32"),
        # a training step on a few small odd-sized crops: latency and launches
        dict(name="train_crops_k3", kind="train", N=4, C=3, H=257, W=251, K=3, border="clamp",
             dtype="float32"),
        # a batch of large images, the largest filter of the size sweep
        dict(name="fwd_4096_k15", kind="fwd", N=8, C=3, H=4096, W=4096, K=15, border="clamp",
             dtype="float32"),
        # a training step on medium images, the 7 x 7 learnable filter
        dict(name="train_2048_k7", kind="train", N=16, C=3, H=2048, W=2048, K=7, border="zero",
             dtype="float32"),
        # the same with BF16 storage and a larger filter
        dict(name="train_2048_k9_bf16", kind="train", N=32, C=3, H=2048, W=2048, K=9,
             border="zero", dtype="bfloat16"),
        # a training step on photos whose rows do not start on 16-byte boundaries
        dict(name="train_photos_k3", kind="train", N=4, C=3, H=1801, W=2399, K=3, border="clamp",
             dtype="float32"),
        # images of many sizes and filters in one launch
        dict(name="ragged_16", kind="ragged", n=16, lo=64, hi=4096, border="zero",
             dtype="float32", layout_seed=3),
        # a 4K photo enlarged four times and sharpened
        dict(name="up_4k_s4_k3", kind="up", N=1, C=3, H=2160, W=3840, K=3, scale=4,
             border="zero", dtype="float32"),
        # a list of photos enlarged by different factors, different filters
        dict(name="updb_24", kind="updb", n=24, lo=64, hi=1024, border="zero",
             dtype="float32", layout_seed=5),
        # a wide Gaussian blur of odd-sized photos
        dict(name="sep_photos_k15", kind="sep", N=4, C=3, H=2731, W=4094, K=15, border="clamp",
             dtype="float32"),
        # photos to grayscale, then the Laplacian
        dict(name="gray_4096_k3", kind="gray", N=4, H=4096, W=4096, K=3, border="zero",
             dtype="float32"),
        # a training step of the dense layer
        dict(name="dense_1024", kind="dense", N=8, H=1024, W=1024),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["fwd", "fwd", "train", "train", "train", "ragged", "up", "updb", "sep",
                       "gray", "dense"])
    dtype = rng.choice(["float32", "float32", "float32", "bfloat16"])
    border = rng.choice(["zero", "clamp"])
    if kind == "ragged":
        return dict(kind=kind, n=rng.randint(3, 18), lo=64, hi=_log(rng, 512, 4096),
                    border=border, dtype=dtype, layout_seed=rng.randrange(1 << 20))
    if kind == "updb":
        return dict(kind=kind, n=rng.randint(4, 24), lo=64, hi=_log(rng, 256, 1024),
                    border=border, dtype=dtype, layout_seed=rng.randrange(1 << 20))
    if kind == "dense":
        while True:
            c = dict(kind=kind, N=rng.randint(1, 8), H=_log(rng, 64, 1024), W=_log(rng, 64, 1024))
            if c["N"] * c["H"] * c["W"] >= 1 << 14:
                return c
    if kind == "up":
        scale = rng.randint(2, 8)
        N, K = rng.randint(1, 2), rng.choice([3, 3, 5, 7, 9, 11])
        side = int(math.sqrt(MAX_PIXELS / 2 / (3 * N))) // scale
        return dict(kind=kind, N=N, C=3, H=_log(rng, 64, min(2160, side)),
                    W=_log(rng, 64, min(3840, side)), K=K, scale=scale, border=border,
                    dtype=dtype)
    while True:
        N = _log(rng, 1, 16)
        H, W = _log(rng, 64, 4096), _log(rng, 64, 4096)
        if rng.random() < 0.4:  # rows of whole 16-byte groups; the rest as they come
            W = max(64, W // 8 * 8)
        if kind == "gray":
            C, K = 3, rng.choice([3, 5, 7, 9])
        elif kind == "sep":
            C, K = rng.choice([1, 3, 3]), rng.choice([3, 5, 7, 9, 11, 15])
        elif kind == "fwd":
            C, K = rng.choice([1, 3, 3]), rng.choice([3, 3, 5, 5, 7, 9, 11, 15, 21, 31])
        else:
            C, K = rng.choice([1, 3, 3]), rng.choice([3, 3, 5, 5, 7, 7, 9, 11, 15])
        px = N * C * H * W
        cost = px * {"train": 3 * K * K, "fwd": K * K, "sep": 2 * K, "gray": K * K}[kind]
        if px <= MAX_PIXELS / (2 if kind == "train" else 1) and cost <= MAX_TAPS / 2:
            break
    if kind == "gray":
        return dict(kind=kind, N=N, H=H, W=W, K=K, border=border, dtype=dtype)
    return dict(kind=kind, N=N, C=C, H=H, W=W, K=K, border=border, dtype=dtype)


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device=DEVICE).manual_seed(2504 + int(seed))


def _uniform(g, shape, dtype):
    return torch.rand(shape, generator=g, device=DEVICE).to(dtype)


def _normal(g, shape, std, dtype=torch.float32):
    return (torch.randn(shape, generator=g, device=DEVICE) * std).to(dtype)


def _dtype(case):
    return getattr(torch, case["dtype"])


def _layout(case):
    """(C, H, W, K, scale) of every image of a list: part of the case, not of the seed."""
    r = random.Random(case["layout_seed"])
    return [(3, r.randint(case["lo"], case["hi"]), r.randint(case["lo"], case["hi"]),
             r.choice([3, 5, 9, 11]), r.randint(2, 8)) for _ in range(case["n"])]


def _inputs(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "dense":
        N, H, W = case["N"], case["H"], case["W"]
        b = torch.bfloat16
        return dict(x=_uniform(g, (N, H, W, 64), b), w=_normal(g, (64, 3, 3, 64), 0.05, b),
                    dy=_normal(g, (N, H, W, 64), 1.0, b))
    dt = _dtype(case)
    if kind == "ragged":
        return [dict(x=_uniform(g, (C, H, W), dt), dy=_normal(g, (C, H, W), 1.0, dt),
                     w=_normal(g, (C, K, K), 0.1)) for C, H, W, K, _ in _layout(case)]
    if kind == "updb":
        return [dict(x=_uniform(g, (C, H, W), dt), w=_normal(g, (C, K, K), 0.1), scale=s)
                for C, H, W, K, s in _layout(case)]
    N, H, W, K = case["N"], case["H"], case["W"], case["K"]
    C = case.get("C", 3)
    if kind == "sep":
        ax = torch.arange(K, dtype=torch.float64) - (K - 1) / 2
        f = torch.exp(-(ax ** 2) / (2.0 * (K / 6.0) ** 2))
        f = (f / f.sum()).to(torch.float32).to(DEVICE)
        return dict(x=_uniform(g, (N, C, H, W), dt), wcol=f.repeat(C, 1), wrow=f.repeat(C, 1))
    if kind == "gray" or kind == "up":
        x = _uniform(g, (N, 3, H, W), dt)
        c = 1 if kind == "gray" else C
        if K == 3:  # the sharpening filter
            w = torch.tensor(LAPLACIAN, device=DEVICE).repeat(c, 1, 1)
        else:
            w = _normal(g, (c, K, K), 0.1)
        return dict(x=x, w=w)
    d = dict(x=_uniform(g, (N, C, H, W), dt), w=_normal(g, (C, K, K), 0.1))
    if kind == "train":
        d["dy"] = _normal(g, (N, C, H, W), 1.0, dt)
    return d


def prepare(case, seed):
    state = dict(case=case, t=_inputs(case, seed))
    t = state["t"]
    if case["kind"] == "train":
        t["x"].requires_grad_(True)
        t["w"].requires_grad_(True)
    elif case["kind"] == "ragged":
        for im in t:
            im.update(y=torch.empty_like(im["x"]), dx=torch.empty_like(im["x"]),
                      dw=torch.empty_like(im["w"]))
        state["plan"] = giga.BatchedPlan(t, OPS_ALL, case["border"], dtype=_dtype(case))
        state["plan"].upload()
    elif case["kind"] == "updb":
        for im in t:
            C, H, W = im["x"].shape
            s = im["scale"]
            im["y"] = torch.empty((C, H * s, W * s), dtype=im["x"].dtype, device=DEVICE)
        state["plan"] = giga.UpsampleBatchedPlan(t, case["border"], dtype=_dtype(case))
        state["plan"].upload()
    return state


def run(state):
    case, t = state["case"], state["t"]
    kind, border = case["kind"], case.get("border")
    if kind == "fwd":
        return giga.conv2d_fwd(t["x"], t["w"], border)
    if kind == "train":
        y = giga.conv2d(t["x"], t["w"], border)
        dx, dw = torch.autograd.grad(y, (t["x"], t["w"]), t["dy"])
        return dict(y=y, dx=dx, dw=dw)
    if kind == "ragged":
        state["plan"].run()
        return [dict(y=im["y"], dx=im["dx"], dw=im["dw"]) for im in t]
    if kind == "up":
        return giga.upsample_conv2d(t["x"], t["w"], case["scale"], border)
    if kind == "updb":
        state["plan"].run()
        return [im["y"] for im in t]
    if kind == "sep":
        return giga.conv2d_separable(t["x"], t["wcol"], t["wrow"], border)
    if kind == "gray":
        return giga.gray_conv2d(t["x"], t["w"], border)
    y = giga.dense_conv2d_fwd(t["x"], t["w"])
    dx = giga.dense_conv2d_bwd_input(t["dy"], t["w"])
    dw = giga.dense_conv2d_bwd_filter(t["x"], t["dy"])
    return dict(y=y, dx=dx, dw=dw)


# -------------------------------------------------------------------- work

def work(case):
    """Each input read once and each output written once; two operations per
    multiply-add of the definition.  The upsampled filter with K > 3 in FP32
    promises the bits of the two calls (upsample, then filter), so it needs the
    definition's K * K; otherwise the taps that land on one input pixel are one."""
    kind = case["kind"]
    if kind == "dense":
        px = case["N"] * case["H"] * case["W"]
        return dict(bytes=3 * px * 256, flops=3 * px * 2 * 64 * 64 * 9)
    es = 2 if case["dtype"] == "bfloat16" else 4
    if kind == "ragged":
        px = [(C * H * W, K) for C, H, W, K, _ in _layout(case)]
        return dict(bytes=sum(p for p, _ in px) * 4 * es, flops=sum(p * 6 * K * K for p, K in px))
    if kind in ("up", "updb"):
        if kind == "up":
            images = [(case["N"] * case["C"], case["H"], case["W"], case["K"], case["scale"])]
        else:
            images = _layout(case)
        b = f = 0
        for C, H, W, K, s in images:
            # input rows under a window, averaged over the s output rows of an input row
            t = K if K > 3 and es == 4 else sum(
                (u + K // 2) // s - (u - K // 2) // s + 1 for u in range(s)) / s
            b += C * H * W * (1 + s * s) * es
            f += C * H * W * s * s * 2 * t * t
        return dict(bytes=b, flops=f)
    px = case["N"] * case["H"] * case["W"]
    K = case["K"]
    if kind == "gray":
        return dict(bytes=px * 4 * es, flops=px * (2 * K * K + 5))
    px *= case["C"]
    if kind == "sep":
        return dict(bytes=px * 2 * es, flops=px * 4 * K)
    if kind == "fwd":
        return dict(bytes=px * 2 * es, flops=px * 2 * K * K)
    return dict(bytes=px * 5 * es, flops=px * 6 * K * K)


# ------------------------------------------------------------------- exact

def _pad(x, r, border):
    return torch.nn.functional.pad(x, (r, r, r, r),
                                   mode="replicate" if border == "clamp" else "constant")


def _filter64(x, w, border):
    """The definition in FP64: x (N, C, H, W), w (C, K, K)."""
    K, (H, W) = w.shape[-1], x.shape[-2:]
    xp = _pad(x, K // 2, border)
    y = torch.zeros_like(x)
    for a in range(K):
        for b in range(K):
            y.addcmul_(xp[..., a:a + H, b:b + W], w[:, a, b].view(1, -1, 1, 1))
    return y


def _input_grad64(dy, w, border):
    K, (H, W) = w.shape[-1], dy.shape[-2:]
    r = K // 2
    g = dy.new_zeros(dy.shape[:2] + (H + 2 * r, W + 2 * r))
    for a in range(K):
        for b in range(K):
            g[..., a:a + H, b:b + W].addcmul_(dy, w[:, a, b].view(1, -1, 1, 1))
    if border == "clamp" and r:  # what was read from a clamped place returns to the edge pixel
        g[..., r, :] += g[..., :r, :].sum(-2)
        g[..., r + H - 1, :] += g[..., r + H:, :].sum(-2)
        g[..., r] += g[..., :r].sum(-1)
        g[..., r + W - 1] += g[..., r + W:].sum(-1)
    return g[..., r:r + H, r:r + W].contiguous()


def _filter_grad64(x, dy, K, border):
    H, W = x.shape[-2:]
    xp = _pad(x, K // 2, border)
    dw = x.new_zeros((x.shape[1], K, K))
    for a in range(K):
        for b in range(K):
            dw[:, a, b] = (dy * xp[..., a:a + H, b:b + W]).sum((0, 2, 3))
    return dw


def _upsample64(x, s):
    return x.repeat_interleave(s, -2).repeat_interleave(s, -1)


def exact(case, seed):
    t = _inputs(case, seed)
    kind, border = case["kind"], case.get("border")
    if kind == "ragged":
        out = []
        for im in t:
            x, dy, w = im["x"].double()[None], im["dy"].double()[None], im["w"].double()
            out.append(dict(y=_filter64(x, w, border)[0], dx=_input_grad64(dy, w, border)[0],
                            dw=_filter_grad64(x, dy, w.shape[-1], border)))
        return out
    if kind == "updb":
        return [_filter64(_upsample64(im["x"].double()[None], im["scale"]), im["w"].double(),
                          border)[0] for im in t]
    t = {k: v.double() for k, v in t.items()}
    if kind == "fwd":
        return _filter64(t["x"], t["w"], border)
    if kind == "train":
        return dict(y=_filter64(t["x"], t["w"], border),
                    dx=_input_grad64(t["dy"], t["w"], border),
                    dw=_filter_grad64(t["x"], t["dy"], case["K"], border))
    if kind == "up":
        return _filter64(_upsample64(t["x"], case["scale"]), t["w"], border)
    if kind == "sep":
        return _filter64(t["x"], t["wcol"][:, :, None] * t["wrow"][:, None, :], border)
    if kind == "gray":
        x = t["x"]
        return _filter64(GRAY[0] * x[:, :1] + GRAY[1] * x[:, 1:2] + GRAY[2] * x[:, 2:],
                         t["w"], border)
    x, w, dy = t["x"], t["w"], t["dy"]
    N, H, W, _ = x.shape
    y, dx, dw = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(w)
    for n in range(N):  # one image at a time; taps as 64 x 64 matrices
        xp = torch.nn.functional.pad(x[n], (0, 0, 1, 1, 1, 1))
        dp = torch.nn.functional.pad(dy[n], (0, 0, 1, 1, 1, 1))
        for a in range(3):
            for b in range(3):
                xs = xp[a:a + H, b:b + W].reshape(-1, 64)
                y[n].view(-1, 64).addmm_(xs, w[:, a, b].t())
                dx[n].view(-1, 64).addmm_(dp[2 - a:2 - a + H, 2 - b:2 - b + W].reshape(-1, 64),
                                          w[:, a, b])
                dw[:, a, b] += dy[n].reshape(-1, 64).t() @ xs
    return dict(y=y, dx=dx, dw=dw)
