"""What a user of this package has it do, as cases that can be timed and compared.

A case is a dict of plain values; `path` names the public entry point it goes through and the other keys give
the sizes and options.  `listed()` holds the named cases, `draw(rng)` makes one more of the same ranges,
`prepare(case, seed)` builds what a program has in hand before the call (packed images, plan, activations),
`run(state)` is one pass, `work(case)` what a pass cannot do without, `tolerance(case)` how far another correct
implementation may be off.

  product   one decode product with its token-shift mix (rwkvq_gemv): a program that issues products one by one
  step      all projections of a stack for one token of a batch, one launch (rwkvq_step_run): decoding
  host      the same step with activations from and outputs to page-locked host memory (rwkvq_step_run_host)
  blocks    a chain of whole blocks, every stage reading what the one before wrote (BlockStack.run_step)
  prefill   the eight projections of a layer over a prompt (rwkvq_gemm_prefill_grouped)
  convert   one layer's weights from fp16 to packed images: proxy, choice of format, quantizers
  segments  the proxy for every tile or every output channel of a matrix (rwkvq_proxy_segments)
  mu        one layer's token-shift vectors quantized against calibration activations
"""
from __future__ import annotations

import math

import torch

from paper_2505_03803_b200 import binding as B
from paper_2505_03803_b200 import inputs
from paper_2505_03803_b200 import stack

TORCH = {"f16": torch.float16, "bf16": torch.bfloat16, "f32": torch.float32}


def listed():
    return [
        # The smallest call: a 512 x 512 matrix for one token.  All launch latency and host work.
        dict(name="product_512_b1", path="product", oc=512, ic=512, format="sq", batch=1, mu=True, y="f32"),
        # Single-stream decoding on the 1.6B-class stack: 96 dependent stages of 5.5 MB each.
        dict(name="step_1p6b_b1", path="step", d=2048, h=7168, layers=24, entries=64, batch=1),
        # Single-stream and small-batch decoding on the 7B-class stack.
        dict(name="step_7b_b1", path="step", d=4096, h=14336, layers=32, entries=64, batch=1),
        dict(name="step_7b_b8", path="step", d=4096, h=14336, layers=32, entries=64, batch=8),
        # Batched decoding on the 14B-class stack with 256-entry codebooks: the largest step.
        dict(name="step_14b_b16", path="step", d=4096, h=14336, layers=61, entries=256, batch=16),
        # A serving loop whose activations and results live in host memory.
        dict(name="host_7b_b8", path="host", d=4096, h=14336, layers=32, entries=64, batch=8),
        # Whole blocks (recurrence, gates, normalisation inside the step), two sequences.
        dict(name="blocks_1p6b_b2", path="blocks", d=2048, h=7168, layers=4, entries=64, batch=2),
        # A long prompt through one 7B-class layer, and a short ragged one through a 1.6B-class layer with bf16 results.
        dict(name="prefill_7b_m2048", path="prefill", d=4096, h=14336, tokens=2048, entries=64, heavy=5, y="f32"),
        dict(name="prefill_1p6b_m203", path="prefill", d=2048, h=7168, tokens=203, entries=64, heavy=2, y="bf16"),
        # Conversion of a checkpoint, one 7B-class layer: seven matrices end up scalar-, one vector-quantized.
        dict(name="convert_7b", path="convert", d=4096, h=14336, entries=64, heavy=2, iters=10),
        # The proxy at the granularity of a codebook tile.
        dict(name="segments_4096_bf16", path="segments", oc=4096, ic=4096, rows=256, cols=256, dtype="bf16"),
        # The five token-shift vectors of a 7B-class layer, 128 calibration samples.
        dict(name="mu_4096", path="mu", d=4096, samples=128, entries=64, iters=10),
    ]


def _log(rng, lo, hi, step=1):
    """A multiple of `step` in [lo, hi], spread over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)) * step))


def draw(rng):
    path = rng.choice(["product", "step", "step", "host", "blocks", "prefill", "prefill", "convert", "segments", "mu"])
    entries = rng.choice([64, 64, 256])
    if path == "product":
        fmt = rng.choice(["sq", "sq", "vq6", "vq8"])
        ro, ri = (16, 128) if fmt == "sq" else (256, 256)
        return dict(path=path, oc=_log(rng, 256, 14336, ro), ic=_log(rng, 256, 14336, ri), format=fmt, batch=rng.randint(1, 16),
                    mu=rng.random() < 0.6, y=rng.choice(["f32", "f32", "f16"]))
    if path in ("step", "host"):
        d = _log(rng, 512, 4096, 128)
        h = int(d * 3.5) // 128 * 128
        layers = _log(rng, 2, 32)
        return dict(path=path, d=d, h=h, layers=layers, entries=entries, batch=_log(rng, 1, 16))
    if path == "blocks":
        d = _log(rng, 512, 4096, 512)           # BlockStack lets the proxy choose: both formats have to take the shape
        return dict(path=path, d=d, h=d * 7 // 2, layers=rng.randint(2, 5), entries=entries, batch=_log(rng, 1, 16))
    if path == "prefill":
        d = _log(rng, 512, 4096, 128)
        return dict(path=path, d=d, h=int(d * 3.5) // 128 * 128, tokens=_log(rng, 17, 2048), entries=entries, heavy=rng.randint(0, 7),
                    y=rng.choice(["f32", "bf16"]))
    if path == "convert":
        d = _log(rng, 512, 4096, 256)
        return dict(path=path, d=d, h=d * 7 // 2 // 256 * 256, entries=64 if d > 2048 else entries, heavy=rng.choice([0, 1, 2, 3, 4, 6]),
                    iters=rng.choice([5, 10]))
    if path == "segments":
        dtype = rng.choice(["f16", "bf16", "f32"])
        oc, ic = _log(rng, 256, 4096), _log(rng, 512, 4096, 8)
        rows, cols = rng.choice([(256, 256), (128, 128), (64, 256), (1, ic)])
        if dtype == "f32" and rows * cols > 32768:
            rows = 128
        return dict(path=path, oc=oc, ic=ic, rows=rows, cols=cols, dtype=dtype)
    return dict(path=path, d=_log(rng, 768, 5120, 128), samples=rng.choice([32, 64, 128, 200]), entries=entries, iters=rng.choice([5, 10]))


# ---- shapes -------------------------------------------------------------------------------------------------
def _method(kind, oc, ic):
    """Heavy-tailed matrices are vector-quantized where the format allows the shape."""
    return B.RWKVQ_VQ if kind == "student" and oc % 256 == 0 and ic % 256 == 0 else B.RWKVQ_SQ


def _bits(method, entries):
    return 3 if method == B.RWKVQ_SQ else 6 if entries == 64 else 8


def _stack_shapes(case):
    """(layer, name, oc, ic, has_mu, stage, method) of a stack: each matrix is heavy-tailed with probability 0.1."""
    out = []
    for l in range(case["layers"]):
        for (name, oc, ic, mu, stage) in inputs.layer_shapes(case["d"], case["h"]):
            kind = inputs.weight_kind(inputs.seed_of("stack", case["d"], l, name))
            out.append((l, name, oc, ic, mu, 4 * l + stage, _method(kind, oc, ic)))
    return out


def _layer_shapes(case):
    """(name, oc, ic, has_mu, kind) of one layer whose matrix number `heavy` is the heavy-tailed one."""
    return [(name, oc, ic, mu, "student" if i == case["heavy"] else "gauss")
            for i, (name, oc, ic, mu, _) in enumerate(inputs.layer_shapes(case["d"], case["h"]))]


# ---- inputs -------------------------------------------------------------------------------------------------
def _gen(seed, *parts):
    return torch.Generator(device="cuda").manual_seed(inputs.seed_of("cases", seed, *parts) & 0x7FFFFFFF)


def _activations(gen, rows, cols, dtype, outliers=8):
    """N(0, 1) with a few channels twenty times as large, as RWKV activations have them."""
    x = torch.randn((rows, cols), generator=gen, device="cuda")
    x[:, torch.randint(cols, (outliers,), generator=gen, device="cuda")] *= 20.0
    return x.to(dtype)


class _Images:
    """Packed images: two matrices (and two token-shift vectors) of every shape are drawn and quantized, and each
    request gets a buffer of its own with one of them."""

    def __init__(self, seed, entries):
        self.seed, self.entries, self.made, self.asked = seed, entries, {}, {}
        self.ws = torch.zeros(B.rwkvq_quantize_workspace_bytes(), dtype=torch.uint8, device="cuda")

    def _new(self, method, oc, ic, n):
        desc = B.rwkvq_desc_for(oc, ic, method, _bits(method, self.entries))
        image = torch.zeros(int(desc.image_bytes), dtype=torch.uint8, device="cuda")
        seed = inputs.seed_of("image", self.seed, method, oc, ic, n)
        if oc == 1:
            w = torch.rand((1, ic), generator=_gen(seed), device="cuda").to(torch.float16)
        else:
            w = stack.gen_weight_device(seed, oc, ic, "gauss" if method == B.RWKVQ_SQ else "student")
        B.rwkvq_quantize_dev_async(w, oc, ic, method, _bits(method, self.entries), image, self.ws, kmeans_iters=2, seed=seed & 0xFFFF)
        return desc, image

    def get(self, method, oc, ic):
        k = self.asked.get((method, oc, ic), 0)
        self.asked[(method, oc, ic)] = k + 1
        key = (method, oc, ic, k % 2)
        if key not in self.made:
            self.made[key] = self._new(method, oc, ic, k % 2)
            return self.made[key]
        desc, image = self.made[key]
        return desc, image.clone()


def _aligned(n):
    return (n + 255) // 256 * 256


class _Step:
    """A stack's images, its activations and outputs in one buffer each, and the plan of its step."""

    plan = None

    def __init__(self, case, seed):
        self.batch, b = case["batch"], case["batch"]
        shapes, images, gen = _stack_shapes(case), _Images(seed, case["entries"]), _gen(seed, "act")
        act = sum(_aligned(2 * b * ic) * (2 if mu else 1) for (_, _, _, ic, mu, _, _) in shapes)
        self.act = torch.zeros(act, dtype=torch.uint8, device="cuda")
        self.y = torch.zeros(sum(_aligned(4 * b * oc) for (_, _, oc, *_r) in shapes) // 4, dtype=torch.float32, device="cuda")
        self.keep, a, o = [], 0, 0
        for (l, name, oc, ic, mu, stage, method) in shapes:
            e = dict(stage=stage, mu_desc=None, mu=None, xprev=None)
            e["desc"], e["W"] = images.get(method, oc, ic)
            for key in ("x", "xprev") if mu else ("x",):
                e[key] = self.act[a:a + 2 * b * ic].view(torch.float16).view(b, ic)
                e[key].copy_(_activations(gen, b, ic, torch.float16))
                a += _aligned(2 * b * ic)
            if mu:
                e["mu_desc"], e["mu"] = images.get(B.RWKVQ_VQ, 1, ic)
            e["y"] = self.y[o:o + b * oc].view(b, oc)
            o += _aligned(4 * b * oc) // 4
            self.keep.append(e)
        ops = B.make_ops(self.keep)
        self.plan = torch.zeros(B.rwkvq_step_plan_bytes(ops, b), dtype=torch.uint8, device="cuda")
        B.rwkvq_step_plan(ops, b, self.plan)

    def __del__(self):
        if self.plan is not None:
            B.rwkvq_step_plan_release(self.plan)


class _Layer:
    """One layer's images, the prompt's activations for each product, outputs and workspaces."""

    def __init__(self, case, seed):
        images, gen, m = _Images(seed, case["entries"]), _gen(seed, "prompt"), case["tokens"]
        self.tokens, self.y_dtype = m, B.RWKVQ_F32 if case["y"] == "f32" else B.RWKVQ_BF16
        self.keep, shared = [], {}
        for (name, oc, ic, mu, kind) in _layer_shapes(case):
            e = dict(mu_desc=None, mu=None, xprev0=None)
            e["desc"], e["W"] = images.get(_method(kind, oc, ic), oc, ic)
            # R, K, V and G read the same sequence, as do the two input projections of channel mixing
            group = name[:2] if name not in ("tm_o", "cm_v") else name
            if group not in shared:
                shared[group] = (_activations(gen, m, ic, torch.bfloat16), _activations(gen, 1, ic, torch.bfloat16))
            e["X"] = shared[group][0]
            if mu:
                e["mu_desc"], e["mu"] = images.get(B.RWKVQ_VQ, 1, ic)
                e["xprev0"] = shared[group][1]
            e["Y"] = torch.zeros((m, oc), dtype=TORCH[case["y"]], device="cuda")
            e["workspace"] = torch.empty(B.rwkvq_prefill_workspace_bytes(e["desc"], m, mu), dtype=torch.uint8, device="cuda")
            self.keep.append(e)
        self.ops, self.alive = B.make_prefill_ops(self.keep)


class _State:
    pass


def prepare(case, seed):
    path = case["path"]
    if path == "step":
        return path, _Step(case, seed)
    if path == "host":
        s = _Step(case, seed)
        s.act_host = s.act.cpu().pin_memory()
        s.y_host = torch.zeros(s.y.numel() * 4, dtype=torch.uint8).pin_memory()
        return path, s
    if path == "prefill":
        return path, _Layer(case, seed)
    if path == "blocks":
        s = stack.BlockStack(case["d"], case["h"], case["layers"], case["entries"], case["batch"], tag="blocks/%d" % seed)
        s.x0.copy_(_activations(_gen(seed, "token"), case["batch"], case["d"], torch.float16))
        return path, s
    s, gen = _State(), _gen(seed, "inputs")
    if path == "product":
        b, oc, ic = case["batch"], case["oc"], case["ic"]
        method = B.RWKVQ_SQ if case["format"] == "sq" else B.RWKVQ_VQ
        images = _Images(seed, 64 if case["format"] == "vq6" else 256)
        s.batch, (s.desc, s.W) = b, images.get(method, oc, ic)
        s.x, s.xprev, s.mu_desc, s.mu = _activations(gen, b, ic, torch.float16), None, None, None
        if case["mu"]:
            s.xprev = _activations(gen, b, ic, torch.float16)
            s.mu_desc, s.mu = images.get(B.RWKVQ_VQ, 1, ic)
        s.y = torch.zeros((b, oc), dtype=TORCH[case["y"]], device="cuda")
        s.ws = torch.zeros(max(256, B.rwkvq_gemv_workspace_bytes(s.desc, b)), dtype=torch.uint8, device="cuda")
    elif path == "convert":
        s.entries, s.iters, s.seed = case["entries"], case["iters"], seed & 0xFFFF
        shapes = _layer_shapes(case)
        s.w = [stack.gen_weight_device(inputs.seed_of("convert", seed, i), oc, ic, kind) for i, (_, oc, ic, _, kind) in enumerate(shapes)]
        s.proxy_ws = torch.empty(B.rwkvq_proxy_workspace_bytes(len(s.w)), dtype=torch.uint8, device="cuda")
        s.ws = torch.zeros(B.rwkvq_quantize_workspace_bytes(), dtype=torch.uint8, device="cuda")
        # the threshold a program sets for its checkpoint: between the two kinds of matrices
        pc, _, _ = B.rwkvq_proxy_select(s.w, 4, math.inf, math.inf, s.proxy_ws)
        heavy = pc[case["heavy"]]
        s.tau = 0.5 * (heavy + max(p for i, p in enumerate(pc) if i != case["heavy"] and p < heavy))
        # one image buffer per matrix, large enough for either format
        s.images = [torch.zeros(max(int(B.rwkvq_desc_for(oc, ic, m, _bits(m, s.entries)).image_bytes) for m in (B.RWKVQ_SQ, B.RWKVQ_VQ)),
                                dtype=torch.uint8, device="cuda") for (_, oc, ic, _, _) in shapes]
    elif path == "segments":
        w = torch.randn((case["oc"], case["ic"]), generator=gen, device="cuda") * 0.02
        # one channel in ten heavy-tailed: tiles and channels differ in their proxies
        w[::10] *= 1.0 / torch.rand((w[::10].shape[0], case["ic"]), generator=gen, device="cuda").clamp_min(1e-3).sqrt()
        s.w, s.rows, s.cols = w.to(TORCH[case["dtype"]]), case["rows"], case["cols"]
    else:
        d, n = case["d"], case["samples"]
        s.entries, s.iters, s.seed = case["entries"], case["iters"], seed & 0xFFFF
        offsets = torch.randn(d, generator=gen, device="cuda") * 0.5
        s.samples = [torch.randn((n, d), generator=gen, device="cuda") + offsets for _ in range(5)]
        s.mu = [torch.rand((1, d), generator=gen, device="cuda").to(torch.float16) for _ in range(5)]
        s.rep_sq = [torch.empty(d, dtype=torch.float32, device="cuda") for _ in range(5)]
        desc = B.rwkvq_desc_for(1, d, B.RWKVQ_VQ, _bits(B.RWKVQ_VQ, s.entries))
        s.images = [torch.zeros(int(desc.image_bytes), dtype=torch.uint8, device="cuda") for _ in range(5)]
        s.ws = torch.zeros(B.rwkvq_quantize_workspace_bytes(), dtype=torch.uint8, device="cuda")
    return path, s


# ---- one pass -----------------------------------------------------------------------------------------------
def run(state):
    path, s = state
    if path == "product":
        B.rwkvq_gemv(s.desc, s.W, s.mu_desc, s.mu, s.x, s.xprev, s.batch, s.y, s.ws)
        return s.y
    if path == "step":
        B.rwkvq_step_run(s.plan)
        return s.y
    if path == "host":
        B.rwkvq_step_run_host(s.plan, s.act_host, s.act, s.y, s.y_host)
        torch.cuda.current_stream().synchronize()       # the results are read on the host
        return s.y_host.view(torch.float32)
    if path == "blocks":
        s.run_step()
        return [s.out_r, s.out_v] + [o.xprev for o in s.ops if o.xprev is not None] + [st[k] for st in s.states for k in ("a", "b", "p")]
    if path == "prefill":
        B.rwkvq_gemm_prefill_grouped(s.ops, s.tokens, s.y_dtype)
        return [e["Y"] for e in s.keep]
    if path == "convert":
        pc, pf, phi = B.rwkvq_proxy_select(s.w, 4, s.tau, math.inf, s.proxy_ws)
        for i, w in enumerate(s.w):
            m = int(phi[i])
            B.rwkvq_quantize_dev_async(w, w.shape[0], w.shape[1], m, _bits(m, s.entries), s.images[i], s.ws, kmeans_iters=s.iters, seed=s.seed + i)
        status = B.rwkvq_quantize_check(s.ws)
        return [pc, pf, phi, status] + s.images
    if path == "segments":
        return B.rwkvq_proxy_segments(s.w, s.rows, s.cols, 4, 8.0, math.inf)
    for i in range(5):
        B.rwkvq_calib_representative(s.samples[i], 1.0, rep_sq=s.rep_sq[i])
        B.rwkvq_quantize_dev_async(s.mu[i], 1, s.mu[i].shape[1], B.RWKVQ_VQ, _bits(B.RWKVQ_VQ, s.entries), s.images[i], s.ws,
                                   elem_weight=s.rep_sq[i], kmeans_iters=s.iters, seed=s.seed + i)
    return s.images + s.rep_sq + [B.rwkvq_quantize_check(s.ws)]


# ---- what a pass cannot do without --------------------------------------------------------------------------
def _stream(method, oc, ic, entries):
    return int(B.rwkvq_desc_for(oc, ic, method, _bits(method, entries)).stream_bytes)


def work(case):
    path = case["path"]
    if path == "product":
        b, oc, ic, e = case["batch"], case["oc"], case["ic"], 64 if case["format"] == "vq6" else 256
        n = _stream(B.RWKVQ_SQ if case["format"] == "sq" else B.RWKVQ_VQ, oc, ic, e) + 2 * b * ic + b * oc * TORCH[case["y"]].itemsize
        return {"bytes": n + (_stream(B.RWKVQ_VQ, 1, ic, e) + 2 * b * ic if case["mu"] else 0), "flops": 2 * b * oc * ic}
    if path in ("step", "host"):
        b, n, f = case["batch"], 0, 0
        for (_, _, oc, ic, mu, _, method) in _stack_shapes(case):
            n += _stream(method, oc, ic, case["entries"]) + 2 * b * ic + 4 * b * oc
            n += _stream(B.RWKVQ_VQ, 1, ic, case["entries"]) + 2 * b * ic if mu else 0
            f += 2 * b * oc * ic
        return {"bytes": n, "flops": f}
    if path == "blocks":
        # per block R, K, V, O, cm_r (d x d), cm_k (h x d), cm_v (d x h), five shift vectors, their previous inputs and the three
        # recurrence states read and written
        d, h, b = case["d"], case["h"], case["batch"]
        weights = 5 * d * d + 2 * d * h
        n = weights * 13 // 32 + 5 * _stream(B.RWKVQ_VQ, 1, d, case["entries"]) + 5 * 4 * b * d + 3 * 8 * b * d
        return {"bytes": case["layers"] * n + 2 * b * d + 8 * b * d, "flops": 2 * b * weights * case["layers"]}
    if path == "prefill":
        m, n, f, groups = case["tokens"], 0, 0, set()
        for (name, oc, ic, mu, kind) in _layer_shapes(case):
            n += _stream(_method(kind, oc, ic), oc, ic, case["entries"]) + m * oc * TORCH[case["y"]].itemsize
            n += _stream(B.RWKVQ_VQ, 1, ic, case["entries"]) if mu else 0
            group = name[:2] if name not in ("tm_o", "cm_v") else name
            if group not in groups:
                groups.add(group)
                n += 2 * m * ic
            f += 2 * m * oc * ic
        return {"bytes": n, "flops": f}
    if path == "convert":
        n = f = 0
        for (_, oc, ic, _, kind) in _layer_shapes(case):
            method = _method(kind, oc, ic)
            n += 2 * oc * ic + _stream(method, oc, ic, case["entries"])
            # at least one distance (two differences, two products and a sum) per vector and pass of the k-means
            f += 5 * (oc * ic // 2) * (case["iters"] + 1) if method == B.RWKVQ_VQ else 0
        return {"bytes": n, "flops": f}
    if path == "segments":
        tiles = -(-case["oc"] // case["rows"]) * -(-case["ic"] // case["cols"])
        return {"bytes": case["oc"] * case["ic"] * TORCH[case["dtype"]].itemsize + 20 * tiles, "flops": 0}
    d = case["d"]
    return {"bytes": 5 * (4 * d * case["samples"] + 4 * d + 2 * d + _stream(B.RWKVQ_VQ, 1, d, case["entries"])),
            "flops": 5 * 7 * (d // 2) * (case["iters"] + 1)}


def tolerance(case):
    path = case["path"]
    if path in ("product", "step", "host"):
        # inputs are mixed in fp32 and rounded to fp16 (2^-11) in front of exact weights and fp32 sums
        return {"rel": 2e-3 if case.get("y") == "f16" else 5e-4}
    if path == "blocks":
        # each stage rounds its input to fp16, and the squared ReLU and the gates of every block amplify what came before
        return {"rel": 1e-2, "max": 0.5}
    if path == "prefill":
        return {"rel": 5e-3}            # bf16 operands, fp32 sums
    if path == "mu":
        return {"rel": 1e-6}            # the squares of fp64 means, stored in fp32; images are bytes
    return {"rel": 1e-8}                # fp64 sums; formats chosen, codes and images are whole values
