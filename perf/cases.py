"""Performance cases: what a user of the library has it do, through its public entry points.

The library encodes camera streams: a frame in full, or incrementally against the frame
before it, for one robot camera up to a batch of 32 views.  Beside the encoder it has two
calls without a handle: the token selection on embeddings that the caller holds, and the
action combine of the flow-matching head.

Encoder cases are either a whole encoder (ViT-Tiny's 12 layers, SigLIP-So400m's 27) or a
stack of four So400m blocks between the patch embedding and the final layer norm, which
keeps the rounding of one layer from travelling through many.  A stream's pass is two
consecutive incremental calls, to the next frame and back, so that a pass leaves the
handle as it found it and every pass over the same frames gives the same outputs.

Sizes are those of the repository's workloads (``synth.WORKLOADS``): 224 px frames of 196
or 256 tokens, 448 px frames of 1024, 1, 3 or 32 views, ~10 % of the patches changed.
"""
import math

import numpy as np
import torch

import paper_2607_12287_gb300 as ivit
from paper_2607_12287_gb300 import synth

TINY = dict(img_h=224, img_w=224, patch=16, dim=192, heads=3, mlp=768, gelu="erf")
SO400M_224 = dict(img_h=224, img_w=224, patch=14, dim=1152, heads=16, mlp=4304, gelu="tanh")
SO400M_448 = dict(SO400M_224, img_h=448, img_w=448)
STREAM = dict(kind="stream", select="threshold", ref="previous", score="embedding", schedule="incremental",
              mlp_tokens="updated")
FULL = dict(kind="full")


def listed():
    return [
        # one robot's action chunk (50 steps of 32 values) after the two solver steps: the smallest call
        dict(name="action_chunk", kind="action", batch=1, width=1600, bias=True),
        # a simulator's batch of chunks of 50 steps x 7 joints (rows that are no multiple of 16 bytes)
        dict(name="action_batch", kind="action", batch=4096, width=350, bias=True),
        # token selection on 32 views' embeddings in a caller that cannot allocate, a tenth of each view
        dict(name="select_topk_32views", kind="select", views=32, tokens=1024, dim=1152, select="topk", change=0.1),
        # ViT-Tiny on one camera: the lightest encoder, where launches are the cost
        dict(name="tiny_224_stream", depth=12, streams=1, views=1, change=0.082, **TINY, **STREAM),
        # ViT-Tiny, first frames of six cameras
        dict(name="tiny_224_full_6views", depth=12, streams=1, views=6, **TINY, **FULL),
        # the So400m encoder of a vision-language-action policy on one camera, frame after frame: the whole call
        dict(name="so400m_224_stream", depth=27, streams=1, views=1, change=0.1, **SO400M_224, **STREAM),
        # its full forward that seeds the caches
        dict(name="so400m_224_full", depth=4, streams=1, views=1, **SO400M_224, **FULL),
        # a robot with three cameras, 8 / 25 / 17 % of whose patches change
        dict(name="so400m_224_3view_stream", depth=4, streams=1, views=3, change=0.167, **SO400M_224, **STREAM),
        # half of the tokens by rank, scored on first-layer keys against their last refresh (the paper's Eq. 3)
        dict(name="so400m_224_topk_half", depth=4, streams=1, views=1, change=0.5, **SO400M_224,
             **dict(STREAM, select="topk", ref="last_refresh", score="key0")),
        # the reading of the paper in which every token passes the MLP
        dict(name="so400m_224_mlp_all", depth=4, streams=1, views=1, change=0.1, **SO400M_224,
             **dict(STREAM, mlp_tokens="all")),
        # a serving batch: 16 camera streams of two 448 px views, incremental and in full
        dict(name="so400m_448_stream_32views", depth=4, streams=16, views=2, change=0.094, **SO400M_448, **STREAM),
        dict(name="so400m_448_full_32views", depth=4, streams=16, views=2, **SO400M_448, **FULL),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["action", "select", "full", "full", "stream", "stream", "stream", "stream"])
    if kind == "action":
        batch = _log(rng, 1, 4096)
        return dict(kind=kind, batch=batch, width=_log(rng, 7, 1600), bias=rng.random() < 0.7)
    if kind == "select":
        return dict(kind=kind, views=_log(rng, 1, 32), tokens=_log(rng, 16, 1024), dim=64 * rng.randint(1, 18),
                    select=rng.choice(["threshold", "topk"]), change=round(rng.uniform(0.01, 0.6), 3))
    while True:
        patch = rng.choice([8, 14, 14, 16])
        gh, gw = rng.randint(7, 32), rng.randint(7, 32)
        # widths of the common encoders (Tiny to So400m and a little beyond), odd MLP widths among them
        head = rng.choice([32, 64, 64, 72, 80, 96, 128])
        heads = rng.choice([h for h in range(1, 21) if h * head % 64 == 0 and 128 <= h * head <= 1280])
        dim = head * heads
        mlp = 8 * int(dim * rng.uniform(2.0, 4.2) / 8)
        case = dict(kind=kind, img_h=gh * patch, img_w=gw * patch, patch=patch, dim=dim, heads=heads, mlp=mlp,
                    gelu=rng.choice(["tanh", "erf"]), depth=rng.randint(1, 6), streams=_log(rng, 1, 16),
                    views=rng.choice([1, 1, 2, 3]))
        if kind == "stream":
            case.update(change=round(math.exp(rng.uniform(math.log(0.01), 0.0)), 3),
                        select=rng.choice(["threshold", "threshold", "topk"]),
                        ref=rng.choice(["previous", "previous", "last_refresh"]),
                        score=rng.choice(["embedding", "embedding", "embedding", "key0"]),
                        schedule=rng.choice(["incremental", "incremental", "incremental", "odd_even"]),
                        mlp_tokens=rng.choice(["updated", "updated", "updated", "updated", "all"]))
        most = work(listed()[-1])
        if work(case)["flops"] <= most["flops"] and work(case)["bytes"] <= most["bytes"]:
            return case


# ------------------------------------------------------------------------- inputs

def _sizes(case):
    n = (case["img_h"] // case["patch"]) * (case["img_w"] // case["patch"])
    return case["streams"] * case["views"], n, case["dim"], case["mlp"]


def _changed(case, sv, n):
    """Changed patches per view: top-k refreshes the same number in every view; under a threshold the
    views differ (half, one and a half times, once the stated share)."""
    k = case["change"] * n
    return [min(n, int(round(k if case["select"] == "topk" else k * (0.5, 1.5, 1.0)[v % 3 if sv > 1 else 2])))
            for v in range(sv)]


def _weights(case, seed):
    """The encoder's tensors in the order of the library's weight buffer (bf16, on the GPU): random, with the
    scales of ``synth.make_weights`` (attention logits of standard deviation 2)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    _, n, d, f = _sizes(case)
    kp = case["patch"] ** 2 * 3

    def normal(*shape, std=0.02, mean=0.0):
        x = torch.randn(*shape, generator=g, device="cuda").clamp_(-2, 2)
        return x.mul_(std).add_(mean).to(torch.bfloat16)

    w = [("pe", normal(d, kp, std=1 / (64 * math.sqrt(kp)))), ("bpe", normal(d)), ("pos", normal(n, d, std=0.1))]
    for l in range(case["depth"]):
        qkv = normal(3 * d, d)
        qkv[:2 * d] = normal(2 * d, d, std=math.sqrt(2 / d))
        w += [(f"{l}.g1", normal(d, std=0.1, mean=1.0)), (f"{l}.c1", normal(d)), (f"{l}.qkv", qkv),
              (f"{l}.bqkv", normal(3 * d)), (f"{l}.o", normal(d, d)), (f"{l}.bo", normal(d)),
              (f"{l}.g2", normal(d, std=0.1, mean=1.0)), (f"{l}.c2", normal(d)), (f"{l}.up", normal(f, d)),
              (f"{l}.bup", normal(f)), (f"{l}.down", normal(d, f)), (f"{l}.bdown", normal(d))]
    return w + [("gf", normal(d, std=0.1, mean=1.0)), ("cf", normal(d))]


def _frames(case, seed):
    """Two frames of every view, uint8 [SV, H, W, 3], and the patches [SV, N] that differ between them: a
    textured still scene with +-1 sensor noise, in whose second frame some patches show other content."""
    g = torch.Generator(device="cuda").manual_seed(seed + 1000003)
    sv, n, _, _ = _sizes(case)
    h, w, p = case["img_h"], case["img_w"], case["patch"]

    def rand(*shape):
        return torch.rand(*shape, generator=g, device="cuda")

    scene = torch.nn.functional.interpolate(rand(sv, 3, h // 16 + 2, w // 16 + 2) * 120 - 60, size=(h, w),
                                            mode="bilinear", align_corners=False)
    a = (scene + rand(sv, 3, h, w) * 80 + 88).round_().clamp_(0, 255).permute(0, 2, 3, 1).contiguous()
    b = (a + (rand(sv, h, w, 3) * 3).floor_() - 1).clamp_(0, 255)
    mask = torch.zeros(sv, n, dtype=torch.bool, device="cuda")
    if case["kind"] == "stream":
        order = rand(sv, n).argsort(1).argsort(1)
        mask = order < torch.tensor(_changed(case, sv, n), device="cuda")[:, None]
    pixels = mask.view(sv, h // p, w // p).repeat_interleave(p, 1).repeat_interleave(p, 2)[..., None]
    b = torch.where(pixels, (rand(sv, h, w, 3) * 256).floor_(), b)
    return a.to(torch.uint8), b.to(torch.uint8), mask


def _action(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    shape = (case["batch"], case["width"])
    x0, v0, v7, b = (torch.randn(*shape, generator=g, device="cuda") for _ in range(4))
    alpha, beta = (torch.rand(case["batch"], generator=g, device="cuda") for _ in range(2))
    return x0, v0, v7, alpha, beta, b.mul_(0.1) if case["bias"] else None


def _select(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    v, n, d = case["views"], case["tokens"], case["dim"]
    ref = torch.randn(v, n, d, generator=g, device="cuda")
    new = torch.randn(v, n, d, generator=g, device="cuda")
    k = int(round(case["change"] * n))
    changed = torch.rand(v, n, generator=g, device="cuda").argsort(1).argsort(1) < k
    mix = torch.where(changed, 0.5 + 0.5 * torch.rand(v, n, generator=g, device="cuda"), 0.02)[..., None]
    return ref + mix * (new - ref), ref, k


def prepare(case, seed):
    if case["kind"] == "action":
        x = _action(case, seed)
        return dict(kind="action", inputs=x, out=torch.empty_like(x[0]))
    if case["kind"] == "select":
        cur, ref, k = _select(case, seed)
        v, n = case["views"], case["tokens"]
        idx = torch.empty(v, n, dtype=torch.int32, device="cuda")
        counts = torch.empty(v, dtype=torch.int32, device="cuda")
        mode = synth.SEL_TOPK if case["select"] == "topk" else synth.SEL_THRESHOLD
        return dict(kind="select", args=(cur, ref, v, n, case["dim"], mode, 0.98, k, idx, counts))
    shape = synth.EncoderShape(case["img_h"], case["img_w"], case["patch"], case["dim"], case["depth"], case["heads"],
                               case["mlp"], synth.GELU_ERF if case["gelu"] == "erf" else synth.GELU_TANH)
    flat = torch.cat([t.reshape(-1) for _, t in _weights(case, seed)]).view(torch.int16).cpu().numpy().view(np.uint16)
    a, b, _ = _frames(case, seed)
    sv, n, _, _ = _sizes(case)
    options = {}
    if case["kind"] == "stream":
        options = dict(
            select_mode=synth.SEL_TOPK if case["select"] == "topk" else synth.SEL_THRESHOLD, threshold=0.98,
            topk=_changed(case, sv, n)[0] if case["select"] == "topk" else 0,
            ref_mode=synth.REF_LAST_REFRESH if case["ref"] == "last_refresh" else synth.REF_PREV_FRAME,
            score_source=synth.SCORE_KEY0 if case["score"] == "key0" else synth.SCORE_EMBED,
            schedule=synth.SCHED_ODD_EVEN if case["schedule"] == "odd_even" else synth.SCHED_INCREMENTAL,
            mlp_tokens=1 if case["mlp_tokens"] == "all" else 0)
    enc = ivit.IncrementalViT(shape, flat, case["streams"], case["views"], **options)
    state = dict(kind=case["kind"], enc=enc, frames=(b, a))
    enc.encode_full(a)
    if case["kind"] == "stream":
        run(state)  # a stream that is under way
    return state


def run(state):
    if state["kind"] == "action":
        ivit.ivit_action_combine(*state["inputs"], state["out"])
        return state["out"]
    if state["kind"] == "select":
        ivit.ivit_select_noalloc(*state["args"])
        return state["args"][-2:]
    if state["kind"] == "full":
        return state["enc"].encode_full(state["frames"][0])
    return [state["enc"].encode_incremental(frame) for frame in state["frames"]]


# ------------------------------------------------------------------- what it takes

def work(case):
    if case["kind"] == "action":
        n = case["batch"] * case["width"]
        return dict(bytes=4 * n * (4 + case["bias"]) + 8 * case["batch"], flops=(4 + case["bias"]) * n)
    if case["kind"] == "select":
        n = case["views"] * case["tokens"]
        return dict(bytes=8 * n * case["dim"] + 4 * n + 4 * case["views"], flops=6 * n * case["dim"])
    sv, n, d, f = _sizes(case)
    m, depth, kp = sv * n, case["depth"], case["patch"] ** 2 * 3
    weights = 2 * (d * kp + n * d + depth * (4 * d * d + 2 * d * f))

    def call(u, mlp_rows):  # u updated rows of m; K/V: written for u, read for every token; references, tokens
        by = weights + m * kp + 8 * m * d + 4 * depth * d * (u + (m if u < m else 0)) + 2 * m * d
        fl = 2 * m * d * kp + depth * (8 * d * d * u + 4 * n * d * u + 4 * d * f * mlp_rows)
        return by, fl

    if case["kind"] == "full":
        calls = [call(m, m)]
    else:
        u = sum(_changed(case, sv, n))
        calls = [call(u, m if case["mlp_tokens"] == "all" else u)] * 2
        if case["schedule"] == "odd_even":
            calls[0] = call(m, m)
    return dict(bytes=sum(c[0] for c in calls), flops=sum(c[1] for c in calls))


def tolerance(case):
    if case["kind"] == "action":
        return dict(rel=3e-7, max=2e-6)  # three fp32 roundings (measured 5e-8)
    if case["kind"] == "select":
        return "exact"
    # bf16 activations: four times the measured distance from 64 bits (0.0046 after 27 layers, 0.0036 after 4)
    return dict(rel=0.018 if case["depth"] > 12 else 0.014, max=0.15)


# ------------------------------------------------------------------ in 64 bits

def exact(case, seed):
    if case["kind"] == "select":
        return None
    if case["kind"] == "action":
        x0, v0, v7, alpha, beta, b = (None if t is None else t.double() for t in _action(case, seed))
        y = x0 + alpha[:, None] * v0 + beta[:, None] * v7
        return y if b is None else y + b
    if work(case)["flops"] > 1e13:
        return None
    w = dict(_weights(case, seed))
    a, b, mask = _frames(case, seed)
    sv, n, d, _ = _sizes(case)
    h, p, heads, dh = case["img_h"], case["patch"], case["heads"], d // case["heads"]
    every = torch.ones_like(mask)
    f64 = {k: t.double() for k, t in w.items() if "." not in k}

    def embed(frame):
        x = frame.double().sub_(128).view(sv, h // p, p, -1, p, 3).permute(0, 1, 3, 2, 4, 5).reshape(sv * n, -1)
        return x @ f64["pe"].T + f64["bpe"]

    def norm(x, g, c):
        return torch.nn.functional.layer_norm(x, (d,), g, c, 1e-6)

    def gelu(x):
        return torch.nn.functional.gelu(x, approximate="none" if case["gelu"] == "erf" else "tanh")

    mlp_all = case["kind"] == "stream" and case["mlp_tokens"] == "all"
    kv = [[torch.zeros(sv * n, d, dtype=torch.float64, device="cuda") for _ in range(3)]
          for _ in range(case["depth"])]  # keys, values, attention outputs of every token
    tokens = torch.zeros(sv * n, d, dtype=torch.float64, device="cuda")

    def encode(frame, updated):
        rows = updated.reshape(-1).nonzero()[:, 0]
        x = embed(frame) + f64["pos"].repeat(sv, 1)
        x = x if mlp_all else x[rows]
        for l in range(case["depth"]):
            t = {k.split(".")[1]: v.double() for k, v in w.items() if k.startswith(f"{l}.")}
            keys, values, attended = kv[l]
            q, k, v = (norm(x[rows] if mlp_all else x, t["g1"], t["c1"]) @ t["qkv"].T + t["bqkv"]).split(d, 1)
            keys[rows], values[rows] = k, v
            o, at = torch.empty_like(q), 0
            for i in range(sv):
                u = int(updated[i].sum())
                if u:
                    qi, ki, vi = (y.view(-1, heads, dh).transpose(0, 1) for y in (
                        q[at:at + u], keys[i * n:(i + 1) * n], values[i * n:(i + 1) * n]))
                    s = (qi @ ki.transpose(1, 2) / math.sqrt(dh)).softmax(-1)
                    o[at:at + u] = (s @ vi).transpose(0, 1).reshape(u, d)
                at += u
            o = o @ t["o"].T + t["bo"]
            if mlp_all:
                attended[rows] = o
                x = x + attended
            else:
                x = x + o
            x = x + gelu(norm(x, t["g2"], t["c2"]) @ t["up"].T + t["bup"]) @ t["down"].T + t["bdown"]
        y = norm(x, f64["gf"], f64["cf"])
        if mlp_all:
            tokens[:] = y
        else:
            tokens[rows] = y
        return tokens.clone().view(sv, n, d)

    if case["kind"] == "full":
        return encode(b, every)
    if case["schedule"] == "odd_even":
        return [(encode(b, every), None), (encode(a, mask), None)]
    encode(a, every)
    return [(encode(b, mask), None), (encode(a, mask), None)]
