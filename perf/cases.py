"""The calls whose speed is watched: what a denoising loop asks of this library, from the smallest call to the largest.

A case is one attention call (or one cache-reuse call) of a denoising step, made through the public entry points of
`paper_2509_22323_b200.binding`.  `listed()` holds one case per kind of use, `draw()` gives others of the same ranges.
The keys of a case:

  kind     "step"    rapid3_gated_step, actions and keep ratios on the host
           "heads"   rapid3_gated_step_heads, a keep ratio per image and head
           "mass"    rapid3_gated_step_mass, a mass share per image instead of a keep ratio
           "device"  rapid3_gated_step_device, actions and keep ratios on the GPU
           "fused"   rapid3_gated_step_fused, from the raw projections (RMS norm, gain, rotary embedding) onwards
           "staged"  rapid3_block_scores, rapid3_select_mask and rapid3_sparse_joint_attn, one after the other
           "cache"   rapid3_cache_step on a batch of block outputs
  B, H, D, text, grid   images, heads, head dimension, text tokens, and the side of the square grid of image tokens
  actions  one digit per image: 0 step skipped, 1 cache reused, 2 attention
  ratios   keep ratio (mass share) per image, separated by commas
  layout   "heads": Q, K, V, O are [B, H, N, D]; "tokens": views of [B, N, H, D] buffers, as a projection leaves them
"""
from __future__ import annotations

import math

import torch

from paper_2509_22323_b200 import binding, inputs


def _case(name, kind, B, H, D, text, grid, actions, ratios, layout="heads"):
    case = {"name": name} if name else {}
    case.update(kind=kind, B=B, H=H, D=D, text=text, grid=grid, actions=actions, ratios=ratios, layout=layout)
    return case


def listed():
    return [
        # the smallest call: one image, two heads, five blocks; all latency and launches
        _case("tiny_step", "step", 1, 2, 64, 64, 16, "2", "0.5"),
        # 512^2 images on 24 heads of 64 channels, a guidance pair of sparse images; Q, K, V, O lie token by token, as the
        # projections in front of the attention write them; 1357 tokens, not a multiple of the block
        _case("sd3_512_tokens", "step", 2, 24, 64, 333, 32, "22", "0.5,0.25", "tokens"),
        # 1024^2 images, 24 heads of 64 channels, one dense and one sparse image, ragged tail (4429 tokens)
        _case("sd3_1024_step", "step", 2, 24, 64, 333, 64, "22", "1.0,0.5"),
        # 1024^2 images, 24 heads of 128 channels, one image at each keep ratio: the benchmark's default workload
        _case("flux_1024_step", "step", 3, 24, 128, 512, 64, "222", "1.0,0.5,0.25"),
        # one 2048^2 image: the longest sequence of the configurations, most blocks dropped
        _case("flux_2048_step", "step", 1, 24, 128, 512, 128, "2", "0.25"),
        # one step of a batch of eight trajectories (step 14 of the configured one): skip, reuse and every keep ratio
        _case("trajectory_step", "step", 8, 24, 128, 512, 64, "20222212", "1.0,1.0,0.25,1.0,0.5,0.5,1.0,0.5"),
        # a policy whose decisions stay on the GPU: four 1024^2 images, one of them reusing its cache
        _case("flux_1024_device", "device", 4, 24, 128, 512, 64, "2122", "1.0,1.0,0.5,0.25"),
        # one image from the raw projections onwards: norm, gain and rotary embedding in front of the same step
        _case("flux_1024_fused", "fused", 1, 24, 128, 512, 64, "2", "0.5"),
        # a policy that sets a ratio for every head
        _case("sd3_1024_heads", "heads", 2, 24, 64, 333, 64, "22", "0.5,0.25"),
        # the cumulative-mass rule in the place of top-k
        _case("flux_1024_mass", "mass", 2, 24, 128, 512, 64, "22", "0.5,0.9"),
        # the three stages called one by one, masks in the caller's hands; odd sizes: 45 x 45 grid, 77 text tokens
        _case("staged_ragged", "staged", 3, 12, 128, 77, 45, "222", "0.75,0.5,0.3"),
        # block outputs of eight images between steps: some refresh their cached residual, some reuse it, one is skipped
        _case("cache_step", "cache", 8, 24, 128, 512, 64, "21012121", "1.0,1.0,1.0,1.0,1.0,1.0,1.0,1.0"),
    ]


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["step", "step", "step", "heads", "mass", "device", "fused", "staged", "cache"])
        B = rng.choice([1, 1, 2, 2, 3, 4, 6, 8])
        H = rng.choice([2, 3, 6, 12, 16, 24, 24])
        D = rng.choice([64, 128])
        text = rng.choice([0, 64, 77, 128, 333, 512, rng.randint(1, 512)])
        grid = round(math.exp(rng.uniform(math.log(16), math.log(128))))
        actions = [rng.choice("22222201") for _ in range(B)]
        actions[rng.randrange(B)] = "2"
        if kind == "staged":                   # the caller of the stages has sorted the batch out already
            actions = ["2"] * B
        ratios = [rng.choice([1.0, 0.5, 0.25, round(rng.uniform(0.1, 0.95), 2)]) for _ in range(B)]
        case = _case(None, kind, B, H, D, text, grid, "".join(actions), ",".join(str(r) for r in ratios),
                     rng.choice(["heads", "heads", "tokens"]) if kind != "cache" else "heads")
        if _cost(case) <= most:
            return case


def _lists(case):
    return [int(a) for a in case["actions"]], [float(r) for r in case["ratios"].split(",")]


def _head_ratios(case):
    """Per-head ratios around the image's: half of it, itself, and half as much again."""
    _, ratios = _lists(case)
    return [[min(1.0, r * (0.5, 1.0, 1.5)[h % 3]) for h in range(case["H"])] for r in ratios]


# softmax temperature of the cumulative-mass rule, in units of the attention's own: pooled scores are small
MASS_TEMPERATURE = 4.0


def _mass_kept(tau):
    """Share of the free blocks that the cumulative-mass rule keeps on these inputs (seen: 0.27 at 0.5, 0.72 at 0.9)."""
    return tau * (0.2 + 0.65 * tau)


def _workload(case, seed):
    _, ratios = _lists(case)
    sigma = max(1.0, case["grid"] / 16)        # the blur of the configurations: 4 tokens at 64, 8 at 128
    return inputs.Workload("case", case["B"], case["H"], case["D"], case["text"], case["grid"], sigma, tuple(ratios),
                           rope=case["D"] == 128 and case["kind"] != "fused", seed=seed)


def _token_major(t):
    """The same [B, H, N, D] values, stored token by token ([B, N, H, D])."""
    return t.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)


def _rotary_table(wl, device):
    """(cos, sin) per token and channel pair: half of the channels by grid row, half by column; text unrotated."""
    pairs = wl.head_dim // 4
    freq = 10000.0 ** (-torch.arange(pairs, device=device, dtype=torch.float64) / pairs)
    at = torch.arange(wl.n_image, device=device)
    ang = torch.cat([(at // wl.grid)[:, None] * freq, (at % wl.grid)[:, None] * freq], dim=1)
    ang = torch.cat([torch.zeros(wl.n_text, 2 * pairs, device=device, dtype=torch.float64), ang])
    return torch.stack([ang.cos(), ang.sin()], dim=-1).float().contiguous()


def _inputs(case, seed, dev="cuda"):
    """The tensors of a case by name, from the seed alone."""
    gen = torch.Generator(device=dev).manual_seed(seed)
    wl = _workload(case, seed)
    if case["kind"] == "cache":
        shape = (case["B"], wl.n_tokens, case["H"] * case["D"])
        return {key: torch.randn(shape, generator=gen, device=dev).mul_(scale).to(torch.bfloat16)
                for key, scale in (("x", 3.0), ("o", 3.0), ("delta", 1.0))}
    q, k, v = inputs.make_qkv(wl, 0, device=dev)
    if case["kind"] != "fused":
        return {"q": q, "k": k, "v": v}
    # raw projections: every token has a magnitude of its own, which the norm takes out again
    mag = torch.exp(0.5 * torch.randn((case["B"], case["H"], wl.n_tokens, 1), generator=gen, device=dev))
    t = {"q_raw": (q * mag).to(torch.bfloat16), "k_raw": (k * mag.flip(2)).to(torch.bfloat16), "v": v}
    t["q_gain"], t["k_gain"] = (0.5 + torch.rand(case["D"], generator=gen, device=dev) for _ in range(2))
    t["rot"] = _rotary_table(wl, dev)
    return t


def prepare(case, seed):
    actions, ratios = _lists(case)
    state = {"case": case, "actions": actions, "ratios": ratios, **_inputs(case, seed)}
    if case["kind"] == "cache":
        return state
    state["out"] = torch.zeros_like(state["v"])
    if case["kind"] == "fused":
        state["q"], state["k"] = torch.zeros_like(state["q_raw"]), torch.zeros_like(state["k_raw"])
    strides = None
    if case["layout"] == "tokens":
        for key in ("q", "k", "v", "out", "q_raw", "k_raw"):
            if key in state:
                state[key] = _token_major(state[key])
        strides = state["q"].stride()[:3]
    state["ctx"] = binding.Context(case["B"], case["H"], case["D"], case["text"], case["grid"] ** 2, strides=strides)
    if case["kind"] == "heads":
        state["ratios"] = _head_ratios(case)
    elif case["kind"] == "device":
        state["actions"] = torch.tensor(actions, dtype=torch.int32, device="cuda")
        state["ratios"] = torch.tensor(ratios, dtype=torch.float32, device="cuda")
    elif case["kind"] == "mass":
        state["mass_scale"] = MASS_TEMPERATURE * case["D"] ** -0.5
    return state


def run(state):
    kind, actions, ratios = state["case"]["kind"], state["actions"], state["ratios"]
    if kind == "cache":
        binding.rapid3_cache_step(state["x"], state["o"], state["delta"], actions)
        return state["o"], state["delta"]
    ctx, q, k, v, out = state["ctx"], state["q"], state["k"], state["v"], state["out"]
    if kind == "step":
        return ctx.rapid3_gated_step(q, k, v, out, actions, ratios)
    if kind == "heads":
        return ctx.rapid3_gated_step_heads(q, k, v, out, actions, ratios)
    if kind == "mass":
        return ctx.rapid3_gated_step_mass(q, k, v, out, actions, ratios, state["mass_scale"])
    if kind == "device":
        return ctx.rapid3_gated_step_device(q, k, v, out, actions, ratios)
    if kind == "fused":
        ctx.rapid3_gated_step_fused(state["q_raw"], state["k_raw"], v, state["q_gain"], state["k_gain"], state["rot"], 1e-6,
                                    q, k, out, actions, ratios)
        return q, k, out
    scores = ctx.rapid3_block_scores(q, k)
    bitmask, kept_idx, kept_cnt = ctx.rapid3_select_mask(scores, ratios)
    ctx.rapid3_sparse_joint_attn(q, k, v, out, kept_idx=kept_idx, kept_cnt=kept_cnt)
    return scores, bitmask, kept_idx, kept_cnt, out


def work(case):
    """Q, K, V read once and O written once for every image that attends, and the multiply-adds of Q K^T and P V on the
    kept blocks alone (4 x rows x columns x D); scores, masks and lists stay inside the call."""
    actions, ratios = _lists(case)
    B, H, D, text = case["B"], case["H"], case["D"], case["text"]
    N = text + case["grid"] ** 2
    if case["kind"] == "cache":
        return {"bytes": sum(a != 0 for a in actions) * 3 * 2 * N * H * D, "flops": 0}
    nb, ntb = -(-N // 64), -(-text // 64)
    n_free = max(nb - ntb - 1, 0)
    per_head = _head_ratios(case) if case["kind"] == "heads" else [[r] * H for r in ratios]
    flops, images = 0.0, 0
    for b in range(B):
        if actions[b] != 2:
            continue
        images += 1
        for r in per_head[b]:
            if case["kind"] == "mass" and r < 1.0:
                r = _mass_kept(r)
            kept = min(n_free, math.ceil(r * n_free - 1e-6))
            columns = min(N, 64 * (kept + ntb + 1))
            text_rows = min(N, 64 * ntb)
            flops += 4.0 * D * (text_rows * N + (N - text_rows) * columns)
    tensors = 6 if case["kind"] == "fused" else 4
    bytes_ = images * tensors * 2 * H * N * D
    if case["kind"] == "staged":               # the scores, bit masks, lists and counts are the caller's
        bytes_ += B * H * nb * (4 * nb + 8 * (-(-nb // 64)) + 4 * nb + 4)
    return {"bytes": bytes_, "flops": flops}


def _cost(case):
    w = work(case)
    return w["bytes"] / 5e12 + w["flops"] / 1e15


def tolerance(case):
    if case["kind"] == "cache":
        return "exact"                         # one fp32 addition and one rounding to bf16 per element
    # P is rounded to bf16 in front of P V and the result once more: against the same attention in 64 bits on the same
    # masks 1.7e-3 in the 2-norm and 7.6e-3 at most were seen; the masks themselves are whole values and do not differ
    return {"rel": 7e-3, "max": 3e-2, "differ": 0.0}


def _f32(x):
    """A float as the C interface hands it on: rounded to single precision."""
    return torch.tensor(x, dtype=torch.float32).double().item()


def _block_scores(q, k):
    """[H, N, D] in 64 bits -> dot products of the 64-token block means, [H, nb, nb]."""
    def means(t):
        n_blocks = -(-t.shape[1] // 64)
        padded = torch.nn.functional.pad(t, (0, 0, 0, 64 * n_blocks - t.shape[1])).unflatten(1, (n_blocks, 64)).sum(2)
        count = torch.full((n_blocks, 1), 64.0, device=t.device, dtype=t.dtype)
        count[-1] = t.shape[1] - 64 * (n_blocks - 1)
        return padded / count
    return means(q) @ means(k).transpose(1, 2)


def _kept(case, scores, ratios):
    """Boolean [H, nb, nb]: text blocks and the diagonal, and of the others the best (equal scores: the lower index)."""
    H, nb, _ = scores.shape
    ntb = -(-case["text"] // 64)
    n_free = max(nb - ntb - 1, 0)
    at = torch.arange(nb, device=scores.device)
    forced = (at[:, None] < ntb) | (at[None, :] < ntb) | (at[:, None] == at[None, :])
    s = scores.float().double().masked_fill(forced, -math.inf)         # the decision is made on single-precision scores
    best, order = s.sort(dim=2, descending=True, stable=True)
    if case["kind"] == "mass" and ratios[0] < 1.0:
        temperature = _f32(MASS_TEMPERATURE * case["D"] ** -0.5)
        w = torch.exp(temperature * (best - best[:, :, :1])).nan_to_num(0.0)     # rows without candidates: nan
        before = w.cumsum(2) - w                                       # mass of the better candidates
        take = before < _f32(ratios[0]) * w.sum(2, keepdim=True)
    else:
        count = torch.tensor([min(n_free, max(0, math.ceil(_f32(r) * n_free - 1e-6))) for r in ratios], device=scores.device)
        take = at[None, None, :] < count[:, None, None]
    take = take & (best > -math.inf)
    return forced | torch.zeros_like(take).scatter(2, order, take)


def _attention(q, k, v, kept):
    """Softmax attention of [H, N, D] in 64 bits over the kept blocks; head by head, 2048 query rows at a time."""
    out = torch.empty_like(v)
    block = torch.arange(q.shape[1], device=q.device) // 64
    for h in range(q.shape[0]):
        for r in range(0, q.shape[1], 2048):
            logits = (q[h, r:r + 2048] @ k[h].T) * q.shape[2] ** -0.5
            logits.masked_fill_(~kept[h][block[r:r + 2048]][:, block], -math.inf)
            out[h, r:r + 2048] = logits.softmax(1) @ v[h]
    return out


def _produce(raw, gain, rot):
    """Norm, gain and rotary embedding of [H, N, D] in 64 bits."""
    x = raw * torch.rsqrt(raw.square().mean(2, keepdim=True) + _f32(1e-6)) * gain
    a, b = x[..., 0::2], x[..., 1::2]
    c, s = rot[..., 0], rot[..., 1]
    return torch.stack((a * c - b * s, a * s + b * c), dim=-1).flatten(2)


def exact(case, seed):
    """What run() returns, in 64 bits.  Masks and lists are whole values, compared as they are: None here."""
    actions, ratios = _lists(case)
    t = _inputs(case, seed)
    if case["kind"] == "cache":
        x, o, delta = (t[key].double() for key in ("x", "o", "delta"))
        for b, a in enumerate(actions):
            if a == 1:
                o[b] = x[b] + delta[b]
            elif a == 2:
                delta[b] = o[b] - x[b]
        return o, delta
    out = torch.zeros_like(t["v"], dtype=torch.float64)
    produced = [torch.zeros_like(out), torch.zeros_like(out)] if case["kind"] == "fused" else []
    all_scores = []
    for b, a in enumerate(actions):
        if a != 2:
            continue
        if produced:
            for p, key in zip(produced, ("q", "k")):
                p[b] = _produce(t[key + "_raw"][b].double(), t[key + "_gain"].double(), t["rot"].double())
            q, k = (p[b].to(torch.bfloat16).double() for p in produced)    # the attention reads them as they are stored
        else:
            q, k = t["q"][b].double(), t["k"][b].double()
        scores = _block_scores(q, k)
        all_scores.append(scores)
        share = _head_ratios(case)[b] if case["kind"] == "heads" else [ratios[b]] * case["H"]
        out[b] = _attention(q, k, t["v"][b].double(), _kept(case, scores, share))
    if case["kind"] == "fused":
        return produced[0], produced[1], out
    if case["kind"] == "staged":
        return torch.stack(all_scores), None, None, None, out
    return out
