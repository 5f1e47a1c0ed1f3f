"""Steps of many quads take their means, scores and selection from one kernel of thread-block clusters, of which the
attention does not wait for what needs no mask.  The same scores, masks, lists and outputs come from the stages called one by
one and from the images alone, whose few quads take the three kernels, bit for bit: at row counts around the tiles of the score
products, at the row lengths at which the register count changes, with infinities and NaN among the numbers, for every rule."""
import pytest
import torch

from paper_2509_22323_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda"


def bits(t):
    return t.contiguous().view({2: torch.int16, 4: torch.int32, 8: torch.int64}[t.element_size()])


@pytest.mark.parametrize("D,n_text,n_image,H,ratios", [
    (64, 333, 1024, 24, (0.3, 0.6)),                            # 22 blocks, clusters of two; text and image rows in one quad
    (128, 512, 61, 16, (1.0, 0.3, 1.0, 0.6, 1.0, 0.15)),        # 9 blocks, the last of 61 tokens: a quad of one row
    (64, 512, 2555, 8, (0.3, 0.6, 0.15, 0.3, 0.6, 0.15)),       # 48 blocks: a whole buffer of columns
    (128, 512, 64 * 89, 8, (0.3, 0.6, 0.15, 0.9)),              # 97 blocks: one more than three registers a lane hold
    (64, 512, 64 * 184, 16, (0.3, 0.6)),                        # 192 blocks: the longest rows of this kernel
])
def test_clusters_equal_the_stages(D, n_text, n_image, H, ratios):
    B, N = len(ratios), n_text + n_image
    sparse = [b for b in range(B) if ratios[b] < 1.0]
    gen = torch.Generator(device=DEV).manual_seed(N)
    q, k, v = (torch.randn((B, H, N, D), generator=gen, device=DEV).to(torch.bfloat16) for _ in range(3))
    k[1, 0, :64] *= 1e-38                                          # subnormal numbers among them
    ctx = binding.Context(B, H, D, n_text, n_image)
    per_head = [[min(1.0, r * (0.5, 1.0, 1.5)[h % 3]) if r < 1.0 else 1.0 for h in range(H)] for r in ratios]
    acts_dev, ratios_dev = torch.full((B,), 2, dtype=torch.int32, device=DEV), torch.tensor(ratios, device=DEV)
    mass_scale = 4 * D ** -0.5
    calls = {
        "step": lambda out, acts: ctx.rapid3_gated_step(q, k, v, out, acts, ratios),
        "heads": lambda out, acts: ctx.rapid3_gated_step_heads(q, k, v, out, acts, per_head),
        "mass": lambda out, acts: ctx.rapid3_gated_step_mass(q, k, v, out, acts, ratios, mass_scale),
        "device": lambda out, acts: ctx.rapid3_gated_step_device(q, k, v, out, acts_dev, ratios_dev),
    }
    scores = ctx.rapid3_block_scores(q, k, img_idx=sparse)
    some = [ratios[b] for b in sparse]
    want = {"step": ctx.rapid3_select_mask(scores, some), "mass": ctx.rapid3_select_mask_mass(scores, some, mass_scale)[1:]}
    want["device"] = want["step"]
    for name, call in calls.items():
        out, alone = torch.zeros_like(q), torch.zeros_like(q)
        n0 = ctx.launch_count()
        call(out, [2] * B)
        torch.cuda.synchronize()
        assert ctx.last_status() == 0
        # clusters and attention; decisions on the GPU, which the host cannot weigh: plan, pool, scores, selection, attention
        assert ctx.launch_count() - n0 == (5 if name == "device" else 2)
        ws = [t.clone() for t in ctx.workspace(len(sparse))]
        assert torch.equal(bits(ws[0]), bits(scores))
        for got, ref in zip(ws[1:], want.get(name, ())):
            assert torch.equal(got, ref), name
        for b in range(B):
            if name == "device":
                acts_dev.copy_(torch.tensor([2 if i == b else 0 for i in range(B)], dtype=torch.int32, device=DEV))
            call(alone, [2 if i == b else 0 for i in range(B)])
        torch.cuda.synchronize()
        assert torch.equal(bits(out), bits(alone)), name


@pytest.mark.parametrize("n_blocks,H,ratios,launches", [
    (44, 24, (0.5,), 2),               # 264 quads: the second round of 148 SMs is 0.78 full
    (57, 24, (0.5,), 4),               # 360: the third is 0.43 full
    (57, 16, (0.25,), 4),              # 240: 0.62
    (72, 16, (0.25,), 2),              # 288: 0.95
    (57, 12, (0.5, 1.0), 4),           # 360, a dense image beside, but less than 16 pairs
    (57, 24, (0.5, 1.0), 2),           # 720, a dense image beside
    (57, 24, (0.5, 0.5), 2),           # 720, two images: 48 pairs
])
def test_which_steps_take_clusters(n_blocks, H, ratios, launches):
    """One sparse image with nothing dense beside it takes the three kernels where its last round of SMs has room."""
    B, N, D = len(ratios), 64 * n_blocks, 128
    q, k, v = (torch.randn((B, H, N, D), device=DEV).to(torch.bfloat16) for _ in range(3))
    ctx, out = binding.Context(B, H, D, 512, N - 512), torch.empty_like(q)
    n0 = ctx.launch_count()
    ctx.rapid3_gated_step(q, k, v, out, [2] * B, ratios)
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
    assert ctx.launch_count() - n0 == launches


def test_means_of_numbers_that_are_not_finite():
    """A block with an infinity or a NaN has them in its scores as sums in 64 bits give them, whichever half of a word holds it."""
    B, H, D, N = 2, 24, 64, 64 * 22
    q, k = (torch.randn((B, H, N, D), device=DEV).to(torch.bfloat16) for _ in range(2))
    q[0, 0, 70, 3] = float("inf")
    q[0, 0, 140, 4] = float("-inf")
    k[0, 1, 200, 9] = float("nan")
    k[1, 2, 300, 0] = float("inf")
    k[1, 2, 301, 0] = float("-inf")
    q[1, 3, 64 * 5:64 * 6] = torch.finfo(torch.bfloat16).max
    ctx = binding.Context(B, H, D, 0, N)
    got = ctx.rapid3_block_scores(q, k)
    ctx.rapid3_gated_step(q, k, q, torch.zeros_like(q), [2, 2], [0.5, 0.25])
    torch.cuda.synchronize()
    ws = ctx.workspace(B)[0]
    mq, mk = (t.double().unflatten(2, (-1, 64)).mean(3) for t in (q, k))
    ref = (mq[:, :, :, None, :] * mk[:, :, None, :, :]).sum(-1).float()
    for s in (got, ws):
        assert torch.equal(s.isnan(), ref.isnan())
        ok = ~ref.isnan()
        assert torch.equal(s[ok].isinf(), ref[ok].isinf())
        fin = ref.isfinite()
        assert float(((s - ref)[fin].abs() / (1e-6 * ref[fin].abs() + 1e-6 * ref[fin].abs().mean().clamp(max=1.0))).max()) <= 1.0


@pytest.mark.parametrize("D,H,n_text,n_image,ratios,packed", [
    (64, 24, 333, 1024, (0.3, 0.6), False),                        # whole text quads write while other rows' means are taken
    (128, 24, 512, 1600, (1.0, 0.5, 0.25), False),                 # a dense image beside two sparse ones
    (128, 24, 512, 1600, (1.0, 0.5, 0.25), True),                  # Q, K, V and the result in turn in one buffer
])
def test_steps_in_place(D, H, n_text, n_image, ratios, packed):
    """The result may take Q's place, or lie between the tensors: the same scores, masks and results as in a buffer of its own."""
    B, N = len(ratios), n_text + n_image
    gen = torch.Generator(device=DEV).manual_seed(N)
    if packed:
        buf = torch.randn((B, N, 4, H, D), generator=gen, device=DEV).to(torch.bfloat16)
        q, k, v, place = (buf[:, :, i].permute(0, 2, 1, 3) for i in range(4))
        strides = q.stride()[:3]
    else:
        q, k, v = (torch.randn((B, H, N, D), generator=gen, device=DEV).to(torch.bfloat16) for _ in range(3))
        place, strides = q, None
    q0 = q.clone()
    n_sparse = sum(r < 1.0 for r in ratios)
    acts_dev, ratios_dev = torch.full((B,), 2, dtype=torch.int32, device=DEV), torch.tensor(ratios, device=DEV)
    ctx = binding.Context(B, H, D, n_text, n_image, strides=strides) if strides else binding.Context(B, H, D, n_text, n_image)
    calls = {
        "step": lambda out: ctx.rapid3_gated_step(q, k, v, out, [2] * B, ratios),
        "heads": lambda out: ctx.rapid3_gated_step_heads(q, k, v, out, [2] * B, [[r] * H for r in ratios]),
        "mass": lambda out: ctx.rapid3_gated_step_mass(q, k, v, out, [2] * B, ratios, 4 * D ** -0.5),
        "device": lambda out: ctx.rapid3_gated_step_device(q, k, v, out, acts_dev, ratios_dev),
    }
    for name, call in calls.items():
        apart = torch.empty_like(buf)[:, :, 3].permute(0, 2, 1, 3) if packed else torch.empty_like(q)
        call(apart)
        torch.cuda.synchronize()
        scores = ctx.workspace(n_sparse)[0].clone()
        call(place)
        torch.cuda.synchronize()
        assert ctx.last_status() == 0
        assert torch.equal(ctx.workspace(n_sparse)[0], scores), name
        assert torch.equal(bits(place), bits(apart)), name
        q.copy_(q0)
