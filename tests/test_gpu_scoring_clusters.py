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


@pytest.mark.parametrize("D,n_text,n_blocks,H", [(128, 512, 97, 8), (64, 512, 192, 16)])
def test_masks_of_a_ratio_for_every_head(D, n_text, n_blocks, H):
    """The masks, lists and counts of the staged selection at each head's own ratio."""
    B, N = 4 if H == 8 else 2, 64 * n_blocks
    q, k, v = (torch.randn((B, H, N, D), device=DEV).to(torch.bfloat16) for _ in range(3))
    per_head = [[(0.15, 0.3, 0.6, 0.9, 1.0)[(b + h) % 5] for h in range(H)] for b in range(B)]
    ctx, out = binding.Context(B, H, D, n_text, N - n_text), torch.empty_like(q)
    n0 = ctx.launch_count()
    ctx.rapid3_gated_step_heads(q, k, v, out, [2] * B, per_head)
    assert ctx.launch_count() - n0 == 2
    got = [t.clone() for t in ctx.workspace(B)]
    scores = ctx.rapid3_block_scores(q, k)
    assert torch.equal(bits(got[0]), bits(scores))
    for ratio in (0.15, 0.3, 0.6, 0.9, 1.0):
        ref = ctx.rapid3_select_mask(scores, [ratio] * B)
        at = torch.tensor(per_head, device=DEV) == torch.tensor(ratio, device=DEV)
        for a, b in zip(got[1:], ref):
            assert torch.equal(a[at], b[at]), ratio
    assert ctx.last_status() == 0


STEP = (2, 24, 64, 128, 28 * 64 - 128)             # images, heads, D, text, image tokens: 336 quads, the last ones by length


def step_inputs(seed):
    B, H, D, n_text, n_image = STEP
    gen = torch.Generator(device=DEV).manual_seed(seed)
    return [torch.randn((B, H, n_text + n_image, D), generator=gen, device=DEV).to(torch.bfloat16) for _ in range(3)]


def step_context():
    return binding.Context(*STEP)


def step_calls(ctx, q, k, v, out, acts_dev, ratios_dev):
    ratios = [1.0, 0.25]
    return {"step": lambda: ctx.rapid3_gated_step(q, k, v, out, [2, 2], ratios),
            "heads": lambda: ctx.rapid3_gated_step_heads(q, k, v, out, [2, 2], [[r] * 24 for r in ratios]),
            "mass": lambda: ctx.rapid3_gated_step_mass(q, k, v, out, [2, 2], ratios, 0.5),
            "device": lambda: ctx.rapid3_gated_step_device(q, k, v, out, acts_dev, ratios_dev)}


@pytest.mark.parametrize("kind", ["step", "heads", "mass", "device"])
def test_replays_of_a_captured_step(kind):
    """A step whose attention runs beside the clusters and ends by length, captured and replayed on buffers refilled in place."""
    q, k, v = step_inputs(0)
    out, ctx, plain = torch.empty_like(q), step_context(), step_context()
    acts, ratios = torch.full((2,), 2, dtype=torch.int32, device=DEV), torch.tensor([1.0, 0.25], device=DEV)
    call = step_calls(ctx, q, k, v, out, acts, ratios)[kind]
    n0 = ctx.launch_count()
    call()
    assert ctx.launch_count() - n0 == (5 if kind == "device" else 2)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    for seed in (1, 2, 3):
        for t, new in zip((q, k, v), step_inputs(seed)):
            t.copy_(new)
        for _ in range(3):                         # replays behind one another
            out.fill_(float("nan"))
            graph.replay()
        want = torch.empty_like(q)
        step_calls(plain, q, k, v, want, acts, ratios)[kind]()
        torch.cuda.synchronize()
        assert ctx.last_status() == 0 and plain.last_status() == 0
        assert torch.equal(bits(out), bits(want)), seed
        for a, b in zip(ctx.workspace(1), plain.workspace(1)):
            assert torch.equal(a, b), seed


@pytest.mark.parametrize("kind", ["step", "heads", "mass", "device"])
def test_two_contexts_on_two_streams(kind):
    """Two contexts, whose clusters and attention kernels share the GPU: the results of each alone."""
    acts, ratios = torch.full((2,), 2, dtype=torch.int32, device=DEV), torch.tensor([1.0, 0.25], device=DEV)
    tensors = [step_inputs(seed) for seed in (4, 5)]
    want, outs = [torch.empty_like(t[0]) for t in tensors], [torch.empty_like(t[0]) for t in tensors]
    alone = step_context()
    for t, o in zip(tensors, want):
        step_calls(alone, *t, o, acts, ratios)[kind]()
    torch.cuda.synchronize()
    ctxs, streams = [step_context() for _ in range(2)], [torch.cuda.Stream() for _ in range(2)]
    calls = [step_calls(c, *t, o, acts, ratios)[kind] for c, t, o in zip(ctxs, tensors, outs)]
    for _ in range(20):
        for call, s in zip(calls, streams):
            with torch.cuda.stream(s):
                call()
    torch.cuda.synchronize()
    for c, o, w in zip(ctxs, outs, want):
        assert c.last_status() == 0
        assert torch.equal(bits(o), bits(w))


def test_host_buffers_whose_head_groups_take_clusters():
    """The last image of a step on host buffers goes in four groups of heads, 16 of 64 here: the step's result on device tensors."""
    B, H, D, n_text, n_image = 2, 64, 64, 512, 56 * 64 - 1
    q, k, v = (torch.randn((B, H, n_text + n_image, D), device=DEV).to(torch.bfloat16) for _ in range(3))
    ctx, out, ratios = binding.Context(B, H, D, n_text, n_image), torch.empty_like(q), [1.0, 0.4]
    ctx.rapid3_gated_step(q, k, v, out, [2, 2], ratios)
    host = [t.cpu().pin_memory() for t in (q, k, v, torch.empty_like(q))]
    n0 = ctx.launch_count()
    ctx.rapid3_gated_step_host(*host, [2, 2], ratios)
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
    assert ctx.launch_count() - n0 == 1 + 4 * 2                # the dense image; clusters and attention of each group
    assert torch.equal(bits(host[3]), bits(out.cpu()))
