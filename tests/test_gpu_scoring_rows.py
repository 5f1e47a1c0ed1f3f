"""Steps of 75 to 221 quads whose scores and selection are one kernel: the scores, masks, lists and counts of the staged calls, bit for
bit, for every rule, for decisions on the GPU and behind the producer, at row lengths around a warp's eight key blocks and the kernel's
three sizes; outputs of the images alone."""
import pytest
import torch

from paper_2509_22323_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda"


def bits(t):
    return t.contiguous().view({2: torch.int16, 4: torch.int32, 8: torch.int64}[t.element_size()])


@pytest.mark.parametrize("D,n_text,n_image,H,B", [
    (64, 0, 64 * 2 - 5, 25, 3),             # 75 quads of two blocks
    (128, 77, 64 * 12, 16, 3),              # 14 blocks: 192 quads, the last ones by length, a quad of two rows
    (64, 512, 64 * 56, 3, 3),               # 64 blocks: a fragment for each of eight warps
    (128, 130, 64 * 62 + 1, 3, 2),          # 65 blocks, one token in the last
    (64, 333, 64 * 91, 2, 2),               # 97 blocks
    (128, 64, 64 * 127, 2, 2),              # 128: the longest rows
])
def test_rows_equal_the_stages(D, n_text, n_image, H, B):
    N, nb = n_text + n_image, (n_text + n_image + 63) // 64
    gen = torch.Generator(device=DEV).manual_seed(N)
    q, k, v = (torch.randn((B, H, N, D), generator=gen, device=DEV).to(torch.bfloat16) for _ in range(3))
    ratios = [(0.4, 0.7, 0.15)[b % 3] for b in range(B)]
    per_head = [[(0.15, 0.4, 0.9)[(b + h) % 3] for h in range(H)] for b in range(B)]
    ctx = binding.Context(B, H, D, n_text, n_image)
    acts_dev, ratios_dev = torch.full((B,), 2, dtype=torch.int32, device=DEV), torch.tensor(ratios, device=DEV)
    calls = {
        "step": lambda out, acts: ctx.rapid3_gated_step(q, k, v, out, acts, ratios),
        "heads": lambda out, acts: ctx.rapid3_gated_step_heads(q, k, v, out, acts, per_head),
        "mass": lambda out, acts: ctx.rapid3_gated_step_mass(q, k, v, out, acts, ratios, 4 * D ** -0.5),
        "device": lambda out, acts: ctx.rapid3_gated_step_device(q, k, v, out, acts_dev, ratios_dev),
    }
    scores = ctx.rapid3_block_scores(q, k)
    want = {"step": ctx.rapid3_select_mask(scores, ratios), "mass": ctx.rapid3_select_mask_mass(scores, ratios, 4 * D ** -0.5)[1:]}
    want["device"] = want["step"]
    parts = ctx.launch_count()
    ctx.rapid3_sparse_joint_attn(q, k, v, torch.empty_like(q))
    attention = ctx.launch_count() - parts                         # two where lists are worked on in parts
    for name, call in calls.items():
        out, alone = torch.full_like(q, float("nan")), torch.full_like(q, float("nan"))
        n0 = ctx.launch_count()
        call(out, [2] * B)
        assert ctx.launch_count() - n0 <= 2 + attention + (name == "device")
        torch.cuda.synchronize()
        assert ctx.last_status() == 0
        ws = [t.clone() for t in ctx.workspace(B)]
        assert torch.equal(bits(ws[0]), bits(scores)), name
        for got, ref in zip(ws[1:], want.get(name, ())):
            assert torch.equal(got, ref), name
        if name == "heads":
            for ratio in (0.15, 0.4, 0.9):
                at = torch.tensor(per_head, device=DEV) == torch.tensor(ratio, device=DEV)
                for got, ref in zip(ws[1:], ctx.rapid3_select_mask(scores, [ratio] * B)):
                    assert torch.equal(got[at], ref[at]), ratio
        for b in range(B):
            if name == "device":
                acts_dev.copy_(torch.tensor([2 if i == b else 0 for i in range(B)], dtype=torch.int32, device=DEV))
            call(alone, [2 if i == b else 0 for i in range(B)])
        torch.cuda.synchronize()
        assert torch.equal(bits(out), bits(alone)), name
        assert torch.isfinite(out).all()


def test_rows_behind_the_producer():
    """The scores of the Q and K that the producer has written."""
    B, H, D, n_text, n_image = 2, 9, 128, 64, 64 * 30 - 7
    gen = torch.Generator(device=DEV).manual_seed(1)
    raw = [torch.randn((B, H, n_text + n_image, D), generator=gen, device=DEV).to(torch.bfloat16) for _ in range(3)]
    q, k, out = (torch.empty_like(raw[0]) for _ in range(3))
    gain = [0.5 + torch.rand(D, generator=gen, device=DEV) for _ in range(2)]
    ctx = binding.Context(B, H, D, n_text, n_image)
    n0 = ctx.launch_count()
    ctx.rapid3_gated_step_fused(*raw, *gain, None, 1e-6, q, k, out, [2] * B, [0.5, 0.3])
    assert ctx.launch_count() - n0 == 3                            # producer, scores and selection, attention
    ws = [t.clone() for t in ctx.workspace(B)]
    scores = ctx.rapid3_block_scores(q, k)
    assert torch.equal(bits(ws[0]), bits(scores))
    for got, ref in zip(ws[1:], ctx.rapid3_select_mask(scores, [0.5, 0.3])):
        assert torch.equal(got, ref)
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
