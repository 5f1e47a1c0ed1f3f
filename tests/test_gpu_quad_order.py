"""Launches of some hundred quads hand their last ones out by length.  In which order a quad is worked on does not touch its
result: every image of such a step equals the same image alone, whose few quads come in order, bit for bit -- for
every selection rule, for batches whose last quads are all, some and not any of the ordered ones, and for decisions on the GPU."""
import pytest
import torch

from paper_2509_22323_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("D,n_text,n_image,H,B", [
    (64, 77, 2400, 8, 4),        # 320 quads, all of those without text in the order; text and image rows in one quad
    (128, 0, 9 * 64 + 5, 25, 4),  # 300 quads, ragged, no text
    (128, 128, 1111, 16, 8),     # 640 quads: the first of those without text come as they are
    (64, 64, 128 * 128, 4, 3),   # 780 quads of two-block grid rows
    (64, 512, 128 * 128, 2, 4),  # 528 column quads
])
def test_ordered_quads_equal_quads_in_order(D, n_text, n_image, H, B):
    N = n_text + n_image
    gen = torch.Generator(device=DEV).manual_seed(N)
    q, k, v = (torch.randn((B, H, N, D), generator=gen, device=DEV).to(torch.bfloat16) for _ in range(3))
    ctx = binding.Context(B, H, D, n_text, n_image)
    ratios = [(0.3, 1.0, 0.7, 0.15)[b % 4] for b in range(B)]
    per_head = [[min(1.0, ratios[b] * (0.5, 1.0, 1.5)[h % 3]) for h in range(H)] for b in range(B)]
    calls = {
        "step": lambda out, acts: ctx.rapid3_gated_step(q, k, v, out, acts, ratios),
        "heads": lambda out, acts: ctx.rapid3_gated_step_heads(q, k, v, out, acts, per_head),
        "mass": lambda out, acts: ctx.rapid3_gated_step_mass(q, k, v, out, acts, ratios, 4 * D ** -0.5),
        "device": lambda out, acts: ctx.rapid3_gated_step_device(q, k, v, out, torch.tensor(acts, dtype=torch.int32, device=DEV),
                                                                 torch.tensor(ratios, device=DEV)),
    }
    for name, call in calls.items():
        for acts in ([2] * B, [2] * (B - 1) + [1]):
            out, alone = torch.full_like(q, float("nan")), torch.full_like(q, float("nan"))
            for _ in range(2):                                     # the counts of the step before are gone
                call(out, acts)
            for b in range(B):
                if acts[b] == 2:
                    (calls["step"] if name == "device" else call)(alone, [2 if i == b else 0 for i in range(B)])
            torch.cuda.synchronize()
            assert ctx.last_status() == 0
            assert torch.equal(out.view(torch.int16), alone.view(torch.int16)), (name, acts)
            assert torch.isfinite(out[[a == 2 for a in acts]]).all()


@pytest.mark.parametrize("D,n_text,n_image,H,B", [
    (64, 77, 75, 4, 2),          # 8 quads
    (128, 0, 12 * 64 + 1, 8, 6),  # 192
    (64, 130, 16 * 64, 15, 4),   # 300, ordered
    (128, 77, 9 * 64, 40, 9),    # 1080
    (64, 0, 5 * 64 + 63, 64, 8),  # 1024
])
def test_masks_and_lists_give_the_same(D, n_text, n_image, H, B):
    """The attention of a step reads the selection's bitmask, the staged call its kept lists: the same outputs, bit for bit."""
    gen = torch.Generator(device=DEV).manual_seed(H)
    q, k, v = (torch.randn((B, H, n_text + n_image, D), generator=gen, device=DEV).to(torch.bfloat16) for _ in range(3))
    ctx = binding.Context(B, H, D, n_text, n_image)
    step, staged = torch.full_like(q, float("nan")), torch.full_like(q, float("nan"))
    ratios = [(0.3, 0.95, 0.7, 0.15)[b % 4] for b in range(B)]
    ctx.rapid3_gated_step(q, k, v, step, [2] * B, ratios)
    idx, cnt = (t.clone() for t in ctx.workspace(B)[2:])
    ctx.rapid3_sparse_joint_attn(q, k, v, staged, kept_idx=idx, kept_cnt=cnt)
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
    assert torch.equal(step.view(torch.int16), staged.view(torch.int16))


@pytest.mark.parametrize("D,n_text,n_image,H,B", [
    (64, 0, 17 * 64 - 3, 17, 3),   # 255 quads, the first 148 of a step without dense images come as they are
    (128, 200, 800, 26, 2),        # 208: 130 dense or with text, of the others the first 18 come as they are
    (64, 512, 8 * 64 + 1, 40, 2),  # 400: every SM begins with a dense quad or one with text
    (64, 512, 60, 67, 1),          # 201: one quad in three has no text, fewer than the SMs begin with
])
def test_ordered_quads_behind_those_that_the_sms_begin_with(D, n_text, n_image, H, B):
    test_ordered_quads_equal_quads_in_order(D, n_text, n_image, H, B)
