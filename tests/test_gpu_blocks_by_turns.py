"""Contexts in which every tile of the largest launch has an SM to itself: a tile's key blocks go to the SM's two tiles by turns, whose
results are put together at the end.  Lists of no block, of one, of odd and of even numbers, ragged last quads and last blocks, rows
that keep nothing in one of the two, against attention in 64 bits; steps against the staged calls and an image alone, bit for bit."""
import pytest
import torch

from paper_2509_22323_b200 import binding
from tests.test_gpu_list_parts import attention_64, random_qkv

pytestmark = pytest.mark.gpu
DEV = "cuda"
SHAPES = [  # D, text and image tokens, heads, images
    (64, 0, 5 * 64 + 1, 1, 1),       # the shortest rows, one token in the last block
    (64, 77, 13 * 64, 3, 2),         # a quad of three rows, 61 tokens in the last block
    (64, 130, 22 * 64 + 5, 12, 1),   # 72 quads
    (128, 64, 7 * 64, 2, 3),         # the shortest rows
    (128, 200, 19 * 64 + 1, 6, 2),   # 72 quads, one token in the last block
]


@pytest.mark.parametrize("D,n_text,n_image,H,B", SHAPES)
def test_lists_by_turns_against_64_bits(D, n_text, n_image, H, B):
    N = n_text + n_image
    nb = (N + 63) // 64
    (q, k, v), gen = random_qkv((B, H, N, D), D + nb)
    keep = torch.rand((B, H, nb, nb), generator=gen, device=DEV) < torch.rand((B, H, nb, 1), generator=gen, device=DEV)
    keep[:, :, 0::5] = False                                       # rows that keep nothing
    keep[:, :, 1::5] = torch.arange(nb, device=DEV) == nb - 1      # one block
    keep[:, :, 2::5] = torch.arange(nb, device=DEV) % 2 == 0       # where their neighbours keep none, all of one tile's turns
    keep[0, 0] &= (torch.arange(nb, device=DEV) >= 4)[:, None]     # a quad that keeps nothing
    cnt = keep.sum(-1).to(torch.int32)
    at = torch.arange(nb, device=DEV, dtype=torch.int32)
    idx = torch.where(keep, at, nb).sort(dim=-1).values
    idx = torch.where(idx < nb, idx, -1).to(torch.int32).contiguous()
    ctx = binding.Context(B, H, D, n_text, n_image)
    out, dense = torch.full_like(q, float("nan")), torch.full_like(q, float("nan"))
    for _ in range(2):
        ctx.rapid3_sparse_joint_attn(q, k, v, out, kept_idx=idx, kept_cnt=cnt)
        ctx.rapid3_sparse_joint_attn(q, k, v, dense)
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
    # P and the result are rounded to bf16 once each: 2^-9 relative to the values' range
    for b in range(B):
        for h in range(H):
            for o, mask in ((out, keep[b, h]), (dense, torch.ones_like(keep[b, h]))):
                ref = attention_64(q[b, h], k[b, h], v[b, h], mask)
                assert float((o[b, h].double() - ref).abs().max()) <= 2 ** -7 * float(v[b, h].abs().max())
    rows = (cnt == 0).repeat_interleave(64, dim=2)[:, :, :N]
    assert (out[rows] == 0).all()


@pytest.mark.parametrize("D,n_text,n_image,H,B", SHAPES[1:])
def test_steps_by_turns_equal_the_stages_and_the_images_alone(D, n_text, n_image, H, B):
    (q, k, v), _ = random_qkv((B, H, n_text + n_image, D), 3)
    ratios = [(0.4, 1.0, 0.2)[b % 3] for b in range(B)]
    ctx = binding.Context(B, H, D, n_text, n_image)
    out, alone, dev, staged = (torch.full_like(q, float("nan")) for _ in range(4))
    ctx.rapid3_gated_step(q, k, v, out, [2] * B, ratios)
    for b in range(B):
        ctx.rapid3_gated_step(q, k, v, alone, [2 if i == b else 0 for i in range(B)], ratios)
    ctx.rapid3_gated_step_device(q, k, v, dev, torch.full((B,), 2, dtype=torch.int32, device=DEV), torch.tensor(ratios, device=DEV))
    _, idx, cnt = ctx.rapid3_select_mask(ctx.rapid3_block_scores(q, k), ratios)
    ctx.rapid3_sparse_joint_attn(q, k, v, staged, kept_idx=idx, kept_cnt=cnt)
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
    for t in (alone, dev, staged):
        assert torch.equal(out.view(torch.int16), t.view(torch.int16))


@pytest.mark.parametrize("D", [64, 128])
def test_scores_of_minus_infinity_in_one_turn(D):
    """A tile whose first block has scores of -inf alone (finite numbers whose products leave the range) counts for nothing there."""
    H, nb = 2, 12
    (q, k, v), _ = random_qkv((1, H, nb * 64, D), 9)
    q, k = q.abs(), k.abs()
    k[:, :, :64] = -3e38
    out = torch.full_like(q, float("nan"))
    ctx = binding.Context(1, H, D, 0, nb * 64)
    ctx.rapid3_sparse_joint_attn(q, k, v, out)
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
    keep = torch.arange(nb, device=DEV).expand(nb, nb) > 0
    for h in range(H):
        ref = attention_64(q[0, h], k[0, h], v[0, h], keep)
        assert float((out[0, h].double() - ref).abs().max()) <= 2 ** -7 * float(v.abs().max())


@pytest.mark.parametrize("D,n_blocks,H", [(64, 6, 18), (64, 22, 3), (128, 8, 37), (128, 20, 1)])
def test_steps_by_turns_queued_equal_steps_alone(D, n_blocks, H):
    """Every thread block's list is there long before its other warps are through with the set-up, or late, behind a selection: steps
    queued without a wait give what each gives alone."""
    (q, k, v), _ = random_qkv((1, H, 64 * n_blocks, D), n_blocks)
    ctx = binding.Context(1, H, D, 64, 64 * (n_blocks - 1))
    ratios = (1.0, 0.3, 1.0, 0.8)
    alone = []
    for r in ratios:
        alone.append(torch.full_like(q, float("nan")))
        ctx.rapid3_gated_step(q, k, v, alone[-1], [2], [r])
        torch.cuda.synchronize()
    outs = [torch.full_like(q, float("nan")) for _ in range(32)]
    for _ in range(8):
        for n, o in enumerate(outs):
            ctx.rapid3_gated_step(q, k, v, o, [2], [ratios[n % 4]])
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
    for n, o in enumerate(outs):
        assert torch.equal(o.view(torch.int16), alone[n % 4].view(torch.int16)), n
