"""A thread block of the attention kernel works through many quads of query blocks, each role at its own pace.  What
an image gets must not depend on what else the launch holds: every image of a large batch, whose kept lists mix full,
short and empty rows, equals the same image run alone (a quad or half of one per thread block) bit for bit, and rows
that keep nothing are zero."""
import pytest
import torch

from paper_2509_22323_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("D,n_text,n_image,H", [
    (64, 0, 64, 24),          # one block, one quad per head
    (128, 77, 200, 24),       # five blocks: the second quad has one query block, the last block 21 tokens
    (128, 64, 1000, 12),      # seventeen blocks: more than the ring holds
    (64, 333, 2025, 6),       # thirty-seven blocks, ragged
    (128, 128, 128 * 128, 1),  # two blocks a grid row after half a quad of text: vertical tiles
])
def test_images_of_a_batch_equal_images_alone(D, n_text, n_image, H):
    B, N = 16, n_text + n_image
    if N > 8192:
        B = 4
    nb = (N + 63) // 64
    gen = torch.Generator(device=DEV).manual_seed(D + nb)
    q, k, v = (torch.randn((B, H, N, D), generator=gen, device=DEV).to(torch.bfloat16) for _ in range(3))
    share = torch.rand((B, H, nb, 1), generator=gen, device=DEV)
    keep = torch.rand((B, H, nb, nb), generator=gen, device=DEV) < share
    keep[:, 0, 1::3] = False                                       # rows that keep nothing
    keep[1] = False                                                # an image whose every list is empty
    keep[2] = True
    cnt = keep.sum(-1).to(torch.int32)
    at = torch.arange(nb, device=DEV, dtype=torch.int32)
    idx = torch.where(keep, at, nb).sort(dim=-1).values
    idx = torch.where(idx < nb, idx, -1).to(torch.int32).contiguous()
    ctx = binding.Context(B, H, D, n_text, n_image)
    out = torch.full_like(q, float("nan"))
    ctx.rapid3_sparse_joint_attn(q, k, v, out, kept_idx=idx, kept_cnt=cnt)
    alone = torch.full_like(q, float("nan"))
    for b in range(B):
        ctx.rapid3_sparse_joint_attn(q, k, v, alone, img_idx=[b], kept_idx=idx[b:b + 1].contiguous(),
                                     kept_cnt=cnt[b:b + 1].contiguous())
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
    assert torch.equal(out.view(torch.int16), alone.view(torch.int16))
    rows = (cnt == 0).repeat_interleave(64, dim=2)[:, :, :N]
    assert (out[rows] == 0).all()
    # against attention in 64 bits: P and the result are rounded to bf16 once each (2^-9 relative to the values' range)
    b, h = 0, H - 1
    mask = keep[b, h].repeat_interleave(64, 0)[:N].repeat_interleave(64, 1)[:, :N]
    s = (q[b, h].double() @ k[b, h].double().T) * D ** -0.5
    p = s.masked_fill(~mask, float("-inf")).softmax(-1).nan_to_num(0.0)
    ref = p @ v[b, h].double()
    assert float((out[b, h].double() - ref).abs().max()) <= 2 ** -7 * float(v[b, h].abs().max())
