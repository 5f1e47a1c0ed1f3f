"""Contexts of few quads: the attention works on a quad's key blocks in parts, whose results a second kernel adds up.
Against attention in 64 bits at lists of every kind (full, short, empty, shorter than the number of parts), and what an
image gets does not depend on the launch: the images of a batch equal the same images alone, decisions on the GPU equal
decisions on the host, bit for bit."""
import pytest
import torch

from paper_2509_22323_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda"


def attention_64(q, k, v, keep):
    """[N, D] each and keep [nb, nb] -> softmax attention over the kept blocks in 64 bits; zero where nothing is kept."""
    at = torch.arange(q.shape[0], device=q.device) // 64
    s = (q.double() @ k.double().T) * q.shape[1] ** -0.5
    return s.masked_fill(~keep[at][:, at], float("-inf")).softmax(-1).nan_to_num(0.0) @ v.double()


def random_qkv(shape, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    return [torch.randn(shape, generator=gen, device=DEV).to(torch.bfloat16) for _ in range(3)], gen


SHAPES = [                        # D, text, image tokens, H, B; parts of dense / text / other quads' lists
    (64, 77, 33 * 64 - 90, 2, 1),      # 8 / 8 / 3, ragged tail
    (128, 77, 34 * 64 - 77, 2, 1),     # 4 / 8 / 3
    (128, 512, 36 * 64 - 512, 3, 1),   # 5 / 7 / 4
    (64, 130, 51 * 64 - 200, 2, 2),    # 5 / 7 / 5, text and image rows in one quad
    (128, 0, 72 * 64 - 63, 2, 1),      # 4 / - / 4, one token in the last block
    (128, 512, 128 * 128, 2, 1),       # 1 / 4 / 1: text rows alone, column quads
]


@pytest.mark.parametrize("D,n_text,n_image,H,B", SHAPES)
def test_parts_of_lists_against_64_bits(D, n_text, n_image, H, B):
    N = n_text + n_image
    nb = (N + 63) // 64
    (q, k, v), gen = random_qkv((B, H, N, D), D + nb)
    keep = torch.rand((B, H, nb, nb), generator=gen, device=DEV) < torch.rand((B, H, nb, 1), generator=gen, device=DEV)
    keep[:, :, 0::7] = False                                       # rows that keep nothing
    keep[:, :, 1::7] = torch.arange(nb, device=DEV) == 3           # one block
    keep[:, 0, 4:8] = False                                        # a quad that keeps nothing
    keep[:, H - 1, -1] = True
    cnt = keep.sum(-1).to(torch.int32)
    at = torch.arange(nb, device=DEV, dtype=torch.int32)
    idx = torch.where(keep, at, nb).sort(dim=-1).values
    idx = torch.where(idx < nb, idx, -1).to(torch.int32).contiguous()
    ctx = binding.Context(B, H, D, n_text, n_image)
    out, dense = torch.full_like(q, float("nan")), torch.full_like(q, float("nan"))
    n0 = ctx.launch_count()
    ctx.rapid3_sparse_joint_attn(q, k, v, out, kept_idx=idx, kept_cnt=cnt)
    assert ctx.launch_count() - n0 == 2                            # attention, sum of the parts
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


@pytest.mark.parametrize("D,n_text,n_image,H", [(64, 77, 36 * 64, 1), (128, 200, 30 * 64, 1)])
def test_an_image_of_a_context_with_parts_does_not_depend_on_its_launch(D, n_text, n_image, H):
    B, N = 2, n_text + n_image
    (q, k, v), _ = random_qkv((B, H, N, D), 5)
    ctx = binding.Context(B, H, D, n_text, n_image)
    for ratios in ([1.0, 1.0], [0.4, 1.0], [0.3, 0.7]):
        out, alone, dev = (torch.full_like(q, float("nan")) for _ in range(3))
        n0 = ctx.launch_count()
        ctx.rapid3_gated_step(q, k, v, out, [2, 2], ratios)
        assert ctx.launch_count() - n0 == (5 if min(ratios) < 1.0 else 2)
        ctx.rapid3_gated_step(q, k, v, alone, [2, 0], ratios)
        ctx.rapid3_gated_step(q, k, v, alone, [0, 2], ratios)
        ctx.rapid3_gated_step_device(q, k, v, dev, torch.tensor([2, 2], dtype=torch.int32, device=DEV),
                                     torch.tensor(ratios, device=DEV))
        torch.cuda.synchronize()
        assert ctx.last_status() == 0
        assert torch.equal(out.view(torch.int16), alone.view(torch.int16))
        assert torch.equal(out.view(torch.int16), dev.view(torch.int16))
        assert torch.isfinite(out).all()


@pytest.mark.parametrize("D,n_text,n_image,H,B", SHAPES)
@pytest.mark.parametrize("finite", ["ends", "even"])
def test_blocks_whose_scores_are_below_all_numbers(D, n_text, n_image, H, B, finite):
    """Finite numbers whose products with Q leave the range of single precision downwards, in whole key blocks: such a block counts
    for nothing, wherever a part of a list begins (behind the row's first block)."""
    N = n_text + n_image
    nb = (N + 63) // 64
    (q, k, v), _ = random_qkv((B, H, N, D), nb)
    at = torch.arange(nb, device=DEV)
    low = (at % 2 == 1) if finite == "even" else (at > 0) & (at < nb - 1)
    q[..., 0] = 8.0
    k[..., 0] = torch.where(low[torch.arange(N, device=DEV) // 64], torch.finfo(torch.bfloat16).min, k[..., 0])
    ctx, out = binding.Context(B, H, D, n_text, n_image), torch.full_like(q, float("nan"))
    ctx.rapid3_gated_step(q, k, v, out, [2] * B, [1.0] * B)
    ratios = [0.5] * B
    sparse = torch.full_like(q, float("nan"))
    ctx.rapid3_gated_step(q, k, v, sparse, [2] * B, ratios)
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
    keep = binding.bitmask_to_dense(ctx.workspace(B)[1], nb).bool().to(DEV)
    for b in range(B):
        for h in range(H):
            for o, mask in ((out, torch.ones_like(keep[b, h])), (sparse, keep[b, h])):
                ref = attention_64(q[b, h], k[b, h], v[b, h], mask)
                first = mask.int().argmax(-1)                      # a row's first block has numbers here: kept by all rows if it is text
                rows = (~low[first]).repeat_interleave(64)[:N]
                assert float((o[b, h].double() - ref).abs()[rows].max()) <= 2 ** -7 * float(v[b, h].abs().max())
