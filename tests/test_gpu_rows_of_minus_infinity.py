"""Rows whose every kept score is -inf (finite numbers whose products leave the range of single precision): softmax has 0 / 0 there, and the
result is not a number, whether the context works on whole lists, on blocks by turns or on lists in parts.  Rows that keep nothing stay 0."""
import pytest
import torch

from paper_2509_22323_b200 import binding
from tests.test_gpu_list_parts import attention_64, random_qkv

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("D,n_text,n_blocks,H", [
    (64, 64, 5, 2), (128, 64, 7, 2),            # whole lists, a tile an SM
    (64, 64, 40, 70),                           # whole lists, both tiles
    (64, 64, 13, 2), (128, 64, 20, 2),          # blocks by turns
    (64, 64, 40, 2), (128, 64, 36, 2),          # lists in parts
    (128, 512, 264, 2),                         # text rows alone in parts
])
def test_rows_of_minus_infinity_are_not_numbers(D, n_text, n_blocks, H):
    (q, k, v), _ = random_qkv((1, H, 64 * n_blocks, D), n_blocks)
    q = q.abs()
    k[:, -1, 64:] = -3e38                                          # the last head's, but for its first block
    ctx = binding.Context(1, H, D, n_text, 64 * n_blocks - n_text)
    keep = torch.zeros((1, H, n_blocks, n_blocks), dtype=torch.bool, device=DEV)
    keep[:, :, 0::4, 1:] = True                                    # without the first block
    keep[:, :, 1::4, n_blocks // 2] = True                         # one block
    keep[:, :, 2::4, 0::2] = True                                  # with the first block; rows 3, 7, ... keep nothing
    cnt = keep.sum(-1).to(torch.int32)
    at = torch.arange(n_blocks, device=DEV, dtype=torch.int32)
    idx = torch.where(keep, at, n_blocks).sort(dim=-1).values
    idx = torch.where(idx < n_blocks, idx, -1).to(torch.int32).contiguous()
    out = torch.full_like(q, float("nan"))
    ctx.rapid3_sparse_joint_attn(q, k, v, out, kept_idx=idx, kept_cnt=cnt)
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
    def of(block):                                                 # the rows of every fourth query block
        return (torch.arange(64 * n_blocks, device=DEV) // 64) % 4 == block
    assert out[0, -1, of(0)].isnan().all() and out[0, -1, of(1)].isnan().all()
    assert (out[0, :, of(3)] == 0).all()
    for h in (0, H - 1):                                           # P and the result rounded to bf16 once each
        rest, rows = keep[0, h].clone(), torch.ones_like(of(0))
        if h == H - 1:
            rest[:, 1:] = False                                    # a score of -inf counts for nothing beside numbers
            rows = of(2)
        ref = attention_64(q[0, h], k[0, h], v[0, h], rest)
        assert float((out[0, h].double() - ref)[rows].abs().max()) <= 2 ** -7 * float(v[0, h].abs().max())
    k[:, -1] = -3e38
    dense = torch.zeros_like(q)
    ctx.rapid3_sparse_joint_attn(q, k, v, dense)
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
    assert dense[:, -1].isnan().all() and dense[:, :-1].isfinite().all()
