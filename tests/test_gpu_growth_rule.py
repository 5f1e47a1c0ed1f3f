"""The rule by which a row's reference maximum moves: a P above 2^8, seen in the partial sum of eight that it is part of.
Scores that rise from key block to key block by steps below, around and far above what the rule lets pass, in few keys of
a block or in all; and values so large that P must not exceed 1 by more than that."""
import math

import pytest
import torch

from paper_2509_22323_b200 import binding

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("step", [4.0, 12.9, 13.1, 15.9, 16.1, 19.0, 200.0])
@pytest.mark.parametrize("every", [1, 64])
def test_scores_rising_by_steps(D, step, every):
    H, N = 2, 640 + 21
    gen = torch.Generator(device=DEV).manual_seed(int(10 * step) + D + every)
    q, k, v = (torch.randn((1, H, N, D), generator=gen, device=DEV) for _ in range(3))
    at = torch.arange(N, device=DEV)
    # channel 0 alone decides: step (in powers of two) per key block, in every `every`-th key; the others stay at 0
    rise = torch.where(at % every == 0, step * (at // 64), 0.0)
    q[..., 0], q[..., 1:] = 8.0, 0.1 * q[..., 1:]
    k[..., 0], k[..., 1:] = rise * math.log(2.0) * D ** 0.5 / 8.0, 0.1 * k[..., 1:]
    q, k, v = (t.to(torch.bfloat16) for t in (q, k, v))
    ctx = binding.Context(1, H, D, 0, N)
    out = torch.full_like(q, float("nan"))
    ctx.rapid3_gated_step(q, k, v, out, [2], [1.0])
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
    ref = (q[0].double() @ k[0].double().transpose(1, 2) * D ** -0.5).softmax(-1) @ v[0].double()
    # P and the result are rounded to bf16 (2^-9 each, relative to the values' range); scores up to 2000 in powers of
    # two are 32-bit products, 2^-24 x 2000 x ln 2 relative in P
    assert float((out[0].double() - ref).abs().max()) <= 2 ** -7 * float(v.abs().max())


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("scale", [1e3, 1e5, 1e7, 1e12])
def test_scores_whose_rounding_exceeds_the_rule(D, scale):
    """Scores so large that the rounding of their scaled value alone is worth more than 2^16 in P: no maximum can bring
    the partial sums under the rule, and the pass must end all the same."""
    gen = torch.Generator(device=DEV).manual_seed(D)
    q, k, v = (torch.randn((1, 2, 300, D), generator=gen, device=DEV) for _ in range(3))
    q, k, v = (q * scale).to(torch.bfloat16), (k * scale).to(torch.bfloat16), v.to(torch.bfloat16)
    ctx = binding.Context(1, 2, D, 0, 300)
    out = torch.full_like(q, float("nan"))
    ctx.rapid3_gated_step(q, k, v, out, [2], [1.0])
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
    if scale <= 1e3:                     # beyond, P itself may leave the range of 32-bit floats
        s = q[0].double() @ k[0].double().transpose(1, 2) * D ** -0.5
        ref = s.softmax(-1) @ v[0].double()
        clear = (s.topk(2, dim=-1).values.diff(dim=-1).squeeze(-1) < -100.0)     # one key decides, in any arithmetic
        assert bool(clear.any())
        assert float((out[0].double() - ref).abs()[clear].max()) <= 2 ** -7 * float(v.abs().max())


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("step", [7.9, 8.1, 12.9])
def test_values_near_the_end_of_their_range(D, step):
    """The accumulator holds a row's sum of P times a value: with P up to 2^8, 661 keys and values of 2^109 to 2^110 that
    is less than 2^128; with P of 2^12.9 in a block of 64 keys it is not."""
    H, N = 2, 640 + 21
    gen = torch.Generator(device=DEV).manual_seed(int(10 * step) + D)
    q, k, v = (torch.randn((1, H, N, D), generator=gen, device=DEV) for _ in range(3))
    q[..., 0], q[..., 1:] = 8.0, 0.1 * q[..., 1:]
    k[..., 0], k[..., 1:] = step * (torch.arange(N, device=DEV) // 64) * math.log(2.0) * D ** 0.5 / 8.0, 0.1 * k[..., 1:]
    v = (v.abs() % 2.0 + 2.0) * 2.0 ** 108
    q, k, v = (t.to(torch.bfloat16) for t in (q, k, v))
    ctx = binding.Context(1, H, D, 0, N)
    out = torch.full_like(q, float("nan"))
    ctx.rapid3_gated_step(q, k, v, out, [2], [1.0])
    torch.cuda.synchronize()
    assert ctx.last_status() == 0
    ref = (q[0].double() @ k[0].double().transpose(1, 2) * D ** -0.5).softmax(-1) @ v[0].double()
    assert float((out[0].double() - ref).abs().max()) <= 2 ** -7 * float(v.double().abs().max())    # as above
