"""Selection at the row lengths where the kernels change the number of registers that hold a row (96, 192, 288, 512 and 768
blocks), around whole warps, and at the shortest rows; scores of both signs over many powers of two, with runs of equal ones."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_22323_b200 import binding
from tests import parity

pytestmark = pytest.mark.gpu
DEV = "cuda"
RATIOS = (0.02, 0.3, 0.5, 0.97)


def make_scores(nb, n_img, H, seed):
    rng = np.random.default_rng(seed)
    S = rng.standard_normal((n_img, H, nb, nb)) * np.exp2(rng.integers(-60, 20, (n_img, H, nb, nb)))
    S[:, 0] = rng.choice(S[0, 0].ravel()[:5], (n_img, nb, nb))          # five values: ties everywhere
    return S.astype(np.float32)


@pytest.mark.parametrize("nb", [1, 2, 31, 32, 33, 34, 35, 95, 96, 97, 287, 288, 289])
@pytest.mark.parametrize("text_blocks", [0, 1, 3])
def test_top_k(nb, text_blocks):
    if text_blocks > nb:
        pytest.skip("no such sequence")
    n_text = 64 * text_blocks
    S = make_scores(nb, len(RATIOS), 2, 31 * nb + text_blocks)
    ctx = binding.Context(len(RATIOS), 2, 64, n_text, 64 * nb - n_text)
    bitmask, idx, cnt = ctx.rapid3_select_mask(torch.from_numpy(S).to(DEV), list(RATIOS))
    torch.cuda.synchronize()
    dense = binding.bitmask_to_dense(bitmask, nb).numpy()
    parity.check_lists(idx, cnt, dense)
    parity.check_padding_bits(bitmask, nb)
    for p, r in enumerate(RATIOS):
        want, _ = oracle.select_mask(S[p].astype(np.float64), n_text, r)
        np.testing.assert_array_equal(dense[p], want)


@pytest.mark.parametrize("nb", [2, 33, 96, 97, 288, 289])
def test_mass_counts(nb):
    shares, scale = (1e-6, 0.3, 0.9, 1.0), 0.5
    rng = np.random.default_rng(nb)
    S = rng.standard_normal((len(shares), 2, nb, nb)).astype(np.float32) * 4
    S[:, 0, ::2] = np.round(S[:, 0, ::2])                               # rows with equal scores
    ctx = binding.Context(len(shares), 2, 64, 0, 64 * nb)
    keep, bitmask, idx, cnt = ctx.rapid3_select_mask_mass(torch.from_numpy(S).to(DEV), list(shares), scale)
    torch.cuda.synchronize()
    parity.check_lists(idx, cnt, binding.bitmask_to_dense(bitmask, nb).numpy())
    keep = keep.cpu().numpy()
    for p, tau in enumerate(shares):
        for h in range(2):
            for i in range(nb):
                s = np.sort(np.delete(S[p, h, i].astype(np.float64), i))[::-1]
                c = np.cumsum(np.exp(scale * (s - s[0])))
                target = float(np.float32(tau)) * c[-1]
                want = len(s) if tau >= 1 else int(np.searchsorted(c, target) + 1)
                # another order of 64-bit sums may fall on the other side only this close to the target
                if want != keep[p, h, i]:
                    assert abs(c[min(want, keep[p, h, i]) - 1] - target) <= 1e-12 * c[-1], (p, h, i, want, keep[p, h, i])


@pytest.mark.parametrize("nb", [191, 192, 193, 511, 512, 513, 767, 768, 769])
def test_both_rules_where_the_count_changes(nb):
    """Two heads each: the top-k masks against the oracle, and the cumulative-mass masks against the oracle's top-k at the
    counts that the rule arrived at, which are checked as above."""
    S = make_scores(nb, 2, 2, nb)
    S[1] = np.random.default_rng(nb).standard_normal((2, nb, nb)).astype(np.float32)
    ctx = binding.Context(2, 2, 64, 64, 64 * nb - 64)
    bitmask, idx, cnt = ctx.rapid3_select_mask(torch.from_numpy(S).to(DEV), [0.3125, 0.5])
    keep, bitmask_m, idx_m, cnt_m = ctx.rapid3_select_mask_mass(torch.from_numpy(S[1:]).to(DEV), [0.5], 1.0)
    torch.cuda.synchronize()
    dense = binding.bitmask_to_dense(bitmask, nb).numpy()
    parity.check_lists(idx, cnt, dense)
    parity.check_padding_bits(bitmask, nb)
    for p, r in enumerate((0.3125, 0.5)):             # exact as 32-bit floats, as the interface hands them on
        want, _ = oracle.select_mask(S[p].astype(np.float64), 64, r)
        np.testing.assert_array_equal(dense[p], want)
    dense_m = binding.bitmask_to_dense(bitmask_m, nb).numpy()
    parity.check_lists(idx_m, cnt_m, dense_m)
    keep = keep.cpu().numpy()
    for h in range(2):
        for i in range(1, nb):
            free = np.delete(np.arange(1, nb), i - 1)
            order = free[np.argsort(-S[1, h, i, free].astype(np.float64), kind="stable")]
            c = np.cumsum(np.exp(S[1, h, i, order].astype(np.float64) - float(S[1, h, i, order[0]])))
            n = keep[0, h, i]
            # another order of 64-bit sums may fall on the other side only this close to the target
            assert c[n - 1] >= (0.5 - 1e-12) * c[-1] and (n == 1 or c[n - 2] <= (0.5 + 1e-12) * c[-1]), (h, i, n)
            assert dense_m[0, h, i].sum() == n + 2 and dense_m[0, h, i, order[:n]].all()
