"""GPU: fp32 forward with infinite scores.  A row whose every score is -inf has no
softmax (0 / 0): O is NaN, unlike a row that lists nothing (O = 0)."""
import numpy as np
import pytest
import torch

from gpu_util import F32_MAX_ABS, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("N,d,b", [(200, 64, 32), (300, 128, 64), (700, 64, 128)])
def test_rows_of_minus_infinity(N, d, b):
    from paper_2609_23169_gb300 import ultratex as u
    H = 2
    g = torch.Generator(device="cuda").manual_seed(N)
    q, k, v = (torch.randn((N, H, d), generator=g, device="cuda") for _ in range(3))
    k = k.abs() + 0.1
    rows = torch.arange(5, N, 37, device="cuda")
    q[rows] = -float("inf")            # every score -inf
    q[0] = 1.0
    k[1, :, 0] = -float("inf")         # one key whose score with row 0 is -inf: weight 0
    nb = -(-N // b)
    bm = torch.ones((H, nb, nb), dtype=torch.uint8, device="cuda")
    bm[1, nb - 1] = 0                  # an empty list
    bm[:, 1:, 0] = 0                   # key 1 is seen by the first block only
    shape = u.attn_shape(q, b)
    rp, ci, _, _ = u.ut_block_mask(shape, u.UT_MASK_BITMAP, bitmap=bm, with_transpose=False)
    o, lse = u.ut_bsattn_fwd(q, k, v, rp, ci, b)
    empty = torch.zeros((H, N), dtype=torch.bool, device="cuda")
    empty[1, (nb - 1) * b:] = True
    low = torch.zeros((H, N), dtype=torch.bool, device="cuda")
    low[:, rows] = True
    low &= ~empty
    assert bool((lse[empty | low] == -float("inf")).all())
    assert bool((o[empty.t()] == 0).all())
    # rows of the first block meet -inf * -inf = inf with key 1
    far = low.clone()
    far[:, :b] = False
    assert bool(torch.isnan(o[far.t()]).all())
    keep = bm.bool().repeat_interleave(b, 1).repeat_interleave(b, 2)[:, :N, :N]
    s = (torch.einsum("nhd,mhd->hnm", q.double(), k.double()) * d ** -0.5).masked_fill(~keep, -float("inf"))
    ref = torch.einsum("hnm,mhd->nhd", torch.softmax(s, 2), v.double())
    assert float((o[0].double() - ref[0]).abs().max()) <= F32_MAX_ABS
    fine = ~(empty | low)
    fine[:, :b] = False
    assert float((o[fine.t()].double() - ref[fine.t()]).abs().max()) <= F32_MAX_ABS
