"""GPU: Top-K lists where many scores are equal, at every form of the selection
(N_k in registers at 8, 16, 24 and 32 keys a lane, and beyond), and the transpose
by both of its ways of counting.  Blocks are powers of two that divide N and
entries small integers, so pooled means, products and sums are exact in fp32 and
the lists are those of a stable sort by falling score."""
import numpy as np
import pytest
import torch

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("N,H,b,bk,k", [(240, 3, 8, 1, 17), (512, 2, 16, 2, 100), (500, 1, 4, 1, 1), (700, 1, 4, 1, 699),
                                        (1024, 2, 32, 1, 333), (1100, 2, 4, 1, 500), (6000, 1, 2, 2, 700), (6000, 1, 2, 2, 3),
                                        (9000, 1, 8, 1, 4000)])
def test_equal_scores_go_to_the_smaller_index(N, H, b, bk, k):
    from paper_2609_23169_gb300 import ultratex as u
    d = 64
    g = np.random.Generator(np.random.PCG64([85, N, k]))
    q, kk = (np.repeat(g.integers(-2, 3, (N, H, d // 8)).astype(np.float32), 8, 2) for _ in range(2))
    nq, nk = N // b, N // bk
    rho = (k + 0.5) / nk
    assert u.ut_topk_count(rho, nk) == k
    shape = u.AttnShape(N, H, d, b, u.UT_F32, H * d, bk)
    rp, ci, cp, ri = (t.cpu().numpy() for t in u.ut_block_mask(shape, u.UT_MASK_TOPK, torch.from_numpy(q).cuda(),
                                                               torch.from_numpy(kk).cuda(), rho))
    pq, pk = (x.astype(np.float64).reshape(N // y, y, H, d).mean(1) for x, y in ((q, b), (kk, bk)))
    sc = np.einsum("ihd,jhd->hij", pq, pk)
    want = np.sort(np.argsort(-sc, axis=2, kind="stable")[:, :, :k], axis=2)
    assert np.array_equal(rp, np.arange(H * nq + 1) * k)
    assert np.array_equal(ci[:H * nq * k].reshape(H, nq, k), want)
    keep = np.zeros((H, nq, nk), bool)
    np.put_along_axis(keep, want, True, 2)
    pairs = np.argwhere(keep.transpose(0, 2, 1))
    assert np.array_equal(cp, np.concatenate([[0], np.cumsum(keep.sum(1).reshape(-1))]))
    assert np.array_equal(ri[:len(pairs)], pairs[:, 2])
