"""GPU: block lists in any order, with a ragged last block.  The last block's
missing rows do not count wherever in a list it stands.  (Lists of 64-row blocks
of the listing side are merged and have to ascend.)"""
import numpy as np
import pytest
import torch

from gpu_util import assert_bf16_close, need_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def _shuffled(bm, g):
    """CSR of a [H, rows, columns] bitmap, every list in random order."""
    ptr = np.concatenate([[0], np.cumsum(bm.reshape(-1, bm.shape[2]).sum(1, dtype=np.int64))]).astype(np.int32)
    idx = np.concatenate([g.permutation(np.nonzero(row)[0]) for row in bm.reshape(-1, bm.shape[2])]).astype(np.int32)
    return torch.from_numpy(ptr).cuda(), torch.from_numpy(idx).cuda()


@pytest.mark.parametrize("d,bq,bk,H,density", [(128, 128, 128, 2, 1.0), (64, 128, 128, 2, 1.0), (128, 128, 128, 40, 0.5),
                                               (64, 128, 128, 40, 0.5), (128, 128, 64, 3, 0.7), (64, 128, 64, 3, 0.7)])
def test_forward_takes_lists_in_any_order(d, bq, bk, H, density):
    from paper_2609_23169_gb300 import ultratex as u
    N = 1000  # 104 rows in the last block of 128, 40 in the last of 64
    g = np.random.Generator(np.random.PCG64([83, d + bk + H]))
    q, k, v = (torch.from_numpy(g.standard_normal((N, H, d)).astype(np.float32)).to(torch.bfloat16).cuda() for _ in range(3))
    nq, nk = -(-N // bq), -(-N // bk)
    bm = (g.random((H, nq, nk)) < density).astype(np.uint8)
    bm[:, :, nk - 1] = 1
    rp, ci = _shuffled(bm, g)
    st = u.status_word()
    o, lse = u.ut_bsattn_fwd(q, k, v, rp, ci, bq, status=st, block_k=bk)
    assert int(st.item()) == 0
    keep = torch.from_numpy(np.repeat(np.repeat(bm, bq, 1), bk, 2)[:, :N, :N]).cuda().bool()
    s = (torch.einsum("nhd,mhd->hnm", q.double(), k.double()) * d ** -0.5).masked_fill(~keep, -float("inf"))
    assert_bf16_close(to_np(o), torch.einsum("hnm,mhd->nhd", torch.softmax(s, 2), v.double()).cpu().numpy(), "O")
    assert np.abs(to_np(lse) - torch.logsumexp(s, 2).cpu().numpy()).max() <= 1e-4


@pytest.mark.parametrize("d,bq,bk", [(128, 128, 128), (64, 128, 128), (128, 64, 128)])
def test_backward_takes_transposed_lists_in_any_order(d, bq, bk):
    from paper_2609_23169_gb300 import ultratex as u
    N, H = 1000, 2
    g = np.random.Generator(np.random.PCG64([84, d + bq]))
    q, k, v, do = (torch.from_numpy(g.standard_normal((N, H, d)).astype(np.float32)).to(torch.bfloat16).cuda()
                   for _ in range(4))
    nq, nk = -(-N // bq), -(-N // bk)
    bm = (g.random((H, nq, nk)) < 0.7).astype(np.uint8)
    bm[:, nq - 1, :] = 1
    bm[:, :, nk - 1] = 1
    rows = _shuffled(bm, g) if bq == 128 else tuple(
        t.cuda() for t in (torch.from_numpy(np.concatenate([[0], np.cumsum(bm.reshape(-1, nk).sum(1))]).astype(np.int32)),
                           torch.from_numpy(np.nonzero(bm)[2].astype(np.int32))))
    cols = _shuffled(np.ascontiguousarray(bm.transpose(0, 2, 1)), g)
    st = u.status_word()
    o, lse = u.ut_bsattn_fwd(q, k, v, *rows, bq, status=st, block_k=bk)
    got = u.ut_bsattn_bwd(q, k, v, o, lse, do, *rows, *cols, bq, status=st, block_k=bk)
    assert int(st.item()) == 0
    x = [t.double().requires_grad_(True) for t in (q, k, v)]
    keep = torch.from_numpy(np.repeat(np.repeat(bm, bq, 1), bk, 2)[:, :N, :N]).cuda().bool()
    s = (torch.einsum("nhd,mhd->hnm", x[0], x[1]) * d ** -0.5).masked_fill(~keep, -float("inf"))
    torch.einsum("hnm,mhd->nhd", torch.softmax(s, 2), x[2]).backward(do.double())
    for name, a, b in zip(("dQ", "dK", "dV"), got, x):
        assert_bf16_close(to_np(a), b.grad.cpu().numpy(), name)
