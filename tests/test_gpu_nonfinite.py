"""GPU: NaN and infinite scores in the forward.  A row that meets a NaN says so in
O and in LSE, whichever tile of its list holds it; other rows do not notice."""
import numpy as np
import pytest
import torch

from gpu_util import bits, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def _lists(bm):
    ptr = np.concatenate([[0], np.cumsum(bm.reshape(-1, bm.shape[2]).sum(1, dtype=np.int64))]).astype(np.int32)
    return torch.from_numpy(ptr).cuda(), torch.from_numpy(np.nonzero(bm)[2].astype(np.int32)).cuda()


@pytest.mark.parametrize("d,bq,bk", [(128, 128, 128), (64, 128, 128), (128, 64, 64), (128, 128, 64), (64, 64, 128)])
def test_a_nan_key_shows_in_every_row_that_lists_it(d, bq, bk):
    from paper_2609_23169_gb300 import ultratex as u
    N, H = 1000, 40
    g = np.random.Generator(np.random.PCG64([82, d + bq + bk]))
    q, k, v = (torch.from_numpy(g.standard_normal((N, H, d)).astype(np.float32)).to(torch.bfloat16).cuda() for _ in range(3))
    nq, nk = -(-N // bq), -(-N // bk)
    bm = (g.random((H, nq, nk)) < 0.5).astype(np.uint8)
    bm[:, :, 1] |= bm[:, :, 0]  # no list ends with its first block
    rp, ci = _lists(bm)
    bad = g.integers(0, nk, H)  # the key block of each head that holds a NaN: early, late, at every parity
    kb = k.clone()
    for h in range(H):
        kb[min(N - 1, bad[h] * bk + 5), h, 3] = float("nan")
    met = torch.from_numpy(np.repeat(bm[np.arange(H), :, bad].astype(bool), bq, 1)[:, :N]).cuda()  # [H, N]
    st = u.status_word()
    o0, l0 = u.ut_bsattn_fwd(q, k, v, rp, ci, bq, status=st, block_k=bk)
    o1, l1 = u.ut_bsattn_fwd(q, kb, v, rp, ci, bq, status=st, block_k=bk)
    assert int(st.item()) == 0
    assert bool(met.any()) and not bool(met.all())
    assert bool(torch.isnan(o1[met.t()]).all())
    # 128-row blocks: NaN; 64-row blocks, where a row may see no key: NaN or -inf
    assert not bool(torch.isfinite(l1[met]).any())
    if bq == bk == 128:
        assert bool(torch.isnan(l1[met]).all())
    assert np.array_equal(bits(l1[~met]), bits(l0[~met]))
    assert np.array_equal(bits(o1[~met.t()]), bits(o0[~met.t()]))
