"""GPU: waits that run out in the middle of the forward's stream of tiles (the
limit is short enough for some waits and long enough for others) leave no load,
copy or product behind: the call reports UT_ERR_TIMEOUT or finishes, and the next
normal call gives the bits that a call before gave."""
import numpy as np
import pytest
import torch

from gpu_util import bits, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("d,bq,bk", [(128, 128, 128), (64, 128, 128), (128, 64, 64)])
def test_forward_after_expired_waits(monkeypatch, d, bq, bk):
    from paper_2609_23169_gb300 import ultratex as u
    N, H = 2500, 16  # 320 items: two or three per CTA
    g = torch.Generator(device="cuda").manual_seed(5)
    q, k, v = (torch.randn((N, H, d), generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    nq, nk = -(-N // bq), -(-N // bk)
    bm = (torch.rand((H, nq, nk), generator=g, device="cuda") < 0.4).to(torch.uint8)
    shape = u.attn_shape(q, bq, bk)
    rp, ci, _, _ = u.ut_block_mask(shape, u.UT_MASK_BITMAP, bitmap=bm, with_transpose=False)

    def call():
        st = u.status_word()
        out = u.ut_bsattn_fwd(q, k, v, rp, ci, bq, status=st, block_k=bk)
        torch.cuda.synchronize()
        return int(st.item()), out

    code, before = call()
    assert code == u.UT_OK
    for limit in ("0", "300", "3000"):
        monkeypatch.setenv("UT_WAIT_TIMEOUT_NS", limit)
        code, _ = call()
        assert code == u.UT_ERR_TIMEOUT or (limit != "0" and code == u.UT_OK)
        monkeypatch.delenv("UT_WAIT_TIMEOUT_NS")
        code, after = call()
        assert code == u.UT_OK
        for x, y in zip(before, after):
            assert np.array_equal(bits(x), bits(y))
