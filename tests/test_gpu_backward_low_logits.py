"""GPU: backward of strongly negative scores with a ragged last key block.  The
key rows past N are zeros, so their scores are 0 and exp(0 - LSE) overflows where
LSE is below -88.7; they must not reach dQ."""
import numpy as np
import pytest
import torch

from gpu_util import err_stats, need_gpu, to_np

pytestmark = pytest.mark.gpu


# Twice what rounding P, dS and O to bf16 costs here in a 64-bit run of the same
# formulas (dQ 2.8e-2 of its RMS: the mean of K, -4, multiplies the rounding of D;
# dK and dV 3.6e-3; single elements 2.7e-2).
REL_RMS = {"dQ": 6e-2, "dK": 1e-2, "dV": 1e-2}
MAX_ABS = 6e-2


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("bq,bk", [(128, 128), (64, 64), (64, 128), (128, 64)])
@pytest.mark.parametrize("N,d", [(129, 64), (129, 128), (300, 64), (300, 128), (193, 128), (63, 64)])
def test_backward_of_low_logits_is_finite(N, d, bq, bk):
    from paper_2609_23169_gb300 import ultratex as u
    H = 2
    g = torch.Generator(device="cuda").manual_seed(N + d)
    noise = [torch.randn((N, H, d), generator=g, device="cuda") for _ in range(4)]
    q, k = (noise[0] + 4).to(torch.bfloat16), (noise[1] - 4).to(torch.bfloat16)
    v, do = (0.25 * noise[2]).to(torch.bfloat16), (0.25 * noise[3]).to(torch.bfloat16)
    shape = u.attn_shape(q, bq, bk)
    nq, nk = -(-N // bq), -(-N // bk)
    bm = torch.ones((H, nq, nk), dtype=torch.uint8, device="cuda")
    if nk > 1:
        bm[0, 0, 0] = 0  # lists of unequal length: merged tiles with a masked sub-block
    rp, ci, cp, ri = u.ut_block_mask(shape, u.UT_MASK_BITMAP, bitmap=bm)
    st = u.status_word()
    o, lse = u.ut_bsattn_fwd(q, k, v, rp, ci, bq, status=st, block_k=bk)
    got = u.ut_bsattn_bwd(q, k, v, o, lse, do, rp, ci, cp, ri, bq, status=st, block_k=bk)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    assert float(lse.max()) < -88.8
    x = [t.double().requires_grad_(True) for t in (q, k, v)]
    keep = bm.bool().repeat_interleave(bq, 1).repeat_interleave(bk, 2)[:, :N, :N]
    s = (torch.einsum("nhd,mhd->hnm", x[0], x[1]) * d ** -0.5).masked_fill(~keep, -float("inf"))
    torch.einsum("hnm,mhd->nhd", torch.softmax(s, 2), x[2]).backward(do.double())
    for name, a, b in zip(("dQ", "dK", "dV"), got, x):
        assert bool(torch.isfinite(a.float()).all()), name
        e = err_stats(to_np(a), b.grad.cpu().numpy())
        assert e["max_abs"] <= MAX_ABS and e["rel_rms"] <= REL_RMS[name], (name, e)
