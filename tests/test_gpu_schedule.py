"""GPU parity of the attention kernels' schedules: many items per CTA with lists
of 0, 1, 2 and more blocks (the forward's stream of key tiles crosses item
boundaries with every parity), lists of very unequal length (the backward's
longest-first order) and a backward workspace without room for that order."""
import ctypes

import numpy as np
import pytest
import torch

from gpu_util import assert_bf16_close, bits, need_gpu, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    need_gpu()


def _lists(bm):
    """CSR of a [H, rows, columns] bitmap on the device."""
    ptr = np.concatenate([[0], np.cumsum(bm.reshape(-1, bm.shape[2]).sum(1, dtype=np.int64))]).astype(np.int32)
    return torch.from_numpy(ptr).cuda(), torch.from_numpy(np.nonzero(bm)[2].astype(np.int32)).cuda()


def _problem(N, H, d, bq, bk, lengths, seed):
    g = np.random.Generator(np.random.PCG64([78, seed]))
    x = [torch.from_numpy(g.standard_normal((N, H, d)).astype(np.float32)).to(torch.bfloat16).cuda() for _ in range(4)]
    nq, nk = -(-N // bq), -(-N // bk)
    bm = np.zeros((H, nq, nk), dtype=np.uint8)
    for h in range(H):
        for i in range(nq):
            n = min(nk, lengths[(h * nq + i) % len(lengths)])
            bm[h, i, g.choice(nk, size=n, replace=False)] = 1
    return x, bm


def _reference(x, bm, bq, bk):
    """O and LSE by the definition, every score in 64 bits."""
    q, k, v = (t.double() for t in x[:3])
    N, H, d = q.shape
    keep = torch.from_numpy(np.repeat(np.repeat(bm, bq, 1), bk, 2)[:, :N, :N]).cuda().bool()
    s = torch.einsum("nhd,mhd->hnm", q, k) * d ** -0.5
    s = s.masked_fill(~keep, -float("inf"))
    lse = torch.logsumexp(s, 2)
    p = torch.nan_to_num(torch.exp(s - lse[:, :, None]))
    return torch.einsum("hnm,mhd->nhd", p, v), lse


LENGTHS = [(1,), (2,), (1, 2, 3), (0, 1, 0, 2, 5), (4, 1, 1, 7)]


@pytest.mark.parametrize("lengths", LENGTHS, ids=lambda x: "-".join(map(str, x)))
@pytest.mark.parametrize("d,bq,bk", [(128, 128, 128), (64, 128, 128), (128, 64, 64), (128, 128, 64), (64, 64, 128)])
def test_forward_short_lists_many_items(d, bq, bk, lengths):
    from paper_2609_23169_gb300 import ultratex as u
    N, H = 1000, 40  # 320 items of 128 rows: two or three per CTA, the last block ragged
    x, bm = _problem(N, H, d, bq, bk, lengths, 1)
    st = u.status_word()
    o, lse = u.ut_bsattn_fwd(*x[:3], *_lists(bm), bq, status=st, block_k=bk)
    ref_o, ref_l = _reference(x, bm, bq, bk)
    assert int(st.item()) == 0
    assert_bf16_close(to_np(o), ref_o.cpu().numpy(), "O")
    got, want = to_np(lse), ref_l.cpu().numpy()
    assert np.array_equal(np.isfinite(got), np.isfinite(want))
    fin = np.isfinite(want)
    assert np.abs(got[fin] - want[fin]).max(initial=0.0) <= 1e-4


@pytest.mark.parametrize("d,bq,bk", [(128, 128, 128), (64, 64, 64)])
def test_backward_order_and_workspace(d, bq, bk):
    """The item order changes nothing but the order in which dQ is summed; a
    workspace without room for it (the size that one version of the library
    asked for) still works."""
    from paper_2609_23169_gb300 import ultratex as u
    N, H = 2100, 7
    x, bm = _problem(N, H, d, bq, bk, (1, 30, 2, 0, 9, 1), 2)
    csr, csc = _lists(bm), _lists(np.ascontiguousarray(bm.transpose(0, 2, 1)))
    st = u.status_word()
    o, lse = u.ut_bsattn_fwd(*x[:3], *csr, bq, status=st, block_k=bk)
    Np = -(-N // 128) * 128
    least = 2 * H * Np * 4 + H * Np * d * 4 + 16
    shape = u.attn_shape(x[0], bq, bk)
    full = u.lib().ut_bsattn_bwd_workspace_size(ctypes.byref(shape))
    assert full >= least + 4 * H * (Np // 128)
    out = []
    for size in (full, least, least + 4 * H * (Np // 128) - 1):
        ws = torch.full((size,), 0xA5, dtype=torch.uint8, device="cuda")
        g = u.ut_bsattn_bwd(x[0], x[1], x[2], o, lse, x[3], *csr, *csc, bq, ws=ws, status=st, block_k=bk)
        torch.cuda.synchronize()
        assert int(st.item()) == 0
        out.append(g)
    for g in out[1:]:
        assert_bf16_close(to_np(g[0]), to_np(out[0][0]), "dQ")
        assert np.array_equal(bits(g[1]), bits(out[0][1])) and np.array_equal(bits(g[2]), bits(out[0][2]))
    q, k, v = (t.double().requires_grad_(True) for t in x[:3])
    keep = torch.from_numpy(np.repeat(np.repeat(bm, bq, 1), bk, 2)[:, :N, :N]).cuda().bool()
    s = (torch.einsum("nhd,mhd->hnm", q, k) * d ** -0.5).masked_fill(~keep, -float("inf"))
    seen = keep.any(2)[:, :, None]
    p = torch.softmax(s.masked_fill(~seen, 0.0), 2) * seen
    torch.einsum("hnm,mhd->nhd", p, v).backward(x[3].double())
    for got, ref, name in zip(out[0], (q.grad, k.grad, v.grad), ("dQ", "dK", "dV")):
        assert_bf16_close(to_np(got), ref.cpu().numpy(), name)


@pytest.mark.parametrize("N,H,d,b", [(1, 1, 64, 32), (33, 2, 128, 32), (130, 1, 64, 128), (200, 3, 128, 64),
                                     (611, 2, 64, 32), (611, 1, 128, 128)])
@pytest.mark.parametrize("aligned", [True, False])
def test_fp32_pieces_and_alignment(N, H, d, b, aligned):
    """fp32 forward and backward at the edges of the 32-row pieces (blocks whose
    last pieces do not exist, lists of odd piece counts, empty lists) and, in
    the backward, tensors aligned to 4 bytes only."""
    from paper_2609_23169_gb300 import ultratex as u
    g = np.random.Generator(np.random.PCG64([79, N]))
    x = [torch.from_numpy(g.standard_normal((N, H, d)).astype(np.float32)).cuda() for _ in range(4)]
    nb = -(-N // b)
    bm = (g.random((H, nb, nb)) < 0.6).astype(np.uint8)
    bm[0, 0] = 0
    if nb > 1:
        bm[0, 1, nb - 1] = 1
    csr, csc = _lists(bm), _lists(np.ascontiguousarray(bm.transpose(0, 2, 1)))
    if csr[1].numel() == 0:
        csr, csc = (csr[0], torch.zeros(1, dtype=torch.int32, device="cuda")), (csc[0], torch.zeros(1, dtype=torch.int32, device="cuda"))
    st = u.status_word()
    o, lse = u.ut_bsattn_fwd(*x[:3], *csr, b, status=st)

    def place(t):
        if aligned:
            return t
        flat = torch.empty(t.numel() + 4, dtype=t.dtype, device="cuda")[1:1 + t.numel()].view(t.shape)
        flat.copy_(t)
        return flat

    grads = [place(torch.zeros_like(x[0])) for _ in range(3)]
    y = [place(t) for t in x]
    u.ut_bsattn_bwd(y[0], y[1], y[2], place(o), lse, y[3], *csr, *csc, b, dq=grads[0], dk=grads[1], dv=grads[2], status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    q, k, v = (t.double().requires_grad_(True) for t in x[:3])
    keep = torch.from_numpy(np.repeat(np.repeat(bm, b, 1), b, 2)[:, :N, :N]).cuda().bool()
    s = (torch.einsum("nhd,mhd->hnm", q, k) * d ** -0.5).masked_fill(~keep, -float("inf"))
    seen = keep.any(2)[:, :, None]
    p = torch.softmax(s.masked_fill(~seen, 0.0), 2) * seen
    ref = torch.einsum("hnm,mhd->nhd", p, v)
    ref.backward(x[3].double())
    # 1e-5 is the stated fp32 tolerance; the sums here have at most 611 terms of order one
    assert np.abs(to_np(o) - ref.detach().cpu().numpy()).max() <= 1e-5
    want = torch.logsumexp(s, 2).detach().cpu().numpy()
    got = to_np(lse)
    assert np.array_equal(np.isneginf(got), np.isneginf(want))
    fin = np.isfinite(want)
    assert np.abs(got[fin] - want[fin]).max(initial=0.0) <= 1e-5
    for gg, rr, name in zip(grads, (q.grad, k.grad, v.grad), ("dQ", "dK", "dV")):
        assert np.abs(to_np(gg) - rr.cpu().numpy()).max() <= 2e-5, name


@pytest.mark.parametrize("N,H,bq,bk,rho", [(100, 2, 128, 128, 1.0), (4000, 3, 128, 64, 0.3), (4160, 2, 32, 32, 0.1),
                                           (5000, 1, 64, 4, 0.02), (9000, 1, 128, 2, 0.01), (129, 5, 64, 128, 0.5),
                                           (5400, 1, 128, 2, 0.02), (50100, 1, 8192, 1, 0.001)])
@pytest.mark.parametrize("ties", [False, True])
def test_topk_lists_and_transpose(N, H, bq, bk, rho, ties):
    """Top-K lists at the edges of the column tiles (N_k of 1, 33, over 1,024 and
    over 4,096, where keys no longer fit registers and fewer rows share a CTA;
    over 49,000, where only the short slice leaves room):
    the scores that the lists imply are the largest, ties go to the smaller
    index, and the transpose holds the same pairs, ascending."""
    from paper_2609_23169_gb300 import ultratex as u
    d = 64
    g = np.random.Generator(np.random.PCG64([80, N]))
    # small integers: pooled means times a power of two and their products are exact in fp32
    q, k = (torch.from_numpy(g.integers(-2, 3, (N, H, d)).astype(np.float32) if not ties else
                             np.repeat(g.integers(-1, 2, (N, H, 1)), d, 2).astype(np.float32)).cuda() for _ in range(2))
    shape = u.AttnShape(N, H, d, bq, u.UT_F32, H * d, bk)
    rp, ci, cp, ri = (t.cpu().numpy() for t in u.ut_block_mask(shape, u.UT_MASK_TOPK, q, k, rho))
    nq, nk = -(-N // bq), -(-N // bk)
    kr = u.ut_topk_count(rho, nk)
    assert np.array_equal(rp, np.arange(H * nq + 1) * kr)
    lists = ci[:H * nq * kr].reshape(H, nq, kr)
    assert (np.diff(lists, axis=2) > 0).all() and lists.min() >= 0 and lists.max() < nk

    def pool(x, b, nb):
        s = np.zeros((H, nb, d))
        for i in range(nb):
            s[:, i] = x[i * b:(i + 1) * b].sum(0, dtype=np.float64) / min(b, N - i * b)
        return s

    xq, xk = q.cpu().numpy().astype(np.float64), k.cpu().numpy().astype(np.float64)
    sc = np.einsum("hid,hjd->hij", pool(xq, bq, nq), pool(xk, bk, nk))
    keep = np.zeros(sc.shape, bool)
    np.put_along_axis(keep, lists, True, 2)
    worst_in = np.where(keep, sc, np.inf).min(2)
    best_out = np.where(keep, -np.inf, sc).max(2)
    eps = 1e-4 * np.abs(sc).max()  # fp32 scores against 64 bits
    assert (worst_in >= best_out - eps).all()
    if not ties:
        order = np.argsort(-sc, axis=2, kind="stable")[:, :, :kr]
        clear = (worst_in - best_out > eps)
        want = np.sort(order, axis=2)
        assert np.array_equal(lists[clear], want[clear])
    pairs = np.argwhere(keep.transpose(0, 2, 1))
    assert np.array_equal(cp, np.concatenate([[0], np.cumsum(keep.sum(1).reshape(-1))]))
    assert np.array_equal(ri[:len(pairs)], pairs[:, 2])
