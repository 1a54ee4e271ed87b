"""The workloads this framework is timed on, each through its public entry points.

A multi-view canvas is 13 images of side x side latent tokens: six noisy
targets, six conditions that share the targets' silhouettes, one reference
(side 32 / 64 / 128 for 512 / 1024 / 2048 pixels).  A share `fg` of every
image's tokens is foreground.  Kinds of a case:

  infer    block-sparse attention forward on compacted tokens: what every layer
           of a denoising step calls
  train    the forward, then the gradient of Q, K and V: one layer of a
           training step
  step     the whole path over one canvas (HotPath.step): compaction, block
           lists, attention forward and backward, scatter
  lists    the block lists of one layer, Top-K over pooled scores, with the
           transpose that the backward walks
  move     compaction of Q, K, V, dO and the scatter of O and the gradients
  rope     the rotated gather of Q, K and the inverse-rotated scatter of their
           gradients, behind a text prefix
  sampler  around the model call of a denoising step: canvas mask from the
           renders' alpha, Euler update fused with the next gather, composite
           latent for decoding

Activations are N(0, 1), alpha renders are soft-edged blobs with faint specks,
silhouettes are sums of Gaussians.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2609_23169_gb300 import ultratex as ut
from paper_2609_23169_gb300.path import HotPath

IMAGES, VIEWS = 13, 6
LATENT = 64        # values of a latent token: 16 VAE channels, 2 x 2 patches
FACTOR = 16        # pixels per token side
DT = -1.0 / 28.0   # one step of a 28-step schedule
EXACT_FLOPS = 1.2e13  # 64-bit products that take some ten seconds on this card


def _attention(name, kind, side, fg, **more):
    case = {"name": name, "kind": kind, "side": side, "fg": fg, "heads": 24, "d": 128, "dtype": "bf16",
            "bq": 128, "bk": 128, "lists": "topk", "rho": 0.12, "ref_full": False}
    case.update(more)
    return case


def listed():
    return [
        # the fp32 configuration: the smallest call of the whole path, host latency and launches
        _attention("step_tiny_f32", "step", 5, 0.6, heads=1, d=64, dtype="f32", bq=32, bk=32, lists="structured"),
        # fp32 training of a small canvas, ragged in every block size
        _attention("train_f32", "train", 16, 0.6, heads=2, d=64, dtype="f32", bq=32, bk=32, lists="structured"),
        # one layer of a denoising step at 512, the reference image kept in full: few items for 152 SMs
        _attention("infer_512", "infer", 32, 0.55, lists="structured", ref_full=True),
        # one layer of a denoising step at 2048 with the paper's Top-K rule
        _attention("infer_2048", "infer", 128, 0.40),
        # one layer of a training step at 1024 with structured lists of unequal lengths
        _attention("train_1024", "train", 64, 0.45, lists="structured"),
        # 64-row blocks on both sides, a thin foreground, sparse lists
        _attention("train_2048_b64", "train", 128, 0.20, bq=64, bk=64, rho=0.10),
        # the smaller head dimension on a small canvas with dense lists
        _attention("train_512_d64", "train", 32, 0.40, d=64, rho=0.5),
        # the whole training path at 2048: the largest call
        _attention("step_2048", "step", 128, 0.40),
        # block lists of one layer at 2048
        _attention("lists_2048", "lists", 128, 0.40),
        # token movement of one layer at 1024
        _attention("move_1024", "move", 64, 0.45),
        # rotated movement of one layer at 2048 behind 512 text tokens
        {"name": "rope_2048", "kind": "rope", "side": 128, "fg": 0.40, "heads": 24, "d": 128, "dtype": "bf16",
         "prefix": 512},
        # the sampler's own work of one denoising step at 2048: small launches
        {"name": "sampler_2048", "kind": "sampler", "side": 128, "fg": 0.40, "dtype": "bf16"},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["infer", "infer", "train", "train", "train", "train_f32", "step", "lists", "move", "rope",
                       "sampler"])
    fg = round(rng.uniform(0.20, 0.80), 4)
    if kind == "train_f32":
        b = rng.choice([32, 64, 128])
        return {"kind": "train", "side": int(_log(rng, 5, 17)), "fg": fg, "heads": rng.randint(1, 4),
                "d": rng.choice([64, 128]), "dtype": "f32", "bq": b, "bk": b, "lists": "structured", "rho": 0.0,
                "ref_full": rng.random() < 0.3}
    side = int(round(_log(rng, 16, 128)))
    if kind == "sampler":
        return {"kind": kind, "side": side, "fg": fg, "dtype": rng.choice(["bf16", "f32"])}
    case = {"kind": kind, "side": side, "fg": fg, "heads": rng.randint(3, 24), "d": rng.choice([64, 128, 128]),
            "dtype": "bf16"}
    if kind == "rope":
        return dict(case, prefix=rng.choice([0, 512, rng.randint(1, 600)]))
    bq, bk = (128, 128) if kind == "step" else rng.choice([(128, 128)] * 5 + [(64, 64), (64, 128), (128, 64)])
    case.update(bq=bq, bk=bk, lists="topk" if kind in ("step", "lists") else rng.choice(["topk", "topk", "structured"]),
                rho=round(_log(rng, 0.05, 1.0), 4), ref_full=rng.random() < 0.3)
    while work(case)["flops"] * (2 if bq == 64 or bk == 64 else 1) > 2.5e13:
        case["side"] = int(case["side"] * 0.8)
    return case


# ----------------------------------------------------------------- sizes
def _counts(case):
    """Foreground tokens of each image."""
    per = case["side"] ** 2
    n = np.full(IMAGES, max(1, int(math.floor(case["fg"] * per + 0.5))), dtype=np.int64)
    if case.get("ref_full"):
        n[-1] = per
    return n


def _tokens(case):
    return int(_counts(case).sum()) + case.get("prefix", 0)


def _canvas(case):
    return IMAGES * case["side"] ** 2 + case.get("prefix", 0)


def _top(case, nk):
    return min(nk, max(1, int(math.floor(case["rho"] * nk))))


def _structured(case):
    """[N_q, N_k] of 0 / 1: a query block sees the key blocks of its own images, of the same views in the other
    modality, and of the reference."""
    n = _tokens(case)
    ends = np.cumsum(_counts(case))
    see = np.eye(IMAGES, dtype=np.int64)
    see[:, -1] = 1
    for v in range(VIEWS):
        see[v, VIEWS + v] = see[VIEWS + v, v] = 1

    def images(b):
        r0 = np.arange(0, n, b)
        first = np.searchsorted(ends, r0, side="right")
        last = np.searchsorted(ends, np.minimum(r0 + b, n) - 1, side="right")
        i = np.arange(IMAGES)
        return ((i >= first[:, None]) & (i <= last[:, None])).astype(np.int64)

    return (images(case["bq"]) @ see @ images(case["bk"]).T > 0).astype(np.uint8)


def _pairs(case):
    """Row pairs (query, key) of one head that the lists retain (Top-K: blocks of average size)."""
    n, bq, bk = _tokens(case), case["bq"], case["bk"]
    if case["lists"] == "structured":
        rows = np.minimum(bq, n - np.arange(0, n, bq)).astype(np.float64)
        cols = np.minimum(bk, n - np.arange(0, n, bk)).astype(np.float64)
        return float(rows @ _structured(case) @ cols)
    nk = -(-n // bk)
    return float(n) * _top(case, nk) * n / nk


def work(case):
    kind, side = case["kind"], case["side"]
    size = 2 if case["dtype"] == "bf16" else 4
    if kind == "sampler":
        t, n = VIEWS * side ** 2, int(_counts(case)[:VIEWS].sum())
        row = LATENT * size
        # alpha in, canvas mask out; idx, v, z in, z and its gather out; mask in, background rows out
        nbytes = (VIEWS + 1) * (side * FACTOR) ** 2 + IMAGES * side ** 2 + n * (4 + 4 * row) + t + (t - n) * row
        return {"bytes": nbytes, "flops": 2 * n * LATENT}
    t, n, row = _canvas(case), _tokens(case), case["heads"] * case["d"] * size
    if kind == "rope":
        return {"bytes": 2 * (2 * n * row + n * row + t * row) + 8 * n, "flops": 4 * 3 * n * case["heads"] * case["d"]}
    # four tensors gathered; O scattered over the kept canvas, three gradients over zeros
    moved = t + 8 * n + (4 * 2 * n + 2 * n + 3 * (n + t)) * row
    if kind == "move":
        return {"bytes": moved, "flops": 0}
    nq, nk = -(-n // case["bq"]), -(-n // case["bk"])
    if kind == "lists":
        entries = case["heads"] * nq * _top(case, nk)
        return {"bytes": 2 * n * row + 4 * (2 * entries + case["heads"] * (nq + nk)),
                "flops": 2 * case["heads"] * case["d"] * nq * nk + 2 * n * case["heads"] * case["d"]}
    flops = case["heads"] * _pairs(case) * case["d"] * (4 if kind == "infer" else 14)
    # Q, K, V in, O and LSE out; backward: dO in, dQ, dK, dV out
    nbytes = n * (4 if kind == "infer" else 8) * row + 4 * n * case["heads"]
    return {"bytes": nbytes + (moved if kind == "step" else 0), "flops": flops}


# ---------------------------------------------------------------- inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _field(g, points, side, fg):
    """Sum of 3 to 6 Gaussians over a square of `points` samples a side, in token units."""
    x = (torch.arange(points, device="cuda", dtype=torch.float32) + 0.5) * (side / points)
    n = 3 + int(torch.randint(0, 4, (1,), generator=g, device="cuda"))
    p = torch.rand((n, 4), generator=g, device="cuda")
    f = torch.zeros((points, points), device="cuda")
    for cy, cx, sig, w in p.tolist():
        s = (0.08 + 0.17 * sig) * side
        gy = torch.exp(-((x - (0.2 + 0.6 * cy) * side) ** 2) / (2 * s * s))
        gx = torch.exp(-((x - (0.2 + 0.6 * cx) * side) ** 2) / (2 * s * s))
        f += (0.5 + 0.5 * w) * gy[:, None] * gx[None, :]
    return f


def _mask(case, g):
    """[T] uint8: exactly the counted tokens of every image, where its field is highest; text tokens are kept."""
    side, counts = case["side"], _counts(case)
    m = torch.zeros((IMAGES, side * side), dtype=torch.uint8, device="cuda")
    for i in list(range(VIEWS)) + [IMAGES - 1]:
        order = torch.sort(_field(g, side, side, case["fg"]).reshape(-1), descending=True, stable=True).indices
        m[i, order[:int(counts[i])]] = 1
        if i < VIEWS:
            m[VIEWS + i] = m[i]
    return torch.cat([torch.ones(case.get("prefix", 0), dtype=torch.uint8, device="cuda"), m.reshape(-1)])


def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _normal(case, g, *shape):
    out = torch.empty(shape, dtype=_dtype(case), device="cuda")
    rows = max(1, (1 << 27) // max(1, out[0].numel()))
    for r in range(0, shape[0], rows):
        part = out[r:r + rows]
        part.copy_(torch.randn(part.shape, generator=g, device="cuda"))
    return out


def _activations(case, seed, rows, count):
    g = _generator(seed)
    return [_normal(case, g, rows, case["heads"], case["d"]) for _ in range(count)]


def _blocks(x, b):
    """[H, blocks, d] 64-bit means over the rows of each block."""
    n, h, d = x.shape
    nb = -(-n // b)
    out = torch.empty((h, nb, d), dtype=torch.float64, device=x.device)
    for i in range(h):
        s = torch.zeros((nb * b, d), dtype=torch.float64, device=x.device)
        s[:n] = x[:, i]
        out[i] = s.view(nb, b, d).sum(1)
    rows = torch.clamp(n - torch.arange(nb, device=x.device) * b, max=b)
    return out / rows[None, :, None]


def _bitmap(case, q, k):
    """[H, N_q, N_k] of 0 / 1, the block mask."""
    if case["lists"] == "structured":
        return torch.from_numpy(_structured(case)).to(q.device)[None].repeat(case["heads"], 1, 1)
    s = _blocks(q, case["bq"]) @ _blocks(k, case["bk"]).transpose(1, 2)
    best = torch.sort(s, dim=2, descending=True, stable=True).indices[:, :, :_top(case, s.shape[2])]
    return torch.zeros(s.shape, dtype=torch.uint8, device=q.device).scatter_(2, best, 1)


def _csr(bitmap):
    """Ascending lists of a [H, rows, columns] bitmap: pointers and columns, rows head-major."""
    ptr = torch.zeros(bitmap.shape[0] * bitmap.shape[1] + 1, dtype=torch.int32, device=bitmap.device)
    ptr[1:] = torch.cumsum(bitmap.reshape(-1, bitmap.shape[2]).sum(1, dtype=torch.int64), 0)
    return ptr, torch.nonzero(bitmap)[:, 2].to(torch.int32).contiguous()


# ------------------------------------------------------ states and passes
def prepare(case, seed):
    kind, dev = case["kind"], torch.device("cuda")
    s = {"kind": kind, "case": case}
    if kind in ("infer", "train"):
        n = _tokens(case)
        x = _activations(case, seed, n, 4 if kind == "train" else 3)
        bm = _bitmap(case, x[0], x[1])
        s.update(x=x, csr=_csr(bm), o=torch.empty_like(x[0]), status=ut.status_word(),
                 lse=torch.empty((case["heads"], n), dtype=torch.float32, device=dev))
        if kind == "train":
            shape = ut.attn_shape(x[0], case["bq"], case["bk"])
            size = ut.lib().ut_bsattn_bwd_workspace_size(ctypes.byref(shape))
            s.update(csc=_csr(bm.transpose(1, 2).contiguous()), grads=[torch.empty_like(x[0]) for _ in range(3)],
                     ws=torch.empty(size, dtype=torch.uint8, device=dev))
        return s
    if kind == "lists":
        n = _tokens(case)
        x = _activations(case, seed, n, 2)
        shape = ut.attn_shape(x[0], case["bq"], case["bk"])
        s.update(x=x, shape=shape)
        return s
    if kind == "sampler":
        g = _generator(seed)
        t, side = VIEWS * case["side"] ** 2, case["side"]
        mask = _mask(case, g)[:t].contiguous()
        idx = torch.nonzero(mask)[:, 0].to(torch.int32).contiguous()
        alpha = torch.empty((VIEWS + 1, side * FACTOR, side * FACTOR), dtype=torch.uint8, device=dev)
        for a in alpha:
            f = _field(g, side * FACTOR, side, case["fg"])
            level = torch.sort(f[::8, ::8].reshape(-1)).values[int((1 - 0.45 * case["fg"]) * f[::8, ::8].numel())]
            a.copy_(torch.clamp((f - level) * 4000.0, 0, 255))
            specks = (torch.rand(f.shape, generator=g, device="cuda") < 2e-4) & (a == 0)
            a[specks] = 7
        s.update(mask=mask, idx=idx, n=idx.numel(), alpha=alpha, z=_normal(case, g, t, LATENT),
                 v=_normal(case, g, idx.numel(), LATENT), tile=_normal(case, g, side * side, LATENT),
                 zc=torch.empty((idx.numel(), LATENT), dtype=_dtype(case), device=dev),
                 canvas=torch.empty(IMAGES * side * side, dtype=torch.uint8, device=dev), status=ut.status_word())
        return s
    t, n = _canvas(case), _tokens(case)
    mask = _mask(case, _generator(seed + (1 << 40)))
    if kind == "rope":
        idx = torch.nonzero(mask)[:, 0].to(torch.int32).contiguous()
        s.update(idx=idx, n=n, src=_activations(case, seed, t, 2), grad=_activations(case, seed + (1 << 41), n, 2),
                 rope=ut.rope_config(case["side"], (16, 56, 56) if case["d"] == 128 else (8, 28, 28),
                                     prefix=case["prefix"]))
        s["rot"] = [torch.empty_like(x) for x in s["grad"]]
        s["out"] = [torch.empty_like(x) for x in s["src"]]
        return s
    x = _activations(case, seed, t, 4)
    if kind == "move":
        o = _activations(case, seed + (1 << 41), n, 4)
        s.update(mask=mask, x=x, o=o, n=n, xc=[torch.empty_like(y) for y in o], canvas=[torch.zeros_like(y) for y in x],
                 idx=torch.empty(n, dtype=torch.int32, device=dev), n_out=torch.empty(1, dtype=torch.int32, device=dev),
                 ws=torch.empty(ut.lib().ut_fg_compact_workspace_size(t) + 16, dtype=torch.uint8, device=dev),
                 status=ut.status_word())
        return s
    mode = ut.UT_MASK_TOPK if case["lists"] == "topk" else ut.UT_MASK_BITMAP
    path = HotPath(t, case["heads"], case["d"], case["bq"], _dtype(case), mode,
                   rho=case["rho"] if case["lists"] == "topk" else 0.0, device=dev)
    bm = _bitmap(case, x[0], x[1]) if mode == ut.UT_MASK_BITMAP else None
    s.update(mask=mask, x=x, path=path, bitmap=bm)
    return s


def run(s):
    kind, case = s["kind"], s["case"]
    if kind in ("infer", "train"):
        q, k, v = s["x"][:3]
        ut.ut_bsattn_fwd(q, k, v, *s["csr"], case["bq"], o=s["o"], lse=s["lse"], status=s["status"],
                         block_k=case["bk"])
        if kind == "infer":
            return {"o": s["o"], "lse": s["lse"]}
        dq, dk, dv = s["grads"]
        ut.ut_bsattn_bwd(q, k, v, s["o"], s["lse"], s["x"][3], *s["csr"], *s["csc"], case["bq"], dq=dq, dk=dk, dv=dv,
                         ws=s["ws"], status=s["status"], block_k=case["bk"])
        return {"o": s["o"], "lse": s["lse"], "dq": dq, "dk": dk, "dv": dv}
    if kind == "lists":
        return list(ut.ut_block_mask(s["shape"], ut.UT_MASK_TOPK, s["x"][0], s["x"][1], rho=case["rho"]))
    if kind == "sampler":
        ut.ut_fg_mask_from_alpha(s["alpha"], FACTOR, out=s["canvas"])
        ut.ut_fg_euler_update_gather(s["idx"], s["n"], s["z"], s["v"], DT, zc=s["zc"], status=s["status"])
        ut.ut_fg_composite(s["mask"], s["z"], s["tile"])
        return {"mask": s["canvas"], "z": s["z"], "zc": s["zc"]}
    if kind == "rope":
        ut.ut_fg_gather_rope(s["idx"], s["n"], s["src"], s["rope"], dsts=s["rot"])
        ut.ut_fg_scatter_rope(s["idx"], s["n"], s["grad"], s["out"], s["rope"], ut.UT_BG_ZERO)
        return {"q": s["rot"][0], "k": s["rot"][1], "dq": s["out"][0], "dk": s["out"][1]}
    if kind == "move":
        ut.ut_fg_compact(s["mask"], s["x"], capacity=s["n"], outs=s["xc"], idx=s["idx"], n_out=s["n_out"], ws=s["ws"],
                         status=s["status"])
        ut.ut_fg_scatter(s["idx"], s["n"], s["o"][:1], s["canvas"][:1], ut.UT_BG_KEEP)
        ut.ut_fg_scatter(s["idx"], s["n"], s["o"][1:], s["canvas"][1:], ut.UT_BG_ZERO)
        return {"idx": s["idx"], "n": s["n_out"], "compacted": s["xc"], "canvas": s["canvas"]}
    p = s["path"]
    n = p.step(s["mask"], *s["x"], bitmap=s["bitmap"])
    return {"idx": p.idx[:n], "o": p.o_canvas, "dq": p.g_canvas[0], "dk": p.g_canvas[1], "dv": p.g_canvas[2]}


# --------------------------------------------------------- 64-bit values
def _exact_attention(case, x, bitmap, backward):
    """Every head and query block by itself: O, LSE and the gradients, in 64 bits."""
    n, heads, d = x[0].shape
    bq, bk, scale = case["bq"], case["bk"], case["d"] ** -0.5
    nk = bitmap.shape[2]
    out = [torch.zeros((n, heads, d), dtype=torch.float64, device=x[0].device) for _ in range(4 if backward else 1)]
    lse = torch.empty((heads, n), dtype=torch.float64, device=x[0].device)
    valid = torch.arange(nk * bk, device=x[0].device).view(nk, bk) < n
    columns = [[np.nonzero(r)[0] for r in h] for h in bitmap.cpu().numpy()]
    for h in range(heads):
        q = x[0][:, h].double()
        k, v = (torch.zeros((nk * bk, d), dtype=torch.float64, device=q.device) for _ in range(2))
        k[:n], v[:n] = x[1][:, h], x[2][:, h]
        k, v = k.view(nk, bk, d), v.view(nk, bk, d)
        do = x[3][:, h].double() if backward else None
        dk, dv = torch.zeros_like(k), torch.zeros_like(v)
        for i, c in enumerate(columns[h]):
            r = slice(i * bq, min(n, i * bq + bq))
            c = torch.from_numpy(c).to(q.device)
            kc, vc = k[c].reshape(-1, d), v[c].reshape(-1, d)
            sc = (q[r] @ kc.T) * scale
            sc.masked_fill_(~valid[c].reshape(1, -1), -math.inf)
            lse[h, r] = torch.logsumexp(sc, 1)
            p = torch.exp(sc - lse[h, r][:, None])
            o = p @ vc
            out[0][r, h] = o
            if backward:
                dv[c] += (p.T @ do[r]).view(-1, bk, d)
                ds = p * (do[r] @ vc.T - (do[r] * o).sum(1, keepdim=True)) * scale
                out[1][r, h] = ds @ kc
                dk[c] += (ds.T @ q[r]).view(-1, bk, d)
        if backward:
            out[2][:, h] = dk.view(-1, d)[:n]
            out[3][:, h] = dv.view(-1, d)[:n]
    return out, lse


def _rotate(case, x, idx, inverse):
    """Pairs (2j, 2j+1) of every head turned by their token's position, in 64 bits."""
    side = case["side"]
    t = idx.long() - case["prefix"]
    text = t < 0
    pos = torch.stack([t // (side * side), (t % (side * side)) // side, t % side]).double()
    pos[:, text] = 0
    angles = []
    for a, dims in enumerate((16, 56, 56) if case["d"] == 128 else (8, 28, 28)):
        freq = 10000.0 ** (-torch.arange(0, dims, 2, dtype=torch.float64, device=x.device) / dims)
        angles.append(pos[a][:, None] * freq)
    ang = torch.cat(angles, 1)[:, None]
    cos, sin = torch.cos(ang), torch.sin(ang) * (-1 if inverse else 1)
    y = x.double()
    return torch.stack([y[..., 0::2] * cos - y[..., 1::2] * sin, y[..., 0::2] * sin + y[..., 1::2] * cos], -1).flatten(2)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("lists", "move"):
        return None  # whole numbers and copies
    if kind in ("infer", "train", "step") and work(case)["flops"] * 12 / 14 > EXACT_FLOPS:
        return None
    s = prepare(case, seed)
    if kind in ("infer", "train"):
        out, lse = _exact_attention(case, s["x"], _bitmap(case, *s["x"][:2]), kind == "train")
        return dict(zip(("o", "dq", "dk", "dv"), out), lse=lse)
    if kind == "sampler":
        z = s["z"].double()
        idx = s["idx"].long()
        # the update rounds once to the latent's type
        zc = z[idx] + float(np.float32(DT)) * s["v"].double()
        z[idx] = zc
        bg = torch.nonzero(s["mask"] == 0)[:, 0]
        z[bg] = s["tile"].double()[bg % case["side"] ** 2]
        return {"mask": None, "z": z, "zc": zc}
    if kind == "rope":
        out = {}
        for name, x in zip(("q", "k"), s["src"]):
            out[name] = _rotate(case, x[s["idx"].long()], s["idx"], False)
        for name, x in zip(("dq", "dk"), s["grad"]):
            out[name] = torch.zeros(s["src"][0].shape, dtype=torch.float64, device=x.device)
            out[name][s["idx"].long()] = _rotate(case, x, s["idx"], True)
        return out
    idx = torch.nonzero(s["mask"])[:, 0]
    x = [y[idx] for y in s["x"]]
    out, _ = _exact_attention(case, x, _bitmap(case, x[0], x[1]), True)
    full = {"idx": None}
    for name, y in zip(("o", "dq", "dk", "dv"), out):
        full[name] = torch.zeros((s["mask"].numel(),) + y.shape[1:], dtype=torch.float64, device=y.device)
        full[name][idx] = y
    return full
