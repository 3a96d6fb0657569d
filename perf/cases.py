"""The work that users of this library have it do, as timed cases.

A case goes through the public binding (``Context``, ``MLP``, ``pca``) and is
one of:

* ``step``     gradient iterations of a run on the screen (2-D) or the voxel
               grid (3-D), and the frame they end in (``step`` + ``get_Y``)
* ``p``        the affinities P of a data set (``affinities``) and the
               neighbour lists, for small sets P itself as well
* ``eval``     the two quality figures of an embedding (``kl``,
               ``nbr_precision``)
* ``pca``      the reduction to 50 dimensions that comes before P
* ``train``    an epoch of the learned warm start's network
* ``predict``  its start positions for a data set

Inputs are drawn on the GPU from the seed alone.  ``exact`` is the same
mathematics in FP64 tensor operations.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1611_02568_gb300 as px

PERPLEXITY = 30.0
THETA = 0.5
EXACT_ROWS = 100_000   # above this the FP64 neighbour search takes too long
WHOLE_ROWS = 20_000    # up to this P itself is read back, too

_stream = None


def _on_stream():
    """The one stream that a program's work runs on."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream.cuda_stream


def listed():
    return [
        # the 10-Gaussian workload (n = 2000 on 512^2): an interactive run of
        # a small set, where launches and latencies are the cost
        dict(name="step_2k", kind="step", n=2000, D=50, L=9, phase="late", iters=20),
        # the 70,000-point workload (1024^2) from its random start, the dense
        # blob of the exaggerated iterations
        dict(name="step_70k", kind="step", n=70_000, D=50, L=10, phase="start", iters=5),
        # the flagship workload (n = 1M on 2048^2) in the long second phase
        # of the schedule
        dict(name="step_1m", kind="step", n=1_000_000, D=50, L=11, phase="late", iters=20),
        # geometric cell centres on a screen that is neither square nor a
        # power of two, an odd number of points
        dict(name="step_geo_300k", kind="step", n=300_007, D=50, L=11, rx=1920, ry=1080, centre=1,
             phase="late", iters=10),
        # the 3-D embedding on a 256^3 grid
        dict(name="step_3d_200k", kind="step", n=200_000, D=50, L=8, dim=3, phase="late", iters=4),
        # P of the smallest workload, from host memory, read back whole
        dict(name="p_2k", kind="p", n=2000, D=50, host=1),
        # P of the 70,000-point workload after its PCA
        dict(name="p_70k", kind="p", n=70_000, D=50),
        # P of the flagship workload
        dict(name="p_1m", kind="p", n=1_000_000, D=128),
        # the quality of a finished embedding
        dict(name="eval_100k", kind="eval", n=100_003, D=50, L=11, k=10),
        # the 784-dimensional workload's PCA
        dict(name="pca_70k", kind="pca", n=70_000, D=784, dout=50),
        # the warm start's network: one epoch of one training embedding, and
        # the start it predicts for the flagship workload
        dict(name="train_50k", kind="train", n=50_000, D=128, batch=4096),
        dict(name="predict_1m", kind="predict", n=1_000_000, D=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step3", "p", "p", "eval", "pca", "train", "predict"])
    if kind == "step":
        c = dict(kind="step", n=_log_int(rng, 500, 900_000), D=rng.choice([20, 50, 64]),
                 phase=rng.choice(["late", "late", "start"]), centre=rng.choice([0, 0, 1]),
                 iters=5)
        if c["phase"] == "late":
            c["iters"] = rng.randint(5, 20)
        # about as many pixels as points up to sixteen times as many
        c["L"] = min(11, max(7, math.ceil(math.log(c["n"], 4)) + rng.choice([0, 1, 2])))
        if rng.random() < 0.3:
            c["rx"] = rng.randint(2 ** c["L"] // 2, 2 ** c["L"])
            c["ry"] = rng.randint(2 ** c["L"] // 2, 2 ** c["L"])
        return c
    if kind == "step3":
        return dict(kind="step", n=_log_int(rng, 500, 200_000), D=50, L=rng.choice([6, 7, 8]), dim=3,
                    phase=rng.choice(["late", "start"]), iters=rng.randint(2, 4))
    if kind == "p":
        return dict(kind="p", n=_log_int(rng, 500, 900_000), D=rng.randint(8, 128),
                    k=rng.choice([90, 90, 60, 45]), host=rng.choice([0, 0, 1]))
    if kind == "eval":
        return dict(kind="eval", n=_log_int(rng, 2000, 100_000), D=50, L=rng.choice([9, 10, 11]),
                    k=rng.choice([5, 10, 20]))
    if kind == "pca":
        return dict(kind="pca", n=_log_int(rng, 2000, 70_000), D=rng.randint(100, 784), dout=50)
    if kind == "train":
        return dict(kind="train", n=_log_int(rng, 5000, 50_000), D=rng.choice([50, 64, 100, 128]),
                    batch=rng.choice([1024, 2048, 4096, 8192]))
    return dict(kind="predict", n=_log_int(rng, 1000, 900_000), D=rng.choice([50, 64, 100, 128]))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _mixture(n, D, seed):
    """An anisotropic Gaussian mixture with Zipf component sizes (as many
    components as the workloads of that size have), rows shuffled, and each
    row's component."""
    g = _gen(seed)
    comps = 10 if n < 100_000 else 100
    w = 1.0 / torch.arange(1, comps + 1, device="cuda", dtype=torch.float64) ** (0.0 if comps == 10 else 1.1)
    edges = torch.round(torch.cumsum(w / w.sum(), 0) * n).long()
    label = torch.searchsorted(edges, torch.arange(n, device="cuda"), right=True).clamp_(max=comps - 1)
    label = label[torch.randperm(n, generator=g, device="cuda")]
    means = 5.0 * torch.randn(comps, D, generator=g, device="cuda")
    scale = torch.sqrt(0.1 + 1.9 * torch.rand(comps, D, generator=g, device="cuda"))
    turn = torch.linalg.qr(torch.randn(D, D, generator=g, device="cuda", dtype=torch.float64))[0].float()
    X = (torch.randn(n, D, generator=g, device="cuda") * scale[label]) @ turn + means[label]
    return X.contiguous(), label


def _layout(n, dim, label, seed):
    """A layout like those of the schedule's second phase: every component an
    even patch whose area (volume) goes with its size, the patches packed
    around the middle; RMS extents as the runs reach them."""
    g = _gen(seed + 1)
    comps = int(label.max()) + 1
    size = torch.bincount(label, minlength=comps).double()
    order = torch.argsort(size, descending=True)
    before = torch.zeros(comps, device="cuda", dtype=torch.float64)
    before[order] = torch.cumsum(size[order], 0) - 0.5 * size[order]
    place = torch.empty(comps, device="cuda", dtype=torch.float64)
    place[order] = torch.arange(comps, device="cuda", dtype=torch.float64)
    r = (before / n) ** (1.0 / dim)
    a = 2.399963229728653 * place
    if dim == 2:
        mid = torch.stack([r * torch.cos(a), r * torch.sin(a)], 1)
    else:
        h = 1.0 - 2.0 * (place + 0.5) / comps
        q = torch.sqrt(1.0 - h * h)
        mid = torch.stack([r * q * torch.cos(a), r * q * torch.sin(a), r * h], 1)
    p = torch.randn(n, dim, generator=g, device="cuda", dtype=torch.float64)
    p = p / p.norm(dim=1, keepdim=True)
    p = p * torch.rand(n, 1, generator=g, device="cuda", dtype=torch.float64) ** (1.0 / dim)
    y = mid[label] + p * ((size[label] / n) ** (1.0 / dim))[:, None]
    y = y * (1.0 + 0.02 * torch.randn(n, 1, generator=g, device="cuda", dtype=torch.float64))
    rms = 23.0 * min(1.0, math.sqrt(50_000 / n)) + 3.0
    return y * (rms / y.pow(2).mean().sqrt())


def _extent(case):
    """Ulps of each axis: r_d 2^(32 - L), 2^32 on a full screen."""
    L, dim = case["L"], case.get("dim", 2)
    if dim == 3:
        return [2.0 ** 32] * 3
    return [float(case.get(k, 0) or 2 ** L) * 2.0 ** (32 - L) for k in ("rx", "ry")]


def _to_screen(y, R):
    lo, hi = y.min(0).values, y.max(0).values
    R = torch.tensor(R, device="cuda", dtype=torch.float64)
    z = torch.minimum(torch.floor((y - lo) * R / (hi - lo)), R - 1.0)
    return z.long(), (hi - lo) / R


def _start(case, seed):
    """X, and the state (positions in ulps, y-units per ulp, iteration) or
    the random start that the case begins from."""
    n, dim = case["n"], case.get("dim", 2)
    X, label = _mixture(n, case["D"], seed)
    if case.get("phase") == "start":
        return X, (1e-4 * torch.randn(n, dim, generator=_gen(seed + 1), device="cuda")).contiguous(), None, None
    z, s = _to_screen(_layout(n, dim, label, seed), _extent(case))
    return X, None, z, s


def _context(case, seed):
    """A run as a program has it before the next iterations."""
    k = case.get("k_nn", 90)
    ctx = px.Context(px.Params(log2_r=case["L"], theta=case.get("theta", THETA), k=k,
                               perplexity=PERPLEXITY, centre_mode=case.get("centre", 0),
                               screen_x=case.get("rx", 0), screen_y=case.get("ry", 0),
                               dim=case.get("dim", 2)), stream=_on_stream())
    X, Y0, z, s = _start(case, seed)
    ctx.affinities(X)
    if Y0 is not None:
        ctx.init(Y0)
    else:
        ctx.set_state(z.cpu().numpy().astype(np.uint32), s.cpu().numpy(), t=300)
    return ctx


def _images(case, seed):
    """Rows in the range of pixel values with a falling spectrum, on the host
    (what the reduction takes)."""
    n, D = case["n"], case["D"]
    g = _gen(seed)
    m = min(D, 90)
    basis = torch.linalg.qr(torch.randn(D, m, generator=g, device="cuda", dtype=torch.float64))[0].float()
    std = 2.0 * 0.96 ** torch.arange(m, device="cuda", dtype=torch.float32)
    X = 0.3 + (torch.randn(n, m, generator=g, device="cuda") * std) @ basis.T
    X += 0.02 * torch.randn(n, D, generator=g, device="cuda")
    return X.cpu().numpy()


def _weights(D, seed):
    """The network's flat parameters: W1, b1, W2, b2, W3, b3 by rows."""
    g = torch.Generator().manual_seed(seed)
    w = [torch.randn(256, D, generator=g) * math.sqrt(2.0 / D), 0.01 * torch.randn(256, generator=g),
         torch.randn(256, 256, generator=g) * math.sqrt(2.0 / 256), 0.01 * torch.randn(256, generator=g),
         torch.randn(2, 256, generator=g) / 16.0, torch.zeros(2)]
    return torch.cat([t.reshape(-1) for t in w])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        ctx = _context(case, seed)
        return dict(case=case, ctx=ctx, Y=torch.empty(case["n"], ctx.dim, device="cuda"))
    if kind == "eval":
        return dict(case=case, ctx=_context(case | {"phase": "late", "k_nn": 90}, seed))
    if kind == "p":
        X, _ = _mixture(case["n"], case["D"], seed)
        k = case.get("k", 90)
        ctx = px.Context(px.Params(k=k, perplexity=min(PERPLEXITY, k / 3)), stream=_on_stream())
        state = dict(case=case, ctx=ctx, X=X.cpu().numpy() if case.get("host") else X)
        if case["n"] <= WHOLE_ROWS:   # room for the largest union pattern
            state["col"] = np.zeros(2 * k * case["n"], np.int32)
            state["val"] = np.zeros(2 * k * case["n"], np.float32)
        return state
    if kind == "pca":
        return dict(case=case, X=_images(case, seed), seed=seed)
    X, label = _mixture(case["n"], case["D"], seed)
    X = (0.1 * X).contiguous()
    m = px.MLP(case["D"], stream=_on_stream())
    m.set_params(_weights(case["D"], seed).numpy())
    if kind == "train":
        T = _layout(case["n"], 2, label, seed)
        T = (T / T.pow(2).mean().sqrt()).float().contiguous()
        return dict(case=case, mlp=m, X=X, T=T, seed=seed)
    return dict(case=case, mlp=m, X=X, Y=torch.empty(case["n"], 2, device="cuda"))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        ctx = state["ctx"]
        ctx.step(case["iters"])
        ctx.get_Y(Y=state["Y"], blocking=False)
        return state["Y"]
    if kind == "p":
        ctx = state["ctx"]
        ctx.affinities(state["X"])
        idx, d2, beta = ctx.get_knn()
        out = dict(idx=idx, d2=d2, beta=beta, nnz=ctx.sizes()[1])
        if case["n"] <= WHOLE_ROWS:   # a larger P stays on the device in use
            out["row_ptr"], col, val = ctx.get_P()
            out["col"], out["val"] = state["col"], state["val"]
            out["col"][:col.size], out["val"][:val.size] = col, val
        return out
    if kind == "eval":
        kl = state["ctx"].kl()
        precision, hits = state["ctx"].nbr_precision(case["k"], per_point=True)
        return dict(kl=kl, precision=precision, hits=hits)
    if kind == "pca":
        proj, V, lam = px.pca(state["X"], case["dout"], seed=state["seed"])
        return dict(proj=proj, V=V, lam=lam)
    if kind == "train":
        loss = state["mlp"].train(state["X"], state["T"], epochs=1, batch=case["batch"], lr=1e-3,
                                  seed=state["seed"])
        return dict(loss=loss, params=state["mlp"].get_params())
    return state["mlp"].predict(state["X"], state["Y"])


def work(case):
    """One pass's inputs and outputs once, and the method's own operations."""
    kind, n, D = case["kind"], case["n"], case["D"]
    if kind in ("step", "eval"):
        dim = case.get("dim", 2)
        nnz = 1.5 * 90 * n        # the union pattern of the 90 nearest
        # a point meets about 80 cells a level (250 in 3-D): an offset, a
        # distance, the kernel value and the sums; an entry of P about as much
        cells = (80 if dim == 2 else 250) * max(1, case["L"] - 2)
        flops = (8 * dim + 4) * cells * n + (6 * dim + 4) * nnz
        if kind == "eval":        # P and the positions; k nearest of about 9 pixels' points
            return {"bytes": 8 * nnz + 8 * n + 4 * (90 + 1) * n, "flops": 20 * nnz + 100 * n * case["k"]}
        # P, positions, velocities and gains once each way, the frame
        per = 8 * nnz + 2 * 3 * 4 * dim * n
        return {"bytes": case["iters"] * per + 4 * dim * n, "flops": case["iters"] * flops}
    if kind == "p":
        k = case.get("k", 90)
        out = 8 * n * k + 4 * n + (8 * 1.5 * k * n if n <= WHOLE_ROWS else 0)
        return {"bytes": 4 * n * D + out, "flops": 2.0 * n * n * D}   # every pair's dot product
    if kind == "pca":
        return {"bytes": 4 * n * D + 4 * n * case["dout"], "flops": 1.0 * n * D * D + 2.0 * n * D * case["dout"]}
    layer = 2.0 * n * (D * 256 + 256 * 256 + 2 * 256)
    if kind == "train":
        return {"bytes": 4 * n * (D + 2), "flops": 3 * layer}
    return {"bytes": 4 * n * (D + 2), "flops": layer}


# ------------------------------------------------------------------ FP64
def _knn64(X, k):
    n = X.shape[0]
    X = X.double()
    idx = torch.empty(n, k, dtype=torch.long, device="cuda")
    d2 = torch.empty(n, k, dtype=torch.float64, device="cuda")
    rows = max(1, 200_000_000 // n)
    for a in range(0, n, rows):
        b = min(n, a + rows)
        d = torch.cdist(X[a:b], X, compute_mode="donot_use_mm_for_euclid_dist").square_()
        d[torch.arange(b - a, device="cuda"), torch.arange(a, b, device="cuda")] = math.inf
        d2[a:b], idx[a:b] = torch.topk(d, k, dim=1, largest=False, sorted=True)
    return idx, d2


def _conditional64(d2, u):
    """The rows' beta by bisection to the perplexity u, and their weights."""
    n = d2.shape[0]
    d = d2 - d2[:, :1]
    beta = torch.ones(n, dtype=torch.float64, device="cuda")
    lo, hi = torch.zeros_like(beta), torch.full_like(beta, math.inf)
    done = torch.zeros(n, dtype=torch.bool, device="cuda")
    for _ in range(200):
        e = torch.exp(-beta[:, None] * d)
        s = e.sum(1)
        H = torch.log(s) + beta * (d * e).sum(1) / s
        done |= (H - math.log(u)).abs() < 1e-5
        up = (H > math.log(u)) & ~done
        down = ~up & ~done
        lo = torch.where(up, beta, lo)
        hi = torch.where(down, beta, hi)
        new = torch.where(torch.isinf(hi), 2.0 * beta, torch.where(lo > 0, 0.5 * (lo + hi), 0.5 * beta))
        beta = torch.where(done, beta, new)
        if bool(done.all()):
            break
    e = torch.exp(-beta[:, None] * d)
    return beta, e / e.sum(1, keepdim=True)


def _symmetric64(idx, p):
    """Rows, columns and values of (p_{j|i} + p_{i|j}) / 2n, by row and column."""
    n, k = idx.shape
    i = torch.arange(n, device="cuda").repeat_interleave(k)
    j = idx.reshape(-1)
    key, at = torch.unique(torch.cat([i * n + j, j * n + i]), return_inverse=True)
    val = torch.zeros(key.numel(), dtype=torch.float64, device="cuda")
    val.index_add_(0, at, torch.cat([p.reshape(-1)] * 2) / (2.0 * n))
    return key // n, key % n, val


def _repulsion64(z, s, case):
    """Barnes-Hut sums (un-normalised force, Z_i) on the screen's tree."""
    n, dim = z.shape
    L, theta, geo = case["L"], case.get("theta", THETA), case.get("centre", 0)
    F = torch.zeros(n, dim, dtype=torch.float64, device="cuda")
    Z = torch.zeros(n, dtype=torch.float64, device="cuda")
    pts = torch.arange(n, device="cuda")
    cell = torch.zeros(n, dim, dtype=torch.long, device="cuda")
    kids = torch.tensor([[(c >> d) & 1 for d in range(dim)] for c in range(2 ** dim)], device="cuda")
    for l in range(1, L + 1):
        side, sh = 2 ** l, 32 - l
        own = z >> sh
        strides = torch.tensor([side ** d for d in range(dim)], device="cuda")
        keys = (own * strides).sum(1)
        cnt = torch.bincount(keys, minlength=side ** dim)
        com = torch.zeros(side ** dim, dim, dtype=torch.float64, device="cuda")
        if not geo:   # sums of offsets in the cell, exact in FP64
            off = (z - (own << sh)).double()
            com.index_add_(0, keys, off)
        total = (pts.numel() + 7_999_999) // 8_000_000
        nxt = []
        for part in range(total):
            sl = slice(part * 8_000_000, (part + 1) * 8_000_000)
            c = (2 * cell[sl, None, :] + kids).reshape(-1, dim)
            i = pts[sl].repeat_interleave(2 ** dim)
            at = (c * strides).sum(1)
            keep = cnt[at] > 0
            c, i, at = c[keep], i[keep], at[keep]
            N = cnt[at].double()
            base = (c << sh)
            if geo:
                centre = (base.double() + 2.0 ** (sh - 1))
            else:
                centre = base.double() + com[at] / N[:, None]
            dz = z[i].double() - centre
            mine = (own[i] == c).all(1)
            if l == L:
                if not geo:
                    more = mine & (N > 1)
                    dz = torch.where(more[:, None], dz * (N / (N - 1.0).clamp(min=1.0))[:, None], dz)
                N = N - mine.double()
                far = N > 0
            dy = dz * s
            d2 = (dy * dy).sum(1)
            if l < L:
                rc2 = 4.0 ** sh * float((s * s).sum())
                far = (d2 * theta * theta > rc2) & ~mine
                nxt.append((i[~far], c[~far]))
            q = 1.0 / (1.0 + d2[far])
            Nq = N[far] * q
            Z.index_add_(0, i[far], Nq)
            F.index_add_(0, i[far], (Nq * q)[:, None] * dy[far])
        if l < L:
            pts = torch.cat([a for a, _ in nxt])
            cell = torch.cat([b for _, b in nxt])
    return F, Z


def _attraction64(z, s, row, col, val):
    F = torch.zeros(z.shape, dtype=torch.float64, device="cuda")
    dy = (z[row] - z[col]).double() * s
    F.index_add_(0, row, (val / (1.0 + (dy * dy).sum(1)))[:, None] * dy)
    return F


def _steps64(case, seed):
    X, Y0, z, s = _start(case, seed)
    idx, d2 = _knn64(X, 90)
    _, p = _conditional64(d2, PERPLEXITY)
    row, col, val = _symmetric64(idx, p)
    t = 300
    if Y0 is not None:
        z, s = _to_screen(Y0.double(), _extent(case))
        t = 0
    u = torch.zeros(z.shape, dtype=torch.float64, device="cuda")
    gain = torch.ones_like(u)
    R = torch.tensor(_extent(case), device="cuda", dtype=torch.float64)
    for _ in range(case["iters"]):
        Fr, Z = _repulsion64(z, s, case)
        Fa = _attraction64(z, s, row, col, val)
        g = 4.0 * ((12.0 if t < 250 else 1.0) * Fa - Fr / Z.sum())
        gain = torch.where(torch.sign(g) != torch.sign(u), gain + 0.2, gain * 0.8).clamp_(min=0.01)
        u = (0.5 if t < 250 else 0.8) * u - 200.0 * gain * g
        zh = z.double() + torch.round(u / s)
        lo, hi = zh.min(0).values, zh.max(0).values
        gamma = hi - lo + 1.0
        z = torch.minimum(torch.floor((zh - lo) * R / gamma), R - 1.0).long()
        s = s * gamma / R
        t += 1
    y = z.double() * s
    return y - y.mean(0)


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind == "step":
        return _steps64(case, seed) if n <= EXACT_ROWS else None
    if kind == "p":
        if n > EXACT_ROWS:
            return None
        X, _ = _mixture(n, case["D"], seed)
        k = case.get("k", 90)
        idx, d2 = _knn64(X, k)
        beta, p = _conditional64(d2, min(PERPLEXITY, k / 3))
        out = dict(idx=None, d2=d2, beta=beta, nnz=None)
        if n <= WHOLE_ROWS:
            val = _symmetric64(idx, p)[2]
            out |= dict(row_ptr=None, col=None, val=torch.zeros(2 * k * n, dtype=torch.float64, device="cuda"))
            out["val"][:val.numel()] = val
        return out
    if kind == "eval":
        if n > 2 * EXACT_ROWS:
            return None
        X, _, z, s = _start(case | {"phase": "late"}, seed)
        idx, d2 = _knn64(X, 90)
        row, col, val = _symmetric64(idx, _conditional64(d2, PERPLEXITY)[1])
        Z = _repulsion64(z, s, case)[1].sum()
        dy = (z[row] - z[col]).double() * s
        kl = (val * torch.log(val * Z * (1.0 + (dy * dy).sum(1)))).nansum()
        return dict(kl=float(kl), precision=None, hits=None)
    if kind == "pca":
        X = torch.from_numpy(_images(case, seed)).cuda().double()
        Xc = X - X.mean(0)
        lam, V = torch.linalg.eigh(Xc.T @ Xc / (n - 1))
        lam, V = lam.flip(0)[:case["dout"]], V.flip(1)[:, :case["dout"]]
        V = V * torch.sign(V.gather(0, V.abs().argmax(0, keepdim=True)))
        return dict(proj=Xc @ V, V=V, lam=lam)
    if kind == "train":
        return None   # the epoch's order is drawn inside the call
    X, _ = _mixture(n, case["D"], seed)
    h = (0.1 * X).double()
    w = _weights(case["D"], seed).double().cuda()
    out, o, wide = [], 0, case["D"]
    for rows in (256, 256, 2):
        W, b = w[o:o + rows * wide].reshape(rows, wide), w[o + rows * wide:o + rows * wide + rows]
        out.append((W, b))
        o, wide = o + rows * wide + rows, rows
    for q, (W, b) in enumerate(out):
        h = h @ W.T + b
        if q < 2:
            h = torch.nn.functional.gelu(h)
    return h
