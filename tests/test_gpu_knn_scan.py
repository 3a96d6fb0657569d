"""The two-pass neighbour search at its edges: the smallest sizes that it takes,
ragged last tiles, row lengths that are no multiple of four, short and long
lists, and rows whose candidates overflow or fall short (those tiles are
scanned again or go to the one-pass search).  The lists are those of a full
FP64 sort outside a 2e-5 band around the k-th distance, d2 within 1e-5 (the bars
of every exact search)."""
import numpy as np
import pytest

import datagen
import oracle

pytestmark = pytest.mark.gpu


def check(X, k, idx, d2):
    n = X.shape[0]
    io, do = oracle.knn(X, k)
    assert (np.sort(idx, 1)[:, 1:] != np.sort(idx, 1)[:, :-1]).all()
    assert not (idx == np.arange(n)[:, None]).any()
    kth = do[:, -1:]
    true = ((X[:, None, :].astype(np.float64) - X[idx].astype(np.float64)) ** 2).sum(2)
    assert (true <= kth * (1 + 2e-5) + 1e-12).all()
    np.testing.assert_allclose(d2, true, rtol=1e-5, atol=1e-9)
    assert (np.diff(d2, axis=1) >= 0).all()
    for i in range(n):
        must = io[i][do[i] < kth[i] * (1 - 2e-5)]
        assert np.isin(must, idx[i]).all(), i


def lists(X, k):
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    with px.Context(px.Params(log2_r=9, k=k, perplexity=max(1.0, k / 3.0))) as ctx:
        try:
            ctx.affinities(X)
        except px.PxsneError as e:   # identical rows have no bandwidth
            assert "bisection" in str(e)
        out = ctx.get_knn()[:2]
        exact, kept, path = ctx.knn_counters()
        # (lists of over 128 entries outgrow the one-pass search's shared memory
        # and go to the FP32 tiles)
        assert (path == 1 and exact >= kept > 0) or k > 128
    return out


@pytest.mark.parametrize("n,D,k", [
    (223, 3, 5), (227, 50, 5), (800, 8, 90), (1100, 50, 90), (2049, 127, 45), (2500, 17, 150),
    (3001, 64, 33), (5003, 1, 12), (4000, 128, 1)])
def test_lists_at_the_edges(n, D, k):
    X, _ = datagen.gauss10(n % 7, n=n, D=D)
    check(X, k, *lists(X, k))


def test_crowded_and_sparse_rows():
    """1,500 rows on one position (every candidate buffer of theirs overflows),
    300 on two positions, a tight and a wide cluster."""
    rng = np.random.default_rng(3)
    X = rng.standard_normal((4003, 20)).astype(np.float32)
    X[:1500] = X[0]
    X[1500:1650], X[1650:1800] = 9.0, 9.25
    X[1800:2400] = 30.0 + 1e-3 * rng.standard_normal((600, 20))
    X[2400:2500] *= 40.0
    X = X[rng.permutation(X.shape[0])]
    check(X, 30, *lists(X, 30))


def test_one_dimension_far_apart():
    """Neighbourhoods that the stratified sample meets unevenly: points at
    geometric distances, whose thresholds fall short or overshoot."""
    x = np.concatenate([1.02 ** np.arange(1200), -(1.02 ** np.arange(1200))])
    X = np.stack([x, 0.5 * x], 1).astype(np.float32)
    check(X, 20, *lists(X, 20))


def test_more_tiles_than_are_decided_first():
    """Visits beyond the first 16,384 tiles, which the loader decides itself:
    sampled rows against a brute force in FP64."""
    import torch
    rng = np.random.default_rng(12)
    n, k = 16384 * 128 + 3 * 4096 + 77, 3
    X = rng.standard_normal((n, 3)).astype(np.float32)
    idx, d2 = lists(X, k)
    dX = torch.from_numpy(X).cuda().double()
    for i in (0, 77, n // 2, n - 1, *rng.integers(0, n, 40)):
        t = ((dX - dX[i]) ** 2).sum(1)
        t[i] = torch.inf
        want = torch.topk(t, k, largest=False).values.cpu().numpy()
        got = t[torch.from_numpy(idx[i].astype(np.int64)).cuda()].cpu().numpy()
        np.testing.assert_allclose(got, want, rtol=2e-5)
        np.testing.assert_allclose(d2[i], got, rtol=1e-5)


def test_symmetric_rows_of_every_class():
    """P with rows of every length class of the symmetrisation (a warp's 256,
    512 and 1,024 keys, a CTA's shared memory and beyond): shells of points
    around centres that are every shell point's nearest neighbour.  Pattern
    equal to the oracle's, values within the bisection tolerance."""
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    rng = np.random.default_rng(8)
    parts = []
    for g, m in enumerate((240, 280, 500, 530, 1015, 1100, 16500)):
        x = rng.standard_normal((m, 120))
        x *= rng.uniform(9.0, 11.0, (m, 1)) / np.linalg.norm(x, axis=1, keepdims=True)
        x[0] = 0.0
        x[:, g] += 200.0 * (g + 1)
        parts.append(x)
    X = rng.permutation(np.concatenate(parts)).astype(np.float32)
    P, _, _, bad = oracle.affinities(X, 3.0, 5)
    lengths = np.diff(P.row_ptr)
    for lo, hi in ((1, 256), (256, 512), (512, 1024), (1024, 16384), (16384, 1 << 30)):
        assert ((lengths > lo) & (lengths <= hi)).any()
    with px.Context(px.Params(log2_r=9, k=5, perplexity=3.0)) as ctx:
        ctx.affinities(X)
        rp, col, val = ctx.get_P()
    assert np.array_equal(rp, P.row_ptr) and np.array_equal(col, P.col)
    np.testing.assert_allclose(val, P.val, rtol=2e-3, atol=1e-9)
