"""The neighbour search on rows with many equal distances: whole numbers, one-hot
rows, rows far from the origin (whose rounding hides their distances) and equal
rows.  Distances of whole numbers are exact in FP32, so the lists must be the k
smallest pairs (distance, index) exactly; of the others the distances within 1e-5
of FP64's.

A narrowed threshold is short for a row with a chance of 1e-4 (3.75 deviations), so
that at most a tenth of the tiles may be left to the one-pass search where the
thresholds can be narrowed at all; where they cannot, all are, without a second
scan."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def rows(kind, n):
    import torch
    g = torch.Generator(device="cuda").manual_seed(1)
    if kind == "grid":
        return torch.randint(0, 4, (n, 8), generator=g, device="cuda").float()
    if kind == "one-hot":
        c = torch.randint(0, 5, (n, 10), generator=g, device="cuda")
        return torch.nn.functional.one_hot(c, 5).float().reshape(n, 50).contiguous()
    x = torch.randn(n, 20, generator=g, device="cuda")
    if kind == "offset":
        return x + 3000.0
    if kind == "equal":
        return x[:n // 1000].round().repeat_interleave(1000, 0)[:n].contiguous()
    raise ValueError(kind)


@pytest.mark.parametrize("kind,n,k", [("grid", 200_000, 90), ("grid", 20_003, 30), ("one-hot", 200_000, 90),
                                      ("one-hot", 30_011, 45), ("offset", 30_011, 90),
                                      ("equal", 30_000, 90), ("equal", 30_000, 5)])
def test_lists_and_passes(kind, n, k):
    import torch

    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    X = rows(kind, n)
    with px.Context(px.Params(log2_r=9, k=k, perplexity=k / 3.0)) as ctx:
        try:
            ctx.affinities(X)
        except px.PxsneError as e:   # equal distances have no bandwidth
            assert "bisection" in str(e)
        idx, d2, _ = ctx.get_knn()
        skipped, pairs = ctx.knn_pruning()
        products, again, left = ctx.knn_work()
    T = (n + 127) // 128
    X64 = X.double()
    for i in np.random.default_rng(0).integers(0, n, 150):
        d = ((X64 - X64[i]) ** 2).sum(1)
        d[i] = torch.inf
        got = d[torch.from_numpy(idx[i].astype(np.int64)).cuda()].cpu().numpy()
        if kind == "offset":
            want = torch.topk(d, k, largest=False).values.cpu().numpy()
            np.testing.assert_allclose(got, want, rtol=2e-5)
            np.testing.assert_allclose(d2[i], got, rtol=1e-5)
        else:
            order = torch.sort(d, stable=True).indices[:k].cpu().numpy()
            assert np.array_equal(idx[i], order), i
            assert np.array_equal(d2[i].astype(np.float64), got), i
    assert skipped <= pairs and pairs == T * T
    if kind == "grid" and n == 200_000:
        assert again > 0 and left <= T // 10
    if kind in ("offset", "equal") and k == 90:
        assert left == T and again <= T // 10
