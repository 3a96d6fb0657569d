"""What the neighbour search says about its own work: the skipped share of the
tile pairs, the products formed, and the query tiles that the two-pass search
scanned again or left to the one-pass search.

Bars: counts, exactly.  A row's threshold comes out short with a chance of at most
2e-4 (5e-5 on the bench's mixtures), so that of these 60,000 rows some send their
tile to the second scan; a row with more identical partners than its buffer or the
sort hold must leave its tile."""
import numpy as np
import pytest

import datagen

pytestmark = pytest.mark.gpu


def search(X, k):
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    with px.Context(px.Params(log2_r=9, k=k, perplexity=k / 3.0)) as ctx:
        try:
            ctx.affinities(X)
        except px.PxsneError as e:   # identical rows have no bandwidth
            assert "bisection" in str(e)
        return (*ctx.knn_pruning(), *ctx.knn_work())


def test_a_mixture_is_done_in_two_passes():
    X, _ = datagen.gauss10(3, n=60_000, D=50)
    skipped, pairs, products, again, left = search(X, 90)
    T = (60_000 + 127) // 128
    assert pairs == T * T
    # every pair that is not skipped is a product; the sample adds at most an
    # eighth of all pairs and a tile
    assert pairs - skipped <= products
    assert 0 < again <= T // 4 and left <= T // 50
    assert products <= (pairs - skipped) * (1 + (again + left) / T * 4) + pairs / 8 + 2 * T


def test_tiles_left_over_are_counted_once():
    """Every row equal to 499 others: no tile can be finished in two passes."""
    rng = np.random.default_rng(0)
    X = np.repeat(rng.standard_normal((200, 20)).astype(np.float32) * 30, 500, axis=0)
    skipped, pairs, products, again, left = search(X, 30)
    T = (X.shape[0] + 127) // 128
    assert pairs == T * T and left == T
    assert skipped <= pairs and pairs - skipped <= products
    assert again <= T
