"""Two points per lane from 600,000 points and half a point per pixel on, the
pixels being those of the r_1 x r_2 screen: a warp step then covers 64 points, so
that a crowded state's steps test more than 32 pairs each, and at most 32
otherwise."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,L,rx,ry,pairs", [
    (1_040_000, 11, 1920, 1080, True), (1_030_000, 11, 1920, 1080, False),
    (1_100_000, 11, 0, 0, False), (600_000, 11, 1200, 1000, True), (599_999, 11, 1200, 999, False),
    (600_000, 10, 0, 1024, True)])
def test_the_rule_counts_the_screens_own_pixels(n, L, rx, ry, pairs):
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    rng = np.random.default_rng(n)
    # in the screen's middle: neighbours in tree order share their nodes
    z = rng.integers(0, 1 << 24, (n, 2), dtype=np.uint64) + (1 << 29)
    i = np.arange(n)
    col = np.sort(np.stack([(i + 1) % n, (i - 1) % n], 1), 1).reshape(-1)
    with px.Context(px.Params(log2_r=L, screen_x=rx, screen_y=ry)) as ctx:
        ctx.set_P(np.arange(n + 1) * 2, col, np.full(2 * n, 0.5 / n))
        ctx.set_state(z.astype(np.uint32), np.array([50.0, 45.0]) / 2.0 ** 32)
        acc, tested, steps, nodes = ctx.counters()
    assert (tested > 32 * steps) == pairs
