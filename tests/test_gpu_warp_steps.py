"""The work counters mean the same for either traversal: a warp step is what up to
32 lanes test at once, in total and by level, on both sides of the size where the
kernel changes.  Bars: the bounds of the definition (1 to 32 lanes a step), and
that warps of spread-out points have at least four lanes at work on average."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [700, 5000, 32_767, 32_768, 60_000])
@pytest.mark.parametrize("centre", [0, 1])
def test_lanes_per_step(n, centre):
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    z = np.random.default_rng(n).integers(0, 1 << 32, (n, 2), dtype=np.uint64).astype(np.uint32)
    i = np.arange(n)
    col = np.sort(np.stack([(i + 1) % n, (i - 1) % n], 1), 1).reshape(-1)
    with px.Context(px.Params(log2_r=10, centre_mode=centre)) as ctx:
        ctx.set_P(np.arange(n + 1) * 2, col, np.full(2 * n, 0.5 / n))
        ctx.set_state(z, np.array([60.0, 55.0]) / 2.0 ** 32)
        acc, tested, steps, nodes = ctx.counters()
        lv = ctx.level_counters()
    assert acc <= tested and tested / 32 <= steps <= tested / 4
    assert (lv[:, 0] <= 32 * lv[:, 2]).all() and (lv[:, 2] <= lv[:, 0]).all()
    assert (int(lv[:, 0].sum()), int(lv[:, 1].sum()), int(lv[:, 2].sum())) == (tested, acc, steps)
    assert nodes * 4 >= steps / 32
