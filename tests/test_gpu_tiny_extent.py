"""Starts so small that squared distances underflow in FP32: every kernel value
is 1, so every point's Z_i is n - 1 less nothing, whatever the tree does, Z is n
(n - 1) and the KL finite; and starts so large that d^2 does, where theta = 0 is
the sum over all pairs still.  Bars: Z_i to 1e-6 (sums of n - 1 ones, exact, with
one rounding of each cell's kernel value), forces to the 1e-4 of every force
comparison against FP64 sums over all pairs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def context(n, dim, L, **kw):
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    i = np.arange(n)
    col = np.sort(np.stack([(i + 1) % n, (i - 1) % n], 1), 1).reshape(-1)
    ctx = px.Context(px.Params(log2_r=L, dim=dim, **kw))
    ctx.set_P(np.arange(n + 1) * 2, col, np.full(2 * n, 0.5 / n))
    return ctx


def start(n, dim, seed=1):
    return np.random.default_rng(seed).standard_normal((n, dim))


SETS = [(500, 2, 9, 0, 0.5), (500, 2, 9, 0, 1.2), (500, 2, 9, 1, 0.5), (40_000, 2, 9, 0, 0.5),
        (40_000, 2, 9, 0, 1.2), (5, 2, 1, 0, 0.5), (500, 3, 6, 0, 0.5), (30_000, 3, 6, 0, 0.5),
        (30_000, 3, 6, 0, 1.2), (7, 3, 1, 0, 0.5)]


@pytest.mark.parametrize("n,dim,L,centre,theta,extent", [
    *((*s, e) for s in SETS for e in (1e-18, 1e-20, 1e-23)), (600_001, 2, 9, 0, 0.5, 1e-23)])
def test_every_pair_counts(n, dim, L, centre, theta, extent):
    with context(n, dim, L, centre_mode=centre, theta=theta) as ctx:
        ctx.init((extent * start(n, dim)).astype(np.float32))
        _, Zi, _, Z = ctx.get_forces()
        assert np.abs(Zi - (n - 1)).max() <= 1e-6 * n
        assert abs(Z - n * (n - 1.0)) <= 1e-6 * n * (n - 1.0)
        assert np.isfinite(ctx.kl())


@pytest.mark.parametrize("dim,L", [(2, 9), (3, 6)])
def test_one_axis_underflows(dim, L):
    """The first axis ordinary, the others 1e-25: exact pair sums with theta 0."""
    n = 400
    Y = start(n, dim)
    Y[:, 1:] *= 1e-25
    with context(n, dim, L, theta=0.0) as ctx:
        ctx.init(Y.astype(np.float32))
        z, s, _, _, _ = ctx.get_state()
        Frep, Zi, _, _ = ctx.get_forces()
    y = z.astype(np.float64) * s
    d = y[:, None] - y[None]
    q = 1.0 / (1.0 + (d * d).sum(2))
    np.fill_diagonal(q, 0.0)
    assert np.linalg.norm(Zi - q.sum(1)) <= 1e-4 * np.linalg.norm(q.sum(1))
    F = ((q * q)[:, :, None] * d).sum(1)
    assert np.linalg.norm(Frep - F) <= 1e-4 * np.linalg.norm(F)


@pytest.mark.parametrize("n,centre", [(300, 0), (300, 1), (33_000, 0)])
def test_theta_zero_on_a_large_extent(n, centre):
    """Extents beyond 1e15, where d^2 passes 1e30: no cell is accepted above the
    pixels with theta = 0, so the sums are the pixels' own."""
    Y = 3e15 * start(n, 2)
    with context(n, 2, 9, theta=0.0, centre_mode=centre) as ctx:
        ctx.init(Y.astype(np.float32))
        lv = ctx.level_counters()
        _, Zi, _, _ = ctx.get_forces()
    # above the pixels only cells of one point may be taken (centres of mass), so
    # every point takes n - 1 points, or fewer terms where pixels hold several
    assert lv[:, 1].sum() <= n * (n - 1)
    if centre == 1:
        assert lv[1:9, 1].sum() == 0
    assert np.isfinite(Zi).all() and (Zi >= 0).all()
