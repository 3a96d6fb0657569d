"""The traversal's kernels at the sizes where one hands over to the next and at
the remainders of their warps, against the oracle's forces (1e-4 relative L2,
the bar of every force comparison), with states whose cells hold one point as
well as crowded ones."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

FORCE_TOL = 1e-4
L = 10


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


def state(n, seed):
    """Half of the points spread over the screen, half in a small patch, a few
    on one position; the corners taken, as a rescaled state has them."""
    rng = np.random.default_rng([seed, n])
    z = rng.integers(0, 1 << 32, (n, 2), dtype=np.uint64)
    m = n // 2
    z[:m] = (1 << 30) + rng.integers(0, 1 << 26, (m, 2), dtype=np.uint64)
    z[m:m + 5] = z[0]
    z[-2], z[-1] = 0, (1 << 32) - 1
    return rng.permutation(z).astype(np.uint32), np.array([50.0, 43.0]) / 2.0 ** 32


def ring_P(n):
    """Each point coupled to its two neighbours by index."""
    i = np.arange(n)
    col = np.sort(np.stack([(i + 1) % n, (i - 1) % n], 1), 1)
    return np.arange(n + 1) * 2, col.reshape(-1), np.full(2 * n, 0.5 / n)


@pytest.mark.parametrize("n,centre,theta", [
    (3, 0, 0.5), (33, 0, 0.5), (33, 1, 1.2), (32767, 0, 0.5), (32768, 0, 0.5), (32801, 0, 1.2),
    (32801, 0, 0.3), (40000, 1, 0.5), (149_999, 1, 0.5), (150_000, 1, 0.5), (150_033, 1, 1.2)])
def test_forces_across_the_kernels(n, centre, theta):
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    z, s = state(n, 5)
    with px.Context(px.Params(log2_r=L, theta=theta, centre_mode=centre)) as ctx:
        ctx.set_P(*ring_P(n))
        ctx.set_state(z, s)
        Frep, Zi, _, Z = ctx.get_forces()
        acc = ctx.counters()[0]
        ctx.step(1)
        ctx.sync()
    rows = np.unique(np.concatenate([np.arange(min(n, 70)), np.arange(max(0, n - 70), n),
                                     np.random.default_rng(1).integers(0, n, 1500)]))
    oF, oZi, _ = oracle.bh_repulsion(z, s, L, theta, rows=rows, centre_mode=centre)
    assert rel(Frep[rows], oF) <= FORCE_TOL
    assert rel(Zi[rows], oZi) <= FORCE_TOL
    assert abs(Z - Zi.astype(np.float64).sum()) <= 1e-6 * Z
    if n <= 40000:
        _, oZ, oacc = oracle.bh_repulsion(z, s, L, theta, centre_mode=centre)
        assert acc == pytest.approx(int(oacc.sum()), rel=1e-4)
        assert rel(Zi, oZ) <= FORCE_TOL


def test_every_cell_opened():
    """theta = 0 opens every occupied cell: the point traversal's ring at its
    fullest, and the same sums from the warp's stack."""
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    z, s = state(6000, 7)
    with px.Context(px.Params(log2_r=L, theta=0.0)) as ctx:
        ctx.set_P(*ring_P(6000))
        ctx.set_state(z, s)
        a = ctx.get_forces()
        ctx.test_stack_limit(48)
        ctx.set_state(z, s)
        b = ctx.get_forces()
    oF, oZi, _ = oracle.bh_repulsion(z, s, L, 0.0)
    for Frep, Zi in ((a[0], a[1]), (b[0], b[1])):
        assert rel(Frep, oF) <= FORCE_TOL and rel(Zi, oZi) <= FORCE_TOL


@pytest.mark.parametrize("n,level,theta", [
    (40, 1, 0.5), (700, 2, 0.5), (900, 3, 1.2), (1500, 4, 0.3), (24575, 6, 0.5), (24576, 6, 0.5),
    (24609, 5, 1.2), (24700, 7, 0.5)])
def test_octree_across_the_kernels(n, level, theta):
    """3-D: counts at every level, the order of the points and the forces on
    both sides of the point traversal's limit and for the smallest octrees."""
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    rng = np.random.default_rng([n, level])
    z = rng.integers(0, 1 << 32, (n, 3), dtype=np.uint64)
    m = n // 2
    z[:m] = (1 << 30) + rng.integers(0, 1 << 27, (m, 3), dtype=np.uint64)
    z[m:m + 4] = z[0]
    z[-2], z[-1] = 0, (1 << 32) - 1
    z, s = z.astype(np.uint32), np.array([40.0, 37.0, 51.0]) / 2.0 ** 32
    rows = np.unique(np.concatenate([np.arange(min(n, 40)), np.arange(max(0, n - 40), n),
                                     rng.integers(0, n, 800)]))
    with px.Context(px.Params(log2_r=level, theta=theta, dim=3)) as ctx:
        ctx.set_P(*ring_P(n))
        for _ in range(2):   # from fresh leaves, and from the cleared ones
            ctx.set_state(z, s)
            Frep, Zi, _, Z = ctx.get_forces()
            cnt_o = oracle.pyramid3(z, level)[0]
            at = 0
            for lv in range(level + 1):
                assert np.array_equal(ctx.get_tree3(lv)[0], cnt_o[at:at + 8 ** lv]), lv
                at += 8 ** lv
            oF, oZi, _ = oracle.bh_repulsion3(z, s, level, theta, rows=rows)
            assert rel(Frep[rows], oF) <= FORCE_TOL
            assert rel(Zi[rows], oZi) <= FORCE_TOL
            assert abs(Z - Zi.astype(np.float64).sum()) <= 1e-6 * Z
            ctx.step(2)
            ctx.sync()


@pytest.mark.parametrize("n,level,k", [(40, 1, 32), (300, 4, 3), (5000, 11, 10), (5000, 3, 32), (20000, 9, 17)])
def test_nbr_precision_on_uneven_states(n, level, k):
    """The 2-D neighbour search over crowded cells, empty stretches and tied
    positions: hit counts equal to the oracle's."""
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    z, s = state(n, 11)
    rng = np.random.default_rng([n, k])
    # half of each row's list true neighbours of the index ring, half random
    hd = np.stack([rng.permutation(n)[:k] for _ in range(50)])[rng.integers(0, 50, n)].astype(np.int32)
    near = np.argsort(z[:, 0].astype(np.float64) * 3 + z[:, 1], kind="stable")
    place = np.empty(n, np.int64)
    place[near] = np.arange(n)
    for a in range(k // 2):
        hd[:, a] = near[(place + a + 1) % n]
    with px.Context(px.Params(log2_r=level)) as ctx:
        ctx.set_P(*ring_P(n))
        ctx.set_state(z, s)
        prec, hits = ctx.nbr_precision(k=k, knn_hd=hd, per_point=True)
    prec_o, hits_o = oracle.nbr_precision(hd, k, z, s, per_row=True)
    assert np.array_equal(hits, hits_o)
    assert prec == pytest.approx(prec_o, abs=1e-15)


@pytest.mark.parametrize("n,level,centre", [
    (2047, 8, 0), (2048, 10, 0), (2049, 7, 1), (2049, 10, 1), (65535, 9, 0), (65536, 8, 0)])
def test_upper_levels_sums_and_rows(n, level, centre):
    """Counts of every level and the forces that read the upper levels'
    records (a wide criterion) on screens whose top is built by each of the
    two ways, Z on both sides of one CTA's share (FP64: 1e-12), and the
    attraction on both sides of a warp's one row and four."""
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    z, s = state(n, 11)
    row, col, val = ring_P(n)
    rows = np.unique(np.concatenate([np.arange(40), np.arange(n - 40, n),
                                     np.random.default_rng(2).integers(0, n, 800)]))
    with px.Context(px.Params(log2_r=level, theta=1.5, centre_mode=centre)) as ctx:
        ctx.set_P(row, col, val)
        for _ in range(2):   # from fresh leaves, and from the cleared ones
            ctx.set_state(z, s)
            Frep, Zi, Fattr, Z = ctx.get_forces()
            cnt_o = oracle.pyramid(z, level)[0]
            for lv in range(level + 1):
                at = oracle.level_offset(lv)
                assert np.array_equal(ctx.get_tree(lv)[0], cnt_o[at:at + 4 ** lv]), lv
            mo = oracle.leaf_keys(z, level)[2]
            assert np.array_equal(ctx.get_tree(0, morton=True)[3], mo)
    oF, oZi, _ = oracle.bh_repulsion(z, s, level, 1.5, rows=rows, centre_mode=centre)
    oA = oracle.attraction(oracle.CSR(row, col.astype(np.int32), val), z, s)
    assert rel(Frep[rows], oF) <= FORCE_TOL
    assert rel(Zi[rows], oZi) <= FORCE_TOL
    assert rel(Fattr, oA) <= FORCE_TOL
    assert abs(Z - Zi.astype(np.float64).sum()) <= 1e-12 * Z


@pytest.mark.parametrize("n,level,k", [(3000, 10, 5), (3000, 12, 5), (9000, 10, 10)])
def test_cells_along_the_curve(n, level, k):
    """The first point of a cell on the screens whose points follow the Hilbert
    curve, for cells of even and odd levels."""
    test_nbr_precision_on_uneven_states(n, level, k)


@pytest.mark.parametrize("n,level", [(599_999, 9), (600_000, 9), (600_001, 10), (600_001, 11)])
def test_forces_on_crowded_screens(n, level):
    """Two points per lane and one on both sides of the rule between them
    (600,000 points, half a point per pixel)."""
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    z, s = state(n, 13)
    rng = np.random.default_rng(3)
    rows = np.unique(np.concatenate([np.arange(70), np.arange(n - 70, n), rng.integers(0, n, 600)]))
    with px.Context(px.Params(log2_r=level)) as ctx:
        ctx.set_P(*ring_P(n))
        ctx.set_state(z, s)
        Frep, Zi, _, Z = ctx.get_forces()
        assert ctx.sync() == 0
    oF, oZi, _ = oracle.bh_repulsion(z, s, level, 0.5, rows=rows)
    assert rel(Frep[rows], oF) <= FORCE_TOL
    assert rel(Zi[rows], oZi) <= FORCE_TOL
    assert abs(Z - Zi.astype(np.float64).sum()) <= 1e-12 * Z
