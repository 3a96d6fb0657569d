"""What calls do where device memory is short, and what they hold afterwards:
the neighbour search without room for its candidate buffers, calls that end
early, and P after a call that could not finish it.

Bars: the search's lists equal (both searches are exact; the data have no ties),
statuses exactly, and at most the 1 GB that a context may keep, with 100 MB for
everything else that a process allocates on the side."""
import numpy as np
import pytest

import datagen

pytestmark = pytest.mark.gpu
E_ARG, E_OOM, E_STATE = -1, -2, -4
KEEP = (1 << 30) + 100_000_000


@pytest.fixture(scope="module")
def px():
    import paper_1611_02568_gb300 as m
    from paper_1611_02568_gb300 import build
    build.build()
    return m


def free_bytes():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_search_without_room_for_candidates(px):
    X, _ = datagen.gauss10(5, n=20_000, D=50)
    with px.Context(px.Params(log2_r=9)) as ctx:
        ctx.affinities(X)
        idx, d2, beta = ctx.get_knn()
        P = ctx.get_P()
        products = ctx.knn_work()[0]
        # the buffers take 51 MB, everything else at most 29
        ctx.test_alloc_limit(40_000_000)
        ctx.affinities(X)
        assert ctx.knn_counters()[2] == 1 and ctx.knn_work()[0] != products
        for a, b in zip((idx, d2, beta, *P), (*ctx.get_knn(), *ctx.get_P())):
            assert np.array_equal(a, b)
        skipped, pairs = ctx.knn_pruning()
        assert 0 < skipped < pairs


def test_a_failed_call_leaves_no_P_and_can_be_repeated(px):
    X, _ = datagen.gauss10(6, n=20_000, D=50)
    Y0 = datagen.init_y0(0, X.shape[0])
    with px.Context(px.Params(log2_r=9)) as ctx:
        ctx.affinities(X)
        want = ctx.get_P()
        for limit, kept in ((1_000_000, True), (4_100_000, False), (20_000_000, False)):
            ctx.test_alloc_limit(limit)
            with pytest.raises(px.PxsneError) as ei:
                ctx.affinities(X)
            assert ei.value.code == E_OOM
            if kept:   # refused before anything was replaced
                for a, b in zip(want, ctx.get_P()):
                    assert np.array_equal(a, b)
            else:
                assert ctx.sizes() == (0, 0)
                with pytest.raises(px.PxsneError) as ei:
                    ctx.init(Y0)
                assert ei.value.code == E_STATE
            ctx.test_alloc_limit(0)
            ctx.affinities(X)
            for a, b in zip(want, ctx.get_P()):
                assert np.array_equal(a, b)
            ctx.init(Y0)
            ctx.step(3)
            assert ctx.sync() == 0
        ctx.test_alloc_limit(1_000_000)
        with pytest.raises(px.PxsneError) as ei:
            ctx.set_P(*want)
        assert ei.value.code == E_OOM and ctx.sizes() == (0, 0)
        ctx.test_alloc_limit(0)
        ctx.set_P(*want)
        ctx.init(Y0)
        assert ctx.sync() == 0


def test_rejected_rows_do_not_stay_on_the_device(px):
    X = np.zeros((2_200_000, 200), np.float32)   # 1.76 GB
    X[-1, -1] = np.nan
    with px.Context(px.Params(log2_r=9)) as ctx:
        before = free_bytes()
        with pytest.raises(px.PxsneError) as ei:
            ctx.affinities(X)
        assert ei.value.code == E_ARG and "non-finite" in str(ei.value)
        assert before - free_bytes() <= KEEP


def test_failed_calls_do_not_add_up(px):
    """The last large request fails (the symmetrisation's 321 MB), with some 170 MB
    of the call's scratch allocated before it."""
    X = np.random.default_rng(1).standard_normal((223_000, 40)).astype(np.float32)
    with px.Context(px.Params(log2_r=9)) as ctx:
        before = free_bytes()
        ctx.test_alloc_limit(310_000_000)
        for _ in range(12):
            with pytest.raises(px.PxsneError) as ei:
                ctx.affinities(X)
            assert ei.value.code == E_OOM
        assert before - free_bytes() <= KEEP
