"""Rows so large that squared distances overflow FP32: the tensor-core searches
cannot fill their lists, and the call says so instead of following entries that
name no row (the FP32 search fills them with the lowest indices at infinity, which
have no bandwidth).  The context is usable afterwards.  Bars: the status; the lists of
ordinary rows after it, the same bits as before."""
import numpy as np
import pytest

import datagen

pytestmark = pytest.mark.gpu
E_ARG, E_STATE, E_DEVICE = -1, -4, -5


@pytest.mark.parametrize("D,kw,path", [
    (20, {}, None), (20, {}, "fp32"), (20, dict(knn_probe=8), None),
    (20, dict(knn_probe=8, knn_explore=2), None), (200, {}, None)])
@pytest.mark.parametrize("scale", [1e19, 1e25, 1e35])
def test_overflowing_distances_are_refused(monkeypatch, scale, D, kw, path):
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    if path:
        monkeypatch.setenv("PXSNE_KNN", path)
    X, _ = datagen.gauss10(1, n=3000, D=D)
    Y0 = datagen.init_y0(0, X.shape[0])
    with px.Context(px.Params(log2_r=9, k=30, perplexity=10.0, **kw)) as ctx:
        ctx.affinities(X)
        want = ctx.get_knn()
        with pytest.raises(px.PxsneError) as ei:
            ctx.affinities((X.astype(np.float64) * scale).astype(np.float32))
        if path or D > 128:
            assert ei.value.code == E_DEVICE and "bisection" in str(ei.value)
            idx = ctx.get_knn()[0]
            assert (idx >= 0).all() and (idx < X.shape[0]).all()
        else:
            assert ei.value.code == E_ARG and "overflow" in str(ei.value)
            assert ctx.sizes() == (0, 0)
            with pytest.raises(px.PxsneError) as ei:
                ctx.init(Y0)
            assert ei.value.code == E_STATE
        ctx.affinities(X)
        for a, b in zip(want, ctx.get_knn()):
            assert np.array_equal(a, b)
        ctx.init(Y0)
        ctx.step(3)
        assert ctx.sync() == 0


def test_one_row_far_away_has_no_list():
    """A single row at 1e20: every other row keeps its list, this one has none."""
    import paper_1611_02568_gb300 as px
    X, _ = datagen.gauss10(2, n=3000, D=10)
    X[77] = 1e20
    with px.Context(px.Params(log2_r=9, k=30, perplexity=10.0)) as ctx:
        with pytest.raises(px.PxsneError) as ei:
            ctx.affinities(X)
        assert ei.value.code == E_ARG and "overflow" in str(ei.value)
