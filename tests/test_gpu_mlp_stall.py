"""Prediction whose pipeline stalls: every wait of the two kernels has a limit,
also where the two warps of a row quarter hand over their halves' sums, so the
call returns PXSNE_E_DEVICE and the network predicts the same as before
afterwards.  The stall is an operand that is never requested.  Bars: the status
exactly, the same bits after it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d", [(50, 8), (40_000, 50), (131_072 + 130, 128), (60_000, 200)])
def test_a_stalled_prediction_returns(n, d):
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    X = np.random.default_rng(n).standard_normal((n, d)).astype(np.float32)
    with px.MLP(d, seed=1) as m:
        want = m.predict(X)
        for polls in (1, 64, 2000):
            m.test_stall(polls)
            with pytest.raises(px.PxsneError) as ei:
                m.predict(X)
            assert ei.value.code == -5 and "timed out" in str(ei.value)
            m.test_stall(0)
            assert np.array_equal(m.predict(X), want)
        with pytest.raises(px.PxsneError):
            m.test_stall(65537)
