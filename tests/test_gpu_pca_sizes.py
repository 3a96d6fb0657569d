"""PCA at the edges of its tiles and of the device iteration: more components
than tile columns, dimensions below and above one tile, all components (one
iteration), fewer rows than the block has columns and constant dimensions (the
block is rank-deficient there and goes to the host iteration).  Bars: the
covariance is summed in FP32 over slices of 4,096 rows, a relative error of
about sqrt(4096) 2^-24 = 4e-6 of its largest entries; the eigenvalues get 1e-4
of the largest and the reconstruction of the covariance restricted to the
components the same."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,D,dout", [
    (500, 5, 5), (1000, 64, 50), (777, 129, 1), (4097, 200, 70), (3000, 130, 96), (9000, 260, 100),
    (40, 300, 30)])
def test_pca_sizes(n, D, dout):
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    rng = np.random.default_rng([n, D])
    m = min(n, D)
    X = rng.standard_normal((n, m)) * 0.93 ** np.arange(m) @ np.linalg.qr(rng.standard_normal((D, D)))[0][:m]
    X = (X + rng.standard_normal(D)).astype(np.float32)
    if D > 100:
        X[:, 7] = 0.5
    Z, V, lam = px.pca(X, dout, seed=3)
    Xc = X.astype(np.float64) - X.astype(np.float64).mean(0)
    C = Xc.T @ Xc / (n - 1)
    w, U = np.linalg.eigh(C)
    w = w[::-1][:dout]
    assert np.abs(lam - w).max() <= 1e-4 * w[0]
    V = V.astype(np.float64)
    full = w > 1e-6 * w[0]
    assert np.abs((V.T @ V - np.eye(dout))[np.ix_(full, full)]).max() <= 1e-4
    assert np.abs(V.T @ C @ V - np.diag(lam))[np.ix_(full, full)].max() <= 1e-4 * w[0]
    assert np.linalg.norm(Z - Xc @ V) <= 1e-5 * np.linalg.norm(Xc)
    big = np.abs(V).argmax(0)
    assert (V[big, np.arange(dout)][full] > 0).all()
