"""The KL's sums over P keep 64 bits: the KL of a P whose one long row has values
over twelve decades equals the sum of the KLs of its even and its odd entries,
whose FP32 terms are the same.  Bar: 2^-42 of the terms' absolute sum (each of
the three sums is off by about 2^-53 of its terms in its three floats and a few
units of FP64; about 2^-38 with two floats)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("decades", [0, 12])
def test_kl_is_additive_in_P(decades):
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    n = 200_000
    rng = np.random.default_rng(decades)
    z = rng.integers(0, 1 << 32, (n, 2), dtype=np.uint64).astype(np.uint32)
    s = np.array([50.0, 40.0]) / 2.0 ** 32
    v = (rng.uniform(0.5, 1.0, n - 1) * 10.0 ** -rng.uniform(0, decades, n - 1)).astype(np.float32)
    v /= np.float32(2.0 ** np.ceil(np.log2(v.sum())))
    col = np.arange(1, n, dtype=np.int32)

    def kl(keep):
        rp = np.full(n + 1, int(keep.sum()), np.int64)
        rp[0] = 0
        with px.Context(px.Params(log2_r=10)) as ctx:
            ctx.set_P(rp, col[keep], v[keep])
            ctx.set_state(z, s)
            return ctx.kl(), ctx.get_forces()[3]

    odd = col % 2 == 1
    (whole, Z), (a, Za), (b, Zb) = kl(np.ones(n - 1, bool)), kl(odd), kl(~odd)
    assert Z == Za == Zb
    p = v.astype(np.float64)
    d = (z[1:].astype(np.float64) - z[0]) * s
    size = np.abs(p * (np.log(p) + np.log1p((d * d).sum(1)))).sum() + p.sum() * np.log(Z)
    assert abs(whole - (a + b)) <= 2.0 ** -42 * size
    want = (p * (np.log(p) + np.log1p((d * d).sum(1)))).sum() + p.sum() * np.log(Z)
    assert abs(whole - want) <= 1e-6 * size
