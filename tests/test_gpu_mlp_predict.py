"""The fused prediction kernels at the edges of their tiles: one row, a ragged
last tile, input widths below, at and above a multiple of 64 up to the widest
that stays in shared memory, one beyond it (the training pass's kernels), more
rows than one round holds, and rows that are not 16-byte aligned.  Bar: 1 %
relative L2 against the FP64 network on the BF16 weights (BF16 activations carry
2^-9 relative rounding per element), and equal results for the same rows wherever
they lie."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def bf16(x):
    u = np.ascontiguousarray(x, np.float32).view(np.uint32)
    return ((u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000).astype(np.uint32).view(np.float32)


def weights64(w, sizes):
    """The parameters the kernels multiply with: matrices in BF16, biases as given."""
    parts = np.split(w, np.cumsum(sizes)[:-1])
    return np.concatenate([bf16(p) if i % 2 == 0 else p for i, p in enumerate(parts)]).astype(np.float64)


@pytest.mark.parametrize("n,d", [(1, 3), (127, 64), (129, 65), (300, 128), (513, 130), (640, 192),
                                 (1000, 255), (700, 256), (400, 300), (131072 + 200, 20)])
def test_predict(n, d):
    import torch
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    rng = np.random.default_rng([n, d])
    X = rng.standard_normal((n, d)).astype(np.float32)
    sizes = [256 * d, 256, 256 * 256, 256, 512, 2]
    w = np.concatenate([rng.standard_normal(s) * a for s, a in zip(
        sizes, (np.sqrt(2.0 / d), 0.1, np.sqrt(2.0 / 256), 0.1, 1 / 16.0, 0.1))]).astype(np.float32)
    with px.MLP(d) as net:
        net.set_params(w)
        host = net.predict(X)
        flat = torch.zeros(n * d + 1, device="cuda")
        for shift in (0, 1):     # 16-byte aligned rows, and rows that are not
            Xd = flat[shift:shift + n * d].view(n, d)
            Xd.copy_(torch.from_numpy(X))
            Y = torch.full((n, 2), np.nan, device="cuda")
            net.predict(Xd, Y)
            assert np.array_equal(Y.cpu().numpy(), host)
    rows = np.unique(np.concatenate([np.arange(min(n, 300)), np.arange(max(0, n - 300), n)]))
    net64 = oracle.MLP.from_flat(weights64(w, sizes), d, 256)
    _, ref, _ = oracle.mlp(net64, bf16(X[rows]))
    assert np.linalg.norm(host[rows] - ref) <= 1e-2 * np.linalg.norm(ref)


@pytest.mark.parametrize("n,d", [(1, 3), (127, 64), (129, 65), (1000, 100), (4096, 50), (8192, 128)])
def test_gradient_sizes(n, d):
    """Loss and gradient where the last block of rows is ragged and where the
    weight gradients' rows are and are not multiples of 16 bytes.  Four stored
    tensors (h1, h2, dz2, dz1) lie between the input and W1's gradient, each
    rounded by at most 2^-9 of an element: 0.8 %, the bar is 1 %."""
    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    rng = np.random.default_rng([n, d, 1])
    X = bf16(0.5 * rng.standard_normal((n, d)))
    T = rng.standard_normal((n, 2)).astype(np.float32)
    with px.MLP(d, seed=2) as net:
        w = bf16(net.get_params())
        net.set_params(w)
        loss, g = net.loss_grad(X, T)
    ref = oracle.MLP.from_flat(w.astype(np.float64), d, 256)
    loss_o, _, g_o = oracle.mlp(ref, X, T, grad=True)
    assert abs(loss - loss_o) <= 1e-2 * loss_o
    go = oracle.MLP.from_flat(g_o, d, 256)
    gg = oracle.MLP.from_flat(g.astype(np.float64), d, 256)
    for name in ("W1", "b1", "W2", "b2", "W3", "b3"):
        a, b = getattr(gg, name), getattr(go, name)
        assert np.linalg.norm(a - b) <= 1e-2 * np.linalg.norm(b), name
