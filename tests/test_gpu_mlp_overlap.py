"""Predictions written over their own inputs: every row's output is that of its
input row, wherever in the rows' memory the outputs go and although the rows are
read in rounds.  Bar: the same bits as with an output buffer of its own."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,at", [(2 * 131_072 + 5, 8, "end"), (2 * 131_072 + 5, 8, "middle"),
                                    (2 * 131_072 + 5, 8, "start"), (131_072 + 70, 2, "start"),
                                    (131_072 + 70, 1, "start")])
def test_outputs_over_the_inputs(n, d, at):
    import torch

    import paper_1611_02568_gb300 as px
    from paper_1611_02568_gb300 import build
    build.build()
    g = torch.Generator(device="cuda").manual_seed(1)
    buf = torch.randn(n * max(d, 2), generator=g, device="cuda")
    X = buf[:n * d].view(n, d)
    with px.MLP(d, seed=3) as m:
        want = torch.empty(n, 2, device="cuda")
        m.predict(X, want)
        o = {"end": buf.numel() - 2 * n, "middle": (buf.numel() - 2 * n) // 2, "start": 0}[at]
        Y = buf[o:o + 2 * n].view(n, 2)
        m.predict(X, Y)
    assert torch.equal(Y, want)
