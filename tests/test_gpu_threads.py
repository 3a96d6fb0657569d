"""Contexts on different host threads at the same time, with sizes that ask for
different amounts of shared memory of the same kernels: every call succeeds, with
the outputs that it has alone (the same bits; for PCA, whose column sums are
added in any order, 1e-5 of the largest entry)."""
import threading

import numpy as np
import pytest

import datagen

pytestmark = pytest.mark.gpu


def run_together(jobs, times):
    """Every job `times` times on a thread of its own; what went wrong."""
    wrong = []

    def loop(job, want):
        for _ in range(times):
            try:
                if not job(want):
                    wrong.append("another output")
            except Exception as e:  # noqa: BLE001
                wrong.append(str(e))

    ts = [threading.Thread(target=loop, args=(job, job(None))) for job in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    return wrong


@pytest.fixture(scope="module")
def px():
    import paper_1611_02568_gb300 as m
    from paper_1611_02568_gb300 import build
    build.build()
    return m


def test_neighbour_searches(px):
    def job(n, D, k, probe=0):
        X, _ = datagen.gauss10(k, n=n, D=D)

        def once(want):
            with px.Context(px.Params(log2_r=9, k=k, perplexity=k / 3.0, knn_probe=probe)) as ctx:
                ctx.affinities(X)
                got = ctx.get_knn()
            return got if want is None else all(np.array_equal(a, b) for a, b in zip(got, want))
        return once

    assert run_together([job(3000, 128, 90), job(1500, 8, 5), job(2000, 50, 60),
                         job(2000, 100, 30, probe=8)], 60) == []


def test_predictions_and_pca(px):
    rng = np.random.default_rng(0)

    def predict(d):
        X = rng.standard_normal((500, d)).astype(np.float32)
        m = px.MLP(d, seed=1)

        def once(want):
            got = m.predict(X)
            return got if want is None else np.array_equal(got, want)
        return once

    def pca(D, dout):
        X = rng.standard_normal((400, D)).astype(np.float32)

        def once(want):
            got = px.pca(X, dout)
            if want is None:
                return got
            return all(np.abs(a - b).max() <= 1e-5 * np.abs(b).max() for a, b in zip(got, want))
        return once

    assert run_together([predict(50), predict(200), predict(128), pca(30, 4), pca(70, 60)], 40) == []
