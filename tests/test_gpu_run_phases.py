"""Runs that compare every point first and skip points later: the steps' results
do not depend on which kernel took them, nor on where one follows the other."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def km():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2405_12052_gb300 as m
    m.build()
    return m


def _equal(a, b):
    assert a["iters"] == b["iters"] and a["E"] == b["E"] and a["converged"] == b["converged"]
    assert np.array_equal(a["labels"], b["labels"]) and np.array_equal(a["centroids"], b["centroids"])


# from 2^23 points on the first steps are the step kernels'; one step and the
# step before the limit are theirs too, a tolerance can be met among them, and a
# second run starts with them again
@pytest.mark.parametrize("n,d,k,kw", [((1 << 23) - 1, 1, 5, {}), (1 << 23, 2, 8, {"e_mode": "squared"}),
                                      ((1 << 23) + 5, 3, 4, {"label_bytes": 1}), ((1 << 23) + 256, 3, 32, {"label_policy": "final"})])
def test_large_sets(km, n, d, k, kw):
    import torch
    g0 = torch.Generator(device="cuda").manual_seed(n)
    mu = (torch.rand(k, d, generator=g0, device="cuda") * 2 - 1) * 20
    c = torch.randint(k, (n,), generator=g0, device="cuda")
    x = torch.empty(d, n, device="cuda")
    x.copy_((mu[c] + torch.randn(n, d, generator=g0, device="cuda")).t())
    mu0 = (x[:, :k].t().double().cpu().numpy() + mu.double().cpu().numpy()) / 2
    a, b = (km.KMeans(n, d, k, use_graph=graph, **kw) for graph in (True, False))
    for g in (a, b):
        g.set_points(x, borrow=True)
    for steps, tol in ((1, 0.0), (2, 0.0), (3, 0.0), (7, 0.0), (40, 1e-3), (5, 1e9), (1, 1e9)):
        for g in (a, b):
            g.set_init(mu0)
        _equal(a.run(steps, tol), b.run(steps, tol))
        _equal(a.run(2, 0.0), b.run(2, 0.0))
        sa, sb = a.stats(), b.stats()
        assert all(sa[q] == sb[q] for q in ("iters", "converged", "e", "e2", "empty_clusters"))
        assert np.array_equal(a.counts(), b.counts()) and a.step() == b.step()
    a.close()
    b.close()


# starts in a corner of evenly spread points: the moves stay large for more steps
# than one launch takes, so every step decides every point afresh, across launches
# too, then settle
@pytest.mark.parametrize("n,d,k,steps", [(20_011, 1, 40, 140), (20_011, 1, 8, 140), (20_000, 2, 30, 140), (700_000, 3, 9, 100)])
def test_moves_that_stay_large(km, oracle, n, d, k, steps):
    rng = np.random.default_rng(n + k)
    x = rng.random((d, n), dtype=np.float32)
    mu0 = rng.random((k, d)) * 0.01
    out = []
    for graph in (True, False):
        g = km.KMeans(n, d, k, use_graph=graph)
        g.set_points(x)
        g.set_init(mu0)
        out.append((g.run(steps, 1e-9), g.run(3, 0.0), g.counts()))
        g.close()
    _equal(out[0][0], out[1][0])
    _equal(out[0][1], out[1][1])
    assert np.array_equal(out[0][2], out[1][2])
    if n < 100_000:
        ref = oracle.run(x, mu0, steps, 1e-9)
        assert np.array_equal(out[0][0]["labels"], ref["labels"]) and out[0][0]["iters"] == ref["iters"]
