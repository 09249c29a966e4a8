"""The tensor-core path (d = 64) where the screen leaves its binade and squared
distances overflow FP32: every point is decided over all K, and the labels,
which index the sorted sums, stay in 0..K-1 and equal the oracle's."""
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


def _check(km, oracle, x, mu0, steps, **kw):
    ref = oracle.run(x, mu0, steps, 0.0)
    g = km.KMeans(x.shape[1], 64, mu0.shape[0], **kw)
    g.set_points(x)
    g.set_init(mu0)
    r = g.run(steps, 0.0)
    assert g.stats()["path"] == 3
    assert r["iters"] == ref["iters"] and np.array_equal(r["labels"], ref["labels"])
    assert np.array_equal(g.counts(), ref["counts"])
    assert np.allclose(r["centroids"], ref["centroids"], rtol=1e-6, atol=1e-6 * np.abs(x).max())
    g.close()


# the last scale inside the binade, the first outside, squares at and beyond
# FP32's largest value, and coordinates near the accepted limit; one group of
# 256 columns with and without padding, and several; from 2^20 points on the
# rescue list is taken in tiles first
@pytest.mark.parametrize("tc", ["bf16", "f16"])
@pytest.mark.parametrize("n,k,scale", [(3001, 40, 1e15), (3001, 40, 3e16), (3001, 300, 1e17), (3001, 256, 1e18),
                                       (3001, 1, 1e18), (2000, 40, 2e19), (2000, 7, 1e28), ((1 << 20) + 5, 3, 1e18)])
def test_large_magnitudes(km, oracle, n, k, scale, tc):
    x, _, _ = synth.iso_mixture(n, 64, max(2, k // 2), sigma=1.0, box=8.0, seed=n + k)
    x = (x.astype(np.float64) * scale).astype(np.float32)
    mu0, _ = synth.init_distinct(x, k, seed=1)
    _check(km, oracle, x, mu0, 3, tc_operands=tc)


# starting centroids whose distances overflow FP32, or FP64 as well (the lowest
# index takes the points), all of them or one
@pytest.mark.parametrize("far,which", [(1e25, slice(None)), (1e200, slice(None)), (1e200, slice(0, 1))])
def test_far_centroids(km, oracle, far, which):
    x, _, _ = synth.iso_mixture(2000, 64, 5, sigma=1.0, box=8.0, seed=9)
    mu0, _ = synth.init_distinct(x, 9, seed=2)
    mu0[which] = np.random.default_rng(3).normal(size=mu0[which].shape) * far
    _check(km, oracle, x, mu0, 3)
