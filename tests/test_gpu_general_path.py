"""The general path's centroid tiles and sum windows at their limits, one step
against the oracle."""
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


# the general path's sums: every number of windows a block can have (from one to 32,
# and none), the limits of the small centroid tile, and more tiles a block than
# windows take between flushes
@pytest.mark.parametrize("n,d,k", [(100, 5, 2), (70_000, 5, 2), (5_200_001, 5, 2), (300_000, 7, 3), (300_000, 31, 5),
                                   (200_003, 33, 16), (200_003, 12, 17), (200_001, 16, 64), (60_000, 40, 130),
                                   (30_000, 48, 200), (20_000, 64, 9)])
def test_general_path_windows(km, oracle, n, d, k):
    x, _, _ = synth.iso_mixture(n, d, max(2, k // 3), sigma=1.0, box=6.0, seed=n + d)
    mu0, _ = synth.init_distinct(x, k, seed=3)
    g = km.KMeans(n, d, k, dist_path="simt")
    g.set_points(x)
    g.set_init(mu0)
    g.step()
    z, mu_ref, cnt, e2 = oracle.step(x, mu0)
    assert g.stats()["path"] == 2
    assert np.array_equal(g.counts(), cnt) and np.array_equal(g.labels(), z)
    assert np.allclose(g.centroids(), mu_ref, rtol=1e-6, atol=1e-6)
    g.close()
