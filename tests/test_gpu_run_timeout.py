"""A whole run whose wait for the other blocks gives up by its limit: the call says
so, the context closes cleanly and the next one works.  The kernel waits for an
arrival that nothing makes; nothing hangs."""
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


@pytest.mark.parametrize("n,d,k", [(300, 2, 3), (200_000, 3, 32), (3_000_000, 3, 200)])
def test_run_wait_gives_up(km, n, d, k):
    import time
    x, _, _ = synth.iso_mixture(n, d, max(2, k // 2), sigma=1.0, box=8.0, seed=n)
    mu0, _ = synth.init_distinct(x, k, seed=1)
    g = km.KMeans(n, d, k)
    g.set_points(x)
    g.set_init(mu0)
    g.debug_run_wait_fails(2_000_000)
    t0 = time.perf_counter()
    with pytest.raises(km.KMError) as e:
        g.run(5, 0.0)
    assert e.value.status == -5 and time.perf_counter() - t0 < 2.0
    g.close()
    out = []
    for graph in (True, False):
        g = km.KMeans(n, d, k, use_graph=graph)
        g.set_points(x)
        g.set_init(mu0)
        out.append(g.run(5, 0.0))
        g.close()
    assert np.array_equal(out[0]["labels"], out[1]["labels"]) and out[0]["E"] == out[1]["E"]
