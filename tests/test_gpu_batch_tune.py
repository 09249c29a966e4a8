"""The tuner's timings do not depend on whether the instances have been run."""
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


def test_tuning_after_a_run(km):
    xs = [synth.iso_mixture(n, 3, 30, sigma=1.0, box=8.0, seed=n)[0] for n in (400_000, 300_000, 3000)]
    mus = [synth.init_distinct(x, 60, seed=1)[0] for x in xs]
    b = km.KMeansBatch([x.shape[1] for x in xs], [3] * 3, [60] * 3)
    b.set_points(xs)
    b.set_init(mus)
    b.tune()
    before = b.info()["tune_ms"]
    r = b.run(3, 0.0)  # every instance stops at the limit
    b.tune()
    after = b.info()["tune_ms"]
    assert len(after) == len(before) == 8
    assert all(q > 0.3 * p for p, q in zip(before, after)), (before, after)
    # centroids, steps and results are as without the tuning
    s = b.run(2, 0.0)
    c = km.KMeansBatch([x.shape[1] for x in xs], [3] * 3, [60] * 3)
    c.set_points(xs)
    c.set_init(mus)
    c.set_shape(1024, 128)
    c.run(3, 0.0)
    t = c.run(2, 0.0)
    assert np.array_equal(s["labels"], t["labels"]) and np.array_equal(s["centroids"], t["centroids"])
    assert np.array_equal(s["iters"], t["iters"]) and np.array_equal(s["iters"], r["iters"] + 2)
    b.close()
    c.close()
