"""Batched runs of few and many steps: launched one by one or from the graph, with
first steps repeated while the moves are large."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def km():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2405_12052_gb300 as m
    m.build()
    return m


# batches: runs shorter than the graph, its length and more, in shapes that skip
# points and in one that compares all; starts in a corner make first steps of
# later ones
@pytest.mark.parametrize("tile,threads", [(8192, 256), (32768, 256), (1024, 256)])
@pytest.mark.parametrize("steps", [1, 3, 8, 11, 40])
def test_batch_of_few_and_many_steps(km, tile, threads, steps):
    rng = np.random.default_rng(steps)
    sizes = [(1, 1, 1), (300, 2, 7), (8193, 3, 64), (20_000, 1, 30), (70_001, 3, 16)]
    xs = [rng.random((d, n), dtype=np.float32) for n, d, _ in sizes]
    mus = [rng.random((k, d)) * (0.01 if q % 2 else 1.0) for q, (_, d, k) in enumerate(sizes)]
    got = []
    for shape, graph in (((tile, threads), True), ((tile, threads), False), ((512, 128), False)):
        b = km.KMeansBatch([s[0] for s in sizes], [s[1] for s in sizes], [s[2] for s in sizes], use_graph=graph)
        b.set_points(xs)
        b.set_init(mus)
        b.set_shape(*shape)
        r, r2 = b.run(steps, 0.0), b.run(steps, 1e-3)
        got.append([np.asarray(v) for s in (r, r2) for v in (s["labels"], s["centroids"], s["iters"], s["E"], s["converged"])]
                   + [b.counts()])
        b.close()
    for other in got[1:]:
        for p, q in zip(got[0], other):
            assert np.array_equal(p, q)
