"""Kernels at the sizes where their tiling, chunking or dispatch changes,
against the FP64 oracle (or plain FP64 numpy)."""
import numpy as np
import pytest

import synth
from oracle import setnet as osn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def km():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2405_12052_gb300 as m
    m.build()
    return m


# one tile; fewer tiles than backward blocks; the last sizes of the 64-point
# forward blocks and the first of the 256-point ones (77,824 points), the
# latter with a last block of 64 points; d below 3, K at its limits
@pytest.mark.parametrize("B,S,d,k", [(1, 64, 3, 16), (5, 192, 1, 1), (1215, 64, 3, 4), (19, 4096, 3, 16),
                                     (1217, 64, 2, 64)])
def test_setnet_tile_edges(km, B, S, d, k):
    rng = np.random.default_rng(B + S)
    p32 = osn.flatten(osn.init_params(d, k, 128, seed=B)).astype(np.float32)
    x = rng.normal(scale=3.0, size=(B, S, d)).astype(np.float32)
    t = rng.normal(scale=3.0, size=(B, k, d)).astype(np.float32)
    pr = osn.unflatten(p32.astype(np.float64), d, k)
    ref_loss, ref_g = osn.loss_and_grads(pr, x.astype(np.float64), t.astype(np.float64), k)
    net = km.SetNet(d, k)
    net.set_params(p32)
    loss = net.loss_grad(x, t)
    g = osn.unflatten(net.grads().astype(np.float64), d, k)
    # the bounds of the set network's other tests: loss 1e-5, gradients 1e-4
    assert abs(loss - ref_loss) <= 1e-5 * abs(ref_loss)
    for n in osn.PARAM_NAMES:
        err = np.linalg.norm(g[n] - ref_g[n]) / max(np.linalg.norm(ref_g[n]), 1e-30)
        assert err <= 1e-4, (n, err)
    c = net.predict(x)
    assert np.max(np.abs(c - osn.predict(pr, x.astype(np.float64), k))) <= 1e-4 * np.abs(x).max()
    net.close()


# chunk edges (4096 points), more chunks than pick threads, every d with its
# own kernel and the general one, magnitudes near the ends of the screen
@pytest.mark.parametrize("n,d,k,scale", [(4095, 1, 6, 1.0), (4096, 2, 9, 1.0), (4097, 3, 40, 1.0), (20_000, 4, 33, 1.0),
                                         (20_000, 5, 12, 1.0), (9_000, 17, 20, 1.0), (4_200_001, 3, 6, 1.0),
                                         (10_000, 3, 12, 1e-30), (10_000, 2, 12, 1e15), (10_000, 3, 12, 2e19)])
def test_kmeanspp_edges(km, oracle, n, d, k, scale):
    x, _, _ = synth.iso_mixture(n, d, max(k // 2, 1), sigma=1.0, box=10.0, seed=n + d)
    x = (x.astype(np.float64) * scale).astype(np.float32)
    x[:, n // 2:n // 2 + n // 10] = x[:, :n // 10]  # repeated points: D^2 = 0 once one of them is a centre
    u = np.random.default_rng(n).random(k)
    g = km.KMeans(n, d, k)
    g.set_points(x)
    mu, idx = g.init_kmeanspp(u)
    mu_ref, idx_ref = oracle.kmeanspp(x, k, u)
    assert np.array_equal(idx, idx_ref) and np.array_equal(mu, mu_ref)
    g.close()


@pytest.mark.parametrize("n,d,k,label_bytes", [(1, 1, 1, 4), (255, 2, 3, 4), (4096, 3, 9, 1), (4097, 6, 9, 4),
                                               (1_048_577 + 4096, 2, 5, 1)])
def test_objective_edges(km, n, d, k, label_bytes):
    x, _, _ = synth.iso_mixture(n, d, 3, sigma=1.0, box=10.0, seed=n + d)
    mu0, _ = synth.init_distinct(x, k, seed=7)
    g = km.KMeans(n, d, k, label_bytes=label_bytes)
    g.set_points(x)
    g.set_init(mu0)
    g.step()
    z, mu = g.labels().astype(np.int64), g.centroids()
    ref = float(((x.astype(np.float64) - mu[z].T) ** 2).sum())
    # two orders of n + d FP64 additions: pairwise and tree sums are each
    # within (log2(n d) + d + 16) ulps of the sum of the (positive) terms
    assert abs(g.objective() - ref) <= 2 * (np.log2(n * d + 1) + d + 16) * 2.0**-53 * ref
    g.close()


def _run_pair(km, x, mu0, max_iter, tol, **kw):
    """The same run by the whole-run kernel and by one host round trip per
    step (which compares every point with every centroid in every step)."""
    d, n = x.shape
    out = []
    for graph in (True, False):
        g = km.KMeans(n, d, mu0.shape[0], use_graph=graph, **kw)
        g.set_points(x)
        g.set_init(mu0)
        r = g.run(max_iter, tol)
        r2 = g.run(3, 0.0)  # continues from the first run's state
        out.append((r, g.stats()["empty_clusters"], r2, g.counts(), g.step(), g.labels()))
        g.close()
    return out


# every d, group counts with their own instance (kpad 32 and 256 in 3-D) and
# without, tiles at and around 256 points, fewer tiles than blocks and many per
# warp; data in clusters (few open points), spread evenly (many, and more steps
# than one launch takes), around an offset, on a grid (exact ties, duplicated
# and empty centroids), and near the ends of the float range
@pytest.mark.parametrize("kind,n,d,k,steps,kw", [
    ("mix", 1, 1, 1, 5, {}), ("mix", 255, 2, 3, 20, {}), ("mix", 257, 3, 8, 20, {}),
    ("even", 20_011, 1, 5, 150, {}), ("even", 30_000, 2, 11, 150, {}), ("even", 100_003, 3, 32, 100, {}),
    ("even", 50_000, 3, 100, 40, {"label_bytes": 1}), ("mix", 60_001, 3, 256, 30, {}), ("even", 40_000, 4, 7, 80, {}),
    ("mix", 30_000, 4, 256, 20, {"e_mode": "squared"}), ("mix", 1_300_007, 3, 17, 70, {"label_bytes": 1}),
    ("offset", 200_000, 3, 64, 40, {}), ("grid", 6_760, 2, 6, 30, {}), ("grid", 6_760, 2, 40, 30, {"label_policy": "final"}),
    ("tiny", 9_000, 3, 9, 40, {}), ("huge", 5_000, 3, 8, 15, {}), ("far", 30_000, 2, 9, 60, {}),
])
def test_whole_run_equals_step_by_step(km, oracle, kind, n, d, k, steps, kw):
    rng = np.random.default_rng(n + k)
    if kind == "even":
        x = rng.random((d, n), dtype=np.float32)
    elif kind == "grid":
        g1 = np.arange(-6, 7, dtype=np.float32)
        x = np.ascontiguousarray(np.tile(np.stack([m.ravel() for m in np.meshgrid(g1, g1)]), (1, 40))[:, :n])
    else:
        x, _, _ = synth.iso_mixture(n, d, max(2, k // 2), sigma=1.0, box=8.0, seed=n + d,
                                    offset=1e4 if kind == "offset" else 0.0)
        x = (x.astype(np.float64) * {"tiny": 1e-30, "huge": 1e18}.get(kind, 1.0)).astype(np.float32)
    mu0, _ = synth.init_distinct(x, k, seed=3)
    if kind == "grid":
        mu0[1] = mu0[0]          # a duplicated centroid (its twin takes no point)
    if kind == "far":
        mu0[:4] += 1e6           # centroids far outside the data, empty at first
    (a, ea, a2, ca, sa, za), (b, eb, b2, cb, sb, zb) = _run_pair(km, x, mu0, steps, 1e-7, **kw)
    for p, q in ((a, b), (a2, b2)):
        assert p["iters"] == q["iters"] and p["E"] == q["E"] and p["converged"] == q["converged"]
        assert np.array_equal(p["labels"], q["labels"]) and np.array_equal(p["centroids"], q["centroids"])
    assert ea == eb and np.array_equal(ca, cb) and sa == sb and np.array_equal(za, zb)
    if n <= 60_001 and not kw.get("label_policy"):
        ref = oracle.run(x, mu0, steps, 1e-7, e_mode=1 if kw.get("e_mode") else 0)
        assert a["iters"] == ref["iters"] and np.array_equal(a["labels"], ref["labels"])


# tiles of 256 points x 64 centroids x 32 coordinates and their edges; sums in
# shared windows with totals beside them, in the block's row, and (K d large)
# by global atomics; more points per block than one window flush
@pytest.mark.parametrize("n,d,k,kw", [
    (1, 5, 1, {}), (255, 31, 3, {}), (257, 32, 64, {}), (3000, 33, 65, {}), (200_003, 5, 7, {}), (100_001, 16, 64, {}),
    (20_000, 40, 130, {}), (5000, 70, 200, {}), (3000, 130, 257, {"label_policy": "final"}), (2000, 2, 1000, {}),
    (50_001, 7, 256, {"label_bytes": 1}), (20_003, 64, 100, {"dist_path": "simt"})])
def test_generic_tile_edges(km, oracle, n, d, k, kw):
    x, _, _ = synth.iso_mixture(n, d, max(2, k // 3), sigma=1.0, box=6.0, seed=n + d)
    x[:, n // 2:n // 2 + n // 20] = x[:, :n // 20]  # repeated points
    mu0, _ = synth.init_distinct(x, k, seed=3)
    if k > 2:
        mu0[2] = mu0[1]                            # an exact tie: the lowest index takes the points
    g = km.KMeans(n, d, k, **kw)
    g.set_points(x)
    mu = mu0
    for _ in range(2):
        g.set_init(mu)
        g.step()
        z, mu_ref, cnt, e2 = oracle.step(x, mu)
        assert np.array_equal(g.counts(), cnt)
        if kw.get("label_policy") is None:
            assert np.array_equal(g.labels(), z)
        assert np.allclose(g.centroids(), mu_ref, rtol=1e-6, atol=1e-6)
        mu = mu_ref
    assert g.stats()["path"] == 2
    g.close()


# the sorted sums' small and large chunks (2^21 points), each reservation of
# near-tie entries, several steps past the stop inside one graph, and a step
# after a converged run (its tables must be the final centroids')
@pytest.mark.parametrize("n,k,ops", [(5, 3, "bf16"), (20_001, 40, "f16"), (60_000, 300, "bf16"), (700_001, 32, "bf16"),
                                     (2_100_000, 16, "bf16")])
def test_tensor_run_and_step_after_it(km, oracle, n, k, ops):
    x, _, _ = synth.iso_mixture(n, 64, max(2, k // 2), sigma=1.0, box=6.0, seed=n)
    mu0, _ = synth.init_distinct(x, k, seed=5)
    steps = 30 if n < 1_000_000 else 3
    ref = oracle.run(x, mu0, steps, 1e-6)
    g = km.KMeans(n, 64, k, tc_operands=ops)
    g.set_points(x)
    g.set_init(mu0)
    r = g.run(steps, 1e-6)
    assert r["iters"] == ref["iters"] and np.array_equal(r["labels"], ref["labels"])
    g.step()
    z, _, cnt, _ = oracle.step(x, r["centroids"])
    assert np.array_equal(g.labels(), z) and np.array_equal(g.counts(), cnt)
    g.close()



# squared distances near FP32's overflow, for each packing width of the screen:
# the labels stay the oracle's
@pytest.mark.parametrize("scale", [1e9, 1e15, 1e18])
@pytest.mark.parametrize("d,k", [(1, 3), (2, 8), (3, 20), (3, 33), (2, 64), (1, 100), (4, 200)])
def test_large_magnitudes(km, oracle, d, k, scale):
    n = 8193
    x, _, _ = synth.iso_mixture(n, d, max(2, k // 2), sigma=1.5, box=8.0, seed=d + k)
    x = (x.astype(np.float64) * scale).astype(np.float32)
    mu0, _ = synth.init_distinct(x, k, seed=1)
    ref = oracle.run(x, mu0, 12, 0.0)
    for graph in (0, 1):
        g = km.KMeans(n, d, k, use_graph=graph)
        g.set_points(x)
        g.set_init(mu0)
        r = g.run(12, 0.0)
        assert r["iters"] == ref["iters"] and np.array_equal(r["labels"], ref["labels"])
        g.close()



# starting centroids so far out that every squared distance overflows FP64: the
# lowest index takes the points, and the moves leave FP32's range
@pytest.mark.parametrize("n,d,k", [(300, 2, 2), (1001, 3, 5), (9001, 1, 40)])
def test_far_centroids(km, oracle, n, d, k):
    x, _, _ = synth.iso_mixture(n, d, 3, sigma=1.0, box=8.0, seed=n)
    mu0 = np.random.default_rng(k).normal(size=(k, d)) * 1e200
    ref = oracle.run(x, mu0, 6, 0.0)
    for graph in (0, 1):
        g = km.KMeans(n, d, k, use_graph=graph)
        g.set_points(x)
        g.set_init(mu0)
        r = g.run(6, 0.0)
        assert np.array_equal(r["labels"], ref["labels"]) and np.allclose(r["centroids"], ref["centroids"], rtol=1e-6)
        g.close()
    for shape in ((8192, 256), (512, 128)):
        b = km.KMeansBatch([n], [d], [k])
        b.set_points([x])
        b.set_init([mu0])
        b.set_shape(*shape)
        r = b.run(6, 0.0)
        assert np.array_equal(r["labels"], ref["labels"])
        b.close()


# many steps of a batch whose tiles are skipped, taken from the lists of open
# points (few, many) or screened whole, against the shape that compares every
# point in every step: whole numbers and centroids are the same.  Instances of
# one point up to past the largest tile, at its edges and the 256-point ones;
# repeated points and a duplicated centroid are exact ties, some in FP64 every
# step; a second run continues the first
@pytest.mark.parametrize("scale", [1.0, 1e18])
@pytest.mark.parametrize("tile", [8192, 32768])
def test_batch_skipping_equals_every_point(km, oracle, tile, scale):
    sizes = [1, 2, 255, 256, 257, 1023, 1025, 2049, 8191, 8192, 8193, 32_767, 32_769, 70_001]
    ks = [1, 2, 7, 8, 33, 64]
    xs, mus = [], []
    for q, n in enumerate(sizes * 3):
        d, k = 1 + q // len(sizes), min(n, ks[q % len(ks)])
        x, _, _ = synth.iso_mixture(n, d, max(2, k // 2), sigma=1.5, box=8.0, seed=q)
        if q % 4 == 1:
            x = np.round(x)                          # a grid: exact ties
        x[:, n // 2:n // 2 + n // 20] = x[:, :n // 20]
        x = (x.astype(np.float64) * scale).astype(np.float32)
        mu = x[:, np.random.default_rng(q).permutation(n)[:k]].T.astype(np.float64)
        if k > 2 and q % 3 == 0:
            mu[1] = mu[0]
        xs.append(x)
        mus.append(mu)
    got = []
    for shape in ((tile, 256), (512, 128)):
        b = km.KMeansBatch([x.shape[1] for x in xs], [x.shape[0] for x in xs], [m.shape[0] for m in mus])
        b.set_points(xs)
        b.set_init(mus)
        b.set_shape(*shape)
        r = b.run(35, 0.0)
        r2 = b.run(12, 0.0)
        got.append([np.asarray(v) for s in (r, r2) for v in (s["labels"], s["centroids"], s["iters"], s["E"])]
                   + [b.counts()])
        b.close()
    for p, q in zip(*got):
        assert np.array_equal(p, q)
    off = 0
    for q, (x, m) in enumerate(zip(xs, mus)):
        if q % 5 == 0:
            ref = oracle.run(x, m, 35, 0.0)
            assert np.array_equal(got[0][0][off:off + x.shape[1]], ref["labels"]) and got[0][2][q] == ref["iters"]
        off += x.shape[1]
