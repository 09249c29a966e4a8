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


# tiles of 128 points x 64 centroids x 32 coordinates and their edges; sums in
# shared windows with totals beside them, in the block's row, and (K d large)
# by global atomics; more points per block than one window flush
@pytest.mark.parametrize("n,d,k,kw", [
    (1, 5, 1, {}), (127, 31, 3, {}), (129, 32, 64, {}), (3000, 33, 65, {}), (200_003, 5, 7, {}), (100_001, 16, 64, {}),
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


# the sorted sums' small and large chunks (2^21 points), several steps past
# the stop inside one graph, and a step after a converged run (its tables must
# be the final centroids')
@pytest.mark.parametrize("n,k,ops", [(5, 3, "bf16"), (20_001, 40, "f16"), (60_000, 300, "bf16"), (2_100_000, 16, "bf16")])
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
