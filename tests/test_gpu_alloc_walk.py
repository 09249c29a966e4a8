"""Every device allocation of a workflow fails once, the optional ones too: the call
reports KM_ENOMEM, or goes on without the memory and gives the same results, and
all memory comes back."""
import gc

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


def _run(km, x, mu0, **kw):
    def fn():
        g = km.KMeans(x.shape[1], x.shape[0], mu0.shape[0], **kw)
        try:
            g.set_points(x)
            g.set_init(mu0)
            r, r2 = g.run(6, 0.0), g.run(3, 0.0)  # the second one without the memory as well
            return [r["labels"], r2["labels"], r2["centroids"], r2["E"], g.counts(), g.objective()]
        finally:
            g.close()
    return fn


def _seed(km, x, k):
    def fn():
        g = km.KMeans(x.shape[1], x.shape[0], k)
        try:
            g.set_points(np.ascontiguousarray(x.T), layout="nxd")
            return list(g.init_kmeanspp(np.random.default_rng(1).random(k)))
        finally:
            g.close()
    return fn


def _batch(km, insts, shape):
    def fn():
        b = km.KMeansBatch([w["n"] for w in insts], [w["d"] for w in insts], [w["k"] for w in insts])
        try:
            b.set_points([w["x"] for w in insts])
            b.set_init([w["mu0"] for w in insts])
            if shape:
                b.set_shape(*shape)
            r = b.run(12, 0.0)
            return [r["labels"], r["centroids"], r["iters"], r["E"], b.counts(), b.objective()]
        finally:
            b.close()
    return fn


def _net(km):
    def fn():
        net = km.SetNet(3, 4)
        try:
            rng = np.random.default_rng(3)
            net.set_params(rng.normal(scale=0.1, size=net.nparam).astype(np.float32))
            x, t = rng.normal(size=(2, 128, 3)).astype(np.float32), rng.normal(size=(2, 4, 3)).astype(np.float32)
            return [net.loss_grad(x, t), net.grads(), net.predict(x)]
        finally:
            net.close()
    return fn


# optional: the slacks of a run, its labels as bytes (unless the context's are) and
# the small buffers; of a batch six
@pytest.mark.parametrize("name,optional", [("run", 3), ("run_bytes", 2), ("run_general", 0), ("run_tensor", 0), ("seed", 0),
                                           ("batch", 6), ("batch_8192", 6), ("net", 0)])
def test_every_allocation_fails_once(km, name, optional):
    import torch
    x3, _, _ = synth.iso_mixture(30_000, 3, 8, seed=3)
    m3, _ = synth.init_distinct(x3, 8, seed=4)
    x6, _, _ = synth.iso_mixture(5_000, 6, 8, seed=5)
    m6, _ = synth.init_distinct(x6, 9, seed=6)
    x64, _, _ = synth.iso_mixture(3_000, 64, 8, seed=5)
    m64, _ = synth.init_distinct(x64, 16, seed=6)
    insts = synth.batch_instances(3, seed=7, n_lo=500, n_hi=9_000)
    fn = {"run": _run(km, x3, m3), "run_bytes": _run(km, x3, m3, label_bytes=1), "run_general": _run(km, x6, m6),
          "run_tensor": _run(km, x64, m64), "seed": _seed(km, x3, 9), "batch": _batch(km, insts, None),
          "batch_8192": _batch(km, insts, (8192, 256)), "net": _net(km)}[name]
    want = fn()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    survived = 0
    for n in range(200):
        km.debug_fail_alloc_after(n)
        try:
            got = fn()
        except km.KMError as e:
            assert e.status == -2, e
            got = None
        finally:
            left = km.debug_allocs_left()
            km.debug_fail_alloc_after(-1)
        gc.collect()
        assert got is not None or left == -1
        if got is not None:
            assert all(np.array_equal(a, b) for a, b in zip(got, want)) and len(got) == len(want)
            if left >= 0:
                break  # the workflow makes no more allocations
            survived += 1
    assert left >= 0 and n > 5 and survived == optional, (n, left, survived)
    torch.cuda.synchronize()
    assert abs(torch.cuda.mem_get_info()[0] - free0) < 64 << 20
