"""What calls around a whole run (km_run in one kernel) see: its last step's sums,
its counters, and streams its grid does not fit on."""
import ctypes

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


# the sums after a run are the last step's, whichever driver ran it; an update
# without an assignment before it divides them again
@pytest.mark.parametrize("n,d,k,steps,kw", [(5000, 1, 3, 4, {}), (30_011, 2, 40, 70, {}), (20_000, 3, 256, 9, {"label_bytes": 1}),
                                            (9000, 4, 7, 5, {"label_policy": "final"}), (4_500_001, 3, 6, 12, {})])
def test_sums_after_a_run(km, n, d, k, steps, kw):
    x, _, _ = synth.iso_mixture(n, d, max(2, k // 2), sigma=1.5, box=8.0, seed=n, offset=50.0)
    mu0, _ = synth.init_distinct(x, k, seed=3)
    got = []
    for graph in (True, False):
        g = km.KMeans(n, d, k, use_graph=graph, **kw)
        g.set_points(x)
        g.set_init(mu0)
        g.run(steps, 0.0)
        t0 = g.shard_totals()
        g.begin(1, 0.0)
        t1 = g.shard_totals()
        g.update_async()
        g.sync()
        mu1, cnt1 = g.centroids(), g.counts()
        g.begin(1, 0.0)
        g.assign_async()
        got.append((t0, t1, mu1, cnt1, g.shard_totals()))
        g.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)


# no point is counted twice in a step.  At this magnitude the screen flags every
# point it decides; the start lies in a corner of the data, so the first moves open
# whole tiles again
@pytest.mark.parametrize("how", ["run", "batch"])
def test_flagged_points_are_counted_once(km, how):
    n, k, steps = 20_000, 20, 2
    x, _, _ = synth.iso_mixture(n, 3, 10, sigma=1.0, box=8.0, seed=5)
    x = (x.astype(np.float64) * 1e17).astype(np.float32)
    mu0, _ = synth.init_distinct(x, k, seed=6)
    mu0 = mu0.min(0) + 0.05 * (mu0 - mu0.min(0))
    if how == "run":
        g = km.KMeans(n, 3, k)
        g.set_points(x)
        g.set_init(mu0)
        g.run(steps, 0.0)
        assert 0 < g.stats()["flagged"] <= n
        g.close()
    else:
        b = km.KMeansBatch([n], [3], [k])
        b.set_points([x])
        b.set_init([mu0])
        b.set_shape(8192, 256)
        b.run(steps, 0.0)
        assert 0 < b.info()["flagged"] <= steps * n
        b.close()


def _green_stream(dev, sms):
    """A stream that owns at least `sms` SMs of the device (a green context), or None."""
    try:
        cu = ctypes.CDLL("libcuda.so.1")
        split, gen, create, stream = (getattr(cu, f) for f in ("cuDevSmResourceSplitByCount", "cuDevResourceGenerateDesc",
                                                              "cuGreenCtxCreate", "cuGreenCtxStreamCreate"))
    except (OSError, AttributeError):
        return None
    res, part, rest = (ctypes.create_string_buffer(256) for _ in range(3))  # CUdevResource: 144 bytes
    groups = ctypes.c_uint(1)
    desc, ctx, st = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    if cu.cuDeviceGetDevResource(dev, res, 1) or split(part, ctypes.byref(groups), res, rest, 0, sms):
        return None
    if gen(ctypes.byref(desc), part, 1) or create(ctypes.byref(ctx), desc, dev, 1):
        return None
    return None if stream(ctypes.byref(st), ctx, 1, 0) else st.value


# a stream on part of the GPU: the run's grid, sized for all of it, is not resident
# there, and the step kernels' graph runs instead
@pytest.mark.parametrize("n,d,k,kw", [(200_000, 3, 11, {}), (3_000_000, 2, 8, {"label_bytes": 1})])
def test_run_on_a_stream_with_fewer_sms(km, oracle, n, d, k, kw):
    import torch
    torch.cuda.init()
    torch.zeros(1, device="cuda")
    st = _green_stream(0, 16)
    if st is None:
        pytest.skip("no green contexts here")
    x, _, _ = synth.iso_mixture(n, d, k, sigma=1.0, box=8.0, seed=n)
    mu0, _ = synth.init_distinct(x, k, seed=3)
    ref = oracle.run(x, mu0, 6, 0.0)
    g = km.KMeans(n, d, k, stream=st, **kw)
    g.set_points(x)
    for _ in range(2):
        g.set_init(mu0)
        r = g.run(6, 0.0)
        assert r["iters"] == ref["iters"] and np.array_equal(r["labels"], ref["labels"])
        assert np.allclose(r["centroids"], ref["centroids"], rtol=1e-6, atol=1e-6)
    g.close()
