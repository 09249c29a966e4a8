"""Distinct contexts used from several threads at a time: the kernels' limits on
shared memory belong to the process, their sizes to each context."""
import threading

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


# the same kernel instance with little and with much shared memory on the fused
# path (steps, whole runs), the general path, the tensor-core path and in the
# set network
@pytest.mark.parametrize("d,ks,how", [(2, (3, 250), "step"), (2, (3, 250), "run"), (3, (5, 200), "run"), (6, (2, 500), "step"),
                                      (64, (4, 1000), "step"), (3, (1, 64), "net")])
def test_contexts_of_different_sizes_in_threads(km, d, ks, how):
    import torch
    n, rounds = 2048, 1500
    errors, out = [], {}
    gate = threading.Barrier(len(ks))

    def work(k):
        try:
            stream = torch.cuda.Stream()
            if how == "net":
                net = km.SetNet(d, k, stream=stream)
                rng = np.random.default_rng(k)
                net.set_params(rng.normal(scale=0.1, size=net.nparam).astype(np.float32))
                with torch.cuda.stream(stream):
                    x = torch.from_numpy(rng.normal(size=(1, 64, d)).astype(np.float32)).cuda()
                stream.synchronize()
                gate.wait()
                res = [net.predict(x) for _ in range(rounds)]
                out[k] = all(np.array_equal(r, res[0]) for r in res)
                net.close()
                return
            x, _, _ = synth.iso_mixture(n, d, max(2, k // 2), sigma=1.0, box=8.0, seed=k)
            mu0, _ = synth.init_distinct(x, k, seed=1)
            g = km.KMeans(n, d, k, stream=stream)
            g.set_points(x)
            gate.wait()
            got = []
            for _ in range(rounds):
                if how == "run":
                    g.set_init(mu0)
                    got.append(g.run(3, 0.0, want_labels=False)["centroids"])
                else:
                    if not got:
                        g.set_init(mu0)
                    g.step()
                    if len(got) < 3:
                        got.append(g.centroids())
            ref = km.KMeans(n, d, k, use_graph=False, stream=stream)
            ref.set_points(x)
            ref.set_init(mu0)
            want = []
            for _ in range(3):
                ref.step()
                want.append(ref.centroids())
            ok = all(np.array_equal(a, want[2]) for a in got) if how == "run" else all(
                np.array_equal(a, b) for a, b in zip(got, want))
            out[k] = ok
            g.close()
            ref.close()
        except Exception as e:  # reported by the test's thread
            errors.append((k, repr(e)))
            gate.abort()

    ts = [threading.Thread(target=work, args=(k,)) for k in ks]
    for t in ts:
        t.start()
    for t in ts:
        t.join(120)
    assert not errors, errors
    assert out == {k: True for k in ks}
