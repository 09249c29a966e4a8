"""A backward pass of the set network whose bounded wait gave up: it is reported,
its gradients change no parameter, and the network goes on from the next pass.
The give-up is marked from the host; no wait is made to fail."""
import numpy as np
import pytest

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


def _net(km):
    net = km.SetNet(3, 4)
    net.set_params(osn.flatten(osn.init_params(3, 4, 128, seed=1)).astype(np.float32))
    rng = np.random.default_rng(2)
    xs = [rng.normal(size=(3, 128, 3)).astype(np.float32) for _ in range(3)]
    ts = [rng.normal(size=(3, 4, 3)).astype(np.float32) for _ in range(3)]
    return net, xs, ts


def test_a_pass_that_gave_up_changes_nothing_and_the_next_one_works(km):
    ref, xs, ts = _net(km)
    ref.train_step(xs[0], ts[0], 1e-2)
    after_one = ref.params()
    ref.train_step(xs[2], ts[2], 1e-2)
    after_two, loss = ref.params(), ref.loss_grad(xs[1], ts[1])
    grads = ref.grads()

    net, _, _ = _net(km)
    net.train_step(xs[0], ts[0], 1e-2)
    net.loss_grad(xs[1], ts[1])
    net.debug_pass_gave_up()
    net.adam(1e-2)
    assert np.array_equal(net.params(), after_one)
    for _ in range(2):  # the pass stays failed until the next one
        with pytest.raises(km.KMError) as e:
            net.grads()
        assert e.value.status == -5
    net.train_step(xs[2], ts[2], 1e-2)  # bias corrections as if the failed step had not been asked for
    assert np.array_equal(net.params(), after_two)
    assert net.loss_grad(xs[1], ts[1]) == loss and np.array_equal(net.grads(), grads)
    net.close()
    ref.close()


def test_a_failed_pass_nobody_read_is_reported_once(km):
    net, xs, ts = _net(km)
    net.train_step(xs[0], ts[0], 1e-2, want_loss=False)
    net.debug_pass_gave_up()
    with pytest.raises(km.KMError) as e:
        net.train_step(xs[1], ts[1], 1e-2)
    assert e.value.status == -5 and "earlier" in str(e.value)
    net.train_step(xs[2], ts[2], 1e-2)
    net.grads()
    net.close()
