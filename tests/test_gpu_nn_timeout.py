"""Bounded waits of the network's tensor-core kernels that run out: with a limit
of a nanosecond copies and products are still in flight when the kernels give
up, finish what they have issued and return; the call reports FH_ERR_TIMEOUT
and nothing faults."""
import numpy as np
import pytest

from gpu_util import cuda_or_skip

pytestmark = pytest.mark.gpu

TIMEOUT = 8  # FH_ERR_TIMEOUT


def _network(torch, N, cin=2, cout=9, seed=0):
    from paper_1004_1122_gb300 import fh, warmstart

    g = torch.Generator(device="cuda").manual_seed(seed)
    net = fh.Net(N, cin, cout)
    net.set_params(warmstart.init_params(cin, 3, seed))
    x = torch.randn((cin,) + N, generator=g, device="cuda")
    t = torch.randn((cout,) + N, generator=g, device="cuda")
    return net, x, t


@pytest.mark.parametrize("N", [(27, 27, 27), (54, 81, 108), (27, 27, 540)])
def test_expired_waits_end_with_a_status(N):
    torch = cuda_or_skip()
    from paper_1004_1122_gb300 import fh

    net, x, t = _network(torch, N)
    ref = net.gradients(x, t)
    try:
        fh.set_wait_limit(1e-9)
        with pytest.raises(fh.FhError) as e:
            net.gradients(x, t)
        net.forward(x)
        torch.cuda.synchronize()
    finally:
        fh.set_wait_limit(0.0)
    assert e.value.status == TIMEOUT
    net.close()
    net, x, t = _network(torch, N)
    loss, grad = net.gradients(x, t)
    net.close()
    assert loss == ref[0] and np.array_equal(grad, ref[1])


@pytest.mark.parametrize("N", [(54, 54, 54), (108, 108, 108)])
def test_a_timeout_is_reported_once_and_changes_nothing(N):
    """The call after a timeout is an ordinary one, and a training step that
    timed out leaves the parameters alone; a forward whose waits expired is
    reported by the next synchronising call."""
    torch = cuda_or_skip()
    from paper_1004_1122_gb300 import fh

    net, x, t = _network(torch, N)
    params = net.get_params()
    ref = net.gradients(x, t)
    for call in (lambda: net.train_step(x, t, 1e-3), lambda: net.gradients(x, t)):
        try:
            fh.set_wait_limit(1e-9)
            with pytest.raises(fh.FhError) as e:
                call()
        finally:
            fh.set_wait_limit(0.0)
        assert e.value.status == TIMEOUT
        assert np.array_equal(net.get_params(), params)
        loss, grad = net.gradients(x, t)
        assert loss == ref[0] and np.array_equal(grad, ref[1])
    try:
        fh.set_wait_limit(1e-9)
        net.forward(x)
    finally:
        fh.set_wait_limit(0.0)
    with pytest.raises(fh.FhError) as e:
        net.gradients(x, t)
    assert e.value.status == TIMEOUT
    loss, grad = net.gradients(x, t)
    assert loss == ref[0] and np.array_equal(grad, ref[1])
    net.close()


def test_a_gradient_is_right_or_a_timeout():
    """The limit drops while the call runs (another thread sets it), so that at
    some of the moments only kernels of the backward pass give up."""
    torch = cuda_or_skip()
    import threading
    import time

    from paper_1004_1122_gb300 import fh

    net, x, t = _network(torch, (108, 108, 135))
    ref = net.gradients(x, t)
    for k in range(40):
        def drop(delay=5e-5 * k):
            end = time.perf_counter() + delay
            while time.perf_counter() < end:
                pass
            fh.set_wait_limit(1e-9)

        th = threading.Thread(target=drop)
        th.start()
        try:
            loss, grad = net.gradients(x, t)
        except fh.FhError as e:
            assert e.status == TIMEOUT
            loss = None
        finally:
            th.join()
            fh.set_wait_limit(0.0)
        if loss is not None:
            assert loss == ref[0] and np.array_equal(grad, ref[1]), k
    loss, grad = net.gradients(x, t)
    assert loss == ref[0] and np.array_equal(grad, ref[1])
    net.close()
