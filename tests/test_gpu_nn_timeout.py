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
