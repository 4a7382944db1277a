"""The network's tensor-core convolutions at the edges of their tiles: lines
longer than a tile (its neighbouring rows are copied as segments), planes
shorter than one, channel counts one above a 16-channel block and at the
64-channel limit.

Bounds as for the network's other parity tests: outputs within 1e-4 of max|y|
(eleven layers of ~2^-17 each), gradients within 2e-3 of the layer's max|g|.
"""
import numpy as np
import pytest

from oracle import nn as onn

from gpu_util import cuda_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,channels,cout", [((27, 27, 540), (3, 4, 5, 6), 4), ((27, 27, 27), (17, 48, 64, 33), 9),
                                             ((54, 27, 81), (16, 1, 15, 32), 17)])
def test_convolutions_at_tile_edges(N, channels, cout):
    torch = cuda_or_skip()
    from paper_1004_1122_gb300 import fh

    rng = np.random.default_rng(7)
    params = [(w, (rng.normal(size=b.shape) * 0.05).astype(np.float32))
              for (w, b) in onn.init_params(2, cout, seed=5, channels=channels)]
    x = rng.normal(size=(2,) + N).astype(np.float32)
    target = rng.normal(size=(cout,) + N).astype(np.float32)
    net = fh.Net(N, 2, cout, channels=channels)
    net.set_params(np.concatenate([np.concatenate([w.reshape(-1), b]) for w, b in params]).astype(np.float32))
    y = net.forward(torch.from_numpy(x).cuda()).cpu().numpy()
    _, flat = net.gradients(torch.from_numpy(x).cuda(), torch.from_numpy(target).cuda())
    net.close()
    ref, _ = onn.forward(params, x.astype(np.float64), round_bf16=True)
    assert np.max(np.abs(y - ref)) <= 1e-4 * np.max(np.abs(ref))
    _, grads, _ = onn.loss_and_grads(params, x.astype(np.float64), target.astype(np.float64))
    k = 0
    for layer, (rw, rb) in enumerate(grads):
        g = flat[k:k + rw.size + rb.size]
        k += g.size
        r = np.concatenate([rw.reshape(-1), rb])
        assert np.max(np.abs(g - r)) <= 2e-3 * np.max(np.abs(r)), layer
    assert k == flat.size
