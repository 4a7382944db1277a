"""Float64 passes on spread FFT plans (one small butterfly per thread and
stage, radix 11, 13 and 17 split into output pairs) against the oracle.

Bounds as for every product: 64 u (1 + max|dL|) max|e|, u = 2^-53.  The CG
solution agrees with the oracle's to kappa times the tolerance.  Grids: split
radices first, after one another (twiddles in front of a split stage) and on
one axis only; a last stage of every whole radix; lengths 1 < n < 32 threads
and the largest grids of the rule; even axes; 3-D; batches of cells.
"""
import numpy as np
import pytest

import oracle
from paper_1004_1122_gb300 import microstructure as micro

from gpu_util import cuda_or_skip, spd

pytestmark = pytest.mark.gpu

GRIDS = [(17 * 11 * 3, 33), (13 * 13 * 5, 21), (187, 6), (33, 17 * 17 * 3), (154, 221), (91, 68), (4, 26), (49, 98),
         (81, 405), (22, 9, 39), (3, 51, 10), (27, 35, 4)]


@pytest.mark.parametrize("N", GRIDS)
def test_spread_product_and_solve(N):
    torch = cuda_or_skip()
    from paper_1004_1122_gb300 import fh

    d = len(N)
    rng = np.random.default_rng(sum(N))
    phase = (rng.random(N) < 0.4).astype(np.uint8)
    L = np.stack([spd(rng, d, 0.5, 2.0), spd(rng, d, 3.0, 9.0)])
    L0 = spd(rng, d, 3.0, 5.0)
    Y = rng.uniform(0.5, 2.0, size=d)
    e = rng.normal(size=(d,) + N)
    tol = 64 * 2.0 ** -53 * (1.0 + np.max(np.abs(L - L0[None]))) * np.max(np.abs(e))
    with fh.Solver(phase, L, L0=L0, Y=Y, precision="fp64") as s:
        for transpose in (False, True):
            got = s.apply(torch.from_numpy(e).cuda(), transpose=transpose).cpu().numpy()
            ref = (oracle.apply_AT if transpose else oracle.apply_A)(e, phase, L, L0, Y)
            assert np.max(np.abs(got - ref)) <= tol
    Li = micro.isotropic_table([1.0, 20.0], d)
    E = np.arange(1.0, d + 1.0)
    with fh.Solver(phase, Li, Y=Y, precision="fp64") as s:
        x, _, info = s.solve(E, tol=1e-10, method="cg", max_iter=2000)
    assert info["status"] == "FH_OK"
    xo, _ = oracle.cg(phase, Li, oracle.reference_medium(Li), E, Y=Y, tol=1e-12, max_iter=2000)
    assert np.linalg.norm(x.cpu().numpy() - xo) <= 1e-8 * np.linalg.norm(xo)
