"""The frequency-domain CG iteration forms (r+, r+) from measured products, so
that it runs the recurrences of CG also where A is not symmetric: with a clearly
anisotropic reference medium its residual history is the oracle's.

Bound: with a loose tolerance the solve is one float32 run from e = E.  Eight
steps, each perturbed by O(2^-24 log2 |N|) < 3e-6 of the residuals before it,
with alpha and beta of order one: 1e-4 of the largest residual so far.
"""
import numpy as np
import pytest

import oracle

from gpu_util import cuda_or_skip, spd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [(75, 81), (135, 225), (49, 35), (16, 34), (25, 75, 81), (9, 21, 15), (6, 8, 10)])
@pytest.mark.parametrize("L0", [(3.0, 6.0, 4.0), (2.5, 3.0, 9.0)])
def test_history_with_an_anisotropic_reference_medium(N, L0):
    cuda_or_skip()
    from paper_1004_1122_gb300 import fh

    d = len(N)
    rng = np.random.default_rng(sum(N))
    phase = (rng.random(N) < 0.35).astype(np.uint8)
    L = np.stack([spd(rng, d, 0.5, 2.0), spd(rng, d, 3.0, 9.0)])
    L0 = np.diag(L0[:d])
    E = np.arange(1.0, d + 1.0) / d
    with fh.Solver(phase, L, L0=L0, precision="fp32_refined") as s:
        _, _, info = s.solve(E, tol=5e-3, method="cg", history=64, max_iter=8)
    _, ref = oracle.cg(phase, L, L0, E, tol=1e-12, max_iter=8)
    h, r = np.asarray(info["history"]), np.asarray(ref["history"])
    n = min(len(h), len(r))
    assert n >= 5
    assert np.all(np.abs(h[:n] - r[:n]) <= 1e-4 * np.maximum.accumulate(r[:n])), (h[:n], r[:n])
