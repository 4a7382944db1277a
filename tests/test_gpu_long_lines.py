"""3-D boxes whose lines are too long for the frequency-layout row pass (one
pair of lines needs more threads than its kernels are compiled for): float32
products and refined solves take the passes on fields there.

Product bound as for the float32 products of shorter lines: 64 u (1 + max|dL|)
max|e| of the FFT stages, times 4 for the packed line transforms.  Solutions at
tolerance 1e-9 agree with the oracle's to kappa * 1e-9 <= 1e-6.
"""
import numpy as np
import pytest

import oracle
from paper_1004_1122_gb300 import microstructure as micro

from gpu_util import cuda_or_skip, spd

pytestmark = pytest.mark.gpu


# threads a pair of lines needs: 384 (one that fits), 544, 576, 640, 736, 768; the kernels take 512
@pytest.mark.parametrize("N", [(3, 3, 2520), (3, 3, 2625), (3, 5, 2835), (5, 3, 4375), (3, 4, 6561), (4, 3, 4096)])
@pytest.mark.parametrize("transpose", [False, True])
def test_float32_product_on_long_lines(N, transpose):
    torch = cuda_or_skip()
    from paper_1004_1122_gb300 import fh

    rng = np.random.default_rng(sum(N))
    phase = (rng.random(N) < 0.35).astype(np.uint8)
    L = np.stack([spd(rng, 3, 0.5, 2.0), spd(rng, 3, 3.0, 9.0)])
    L0 = oracle.reference_medium(L)
    e = rng.normal(size=(3,) + N).astype(np.float32)
    ref = (oracle.apply_AT if transpose else oracle.apply_A)(e.astype(np.float64), phase, L, L0)
    with fh.Solver(phase, L, L0=L0, precision="fp32") as s:
        got = s.apply(torch.from_numpy(e).cuda(), transpose=transpose).double().cpu().numpy()
    tol = 4 * 64 * 2.0 ** -24 * (1.0 + np.max(np.abs(L - L0[None]))) * np.max(np.abs(e))
    assert np.max(np.abs(got - ref)) <= tol


@pytest.mark.parametrize("N", [(3, 3, 2640), (3, 3, 2805), (3, 5, 2975)])
def test_refined_solve_on_long_lines(N):
    cuda_or_skip()
    from paper_1004_1122_gb300 import fh

    phase = (np.random.default_rng(sum(N)).random(N) < 0.35).astype(np.uint8)
    L = micro.isotropic_table([1.0, 30.0], 3)
    E = np.array([1.0, -0.5, 0.25])
    with fh.Solver(phase, L, precision="fp32_refined") as s:
        x, _, info = s.solve(E, tol=1e-9, method="cg", max_iter=5000)
    assert info["status"] == "FH_OK", info
    xo, _ = oracle.cg(phase, L, oracle.reference_medium(L), E, tol=1e-12, max_iter=5000)
    assert np.linalg.norm(x.cpu().numpy() - xo) <= 1e-6 * np.linalg.norm(xo)
