"""What a refined solve reports when its last inner solve takes no iteration:
eta_r is the norm of a step that was not made, exactly 0, whatever the
direction buffer held before."""
import numpy as np
import pytest

from paper_1004_1122_gb300 import microstructure as micro

from gpu_util import cuda_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [(45, 27), (81, 81), (405, 375), (21, 27, 15)])
@pytest.mark.parametrize("case", ["homogeneous", "zero load", "start off by a constant"])
def test_eta_r_is_zero_without_a_step(N, case):
    torch = cuda_or_skip()
    from paper_1004_1122_gb300 import fh

    d = len(N)
    E = np.zeros(d) if case == "zero load" else np.arange(1.0, d + 1.0)
    phase = (np.random.default_rng(3).random(N) < 0.3).astype(np.uint8)
    e_init = None
    if case == "start off by a constant":  # the complement part is corrected before the iteration
        e_init = torch.full((d,) + N, 1.5, device="cuda", dtype=torch.float64)
    with fh.Solver(phase, micro.isotropic_table([1e8, 7e8], d), precision="fp32_refined") as s:
        # leaves a direction whose norm ||L0 p||^2 is beyond float32
        s.solve(1e17 * np.arange(1.0, d + 1.0), tol=1e-2, method="cg")
        if case != "zero load":
            s.set_phase(np.zeros(N, np.uint8))
        x, _, info = s.solve(E, tol=1e-8, method="cg", e_init=e_init)
    assert info["status"] == "FH_OK" and info["iters"] == 0, info
    assert info["eta_r"] == 0.0
    ref = torch.tensor(E, device="cuda").reshape((d,) + (1,) * d)
    assert float((x - ref).abs().max()) <= 1e-7 * max(1.0, float(np.abs(E).max()))
