"""Refined solves are linear in the load over many orders of magnitude: the same
iterations, the same solution times the load's scale.

Bound: two solutions at tolerance 1e-8 differ by at most 2 kappa 1e-8 = 1e-6.
eta_r, the norm of a float32 step, agrees to the decrease of one step or two
where a last iteration falls differently: within a factor of 2.
"""
import numpy as np
import pytest

from paper_1004_1122_gb300 import microstructure as micro

from gpu_util import cuda_or_skip

pytestmark = pytest.mark.gpu

SCALES = [1e-14, 1e-13, 1e-12, 1e-11, 1e-9, 1e9, 1e15, 1e17]


@pytest.mark.parametrize("N", [(81, 81), (405, 375), (1215, 729), (45, 63, 81)])
def test_solution_scales_with_the_load(N):
    cuda_or_skip()
    from paper_1004_1122_gb300 import fh

    d = len(N)
    phase = (np.random.default_rng(5).random(N) < 0.35).astype(np.uint8)
    E = np.arange(1.0, d + 1.0) / d
    with fh.Solver(phase, micro.isotropic_table([1.0, 50.0], d), precision="fp32_refined") as s:
        x, col, info = s.solve(E, tol=1e-8, method="cg", max_iter=2000)
        x = x.clone()
        for scale in SCALES:
            xs, cs, i = s.solve(scale * E, tol=1e-8, method="cg", max_iter=2000)
            assert i["status"] == "FH_OK", (scale, i)
            assert abs(i["iters"] - info["iters"]) <= 2, (scale, i["iters"], info["iters"])
            assert float((xs / scale - x).norm()) <= 1e-6 * float(x.norm()), scale
            assert np.max(np.abs(cs / scale - col)) <= 1e-6 * np.max(np.abs(col)), scale
            assert 0.5 <= i["eta_r"] / info["eta_r"] <= 2.0, scale


@pytest.mark.parametrize("unit", [1e-15, 1e-8, 1e8])
def test_eta_r_scales_with_the_conductivity(unit):
    cuda_or_skip()
    from paper_1004_1122_gb300 import fh

    phase = (np.random.default_rng(5).random((135, 81)) < 0.35).astype(np.uint8)
    eta = []
    for u in (1.0, unit):
        with fh.Solver(phase, micro.isotropic_table([u, 50.0 * u], 2), precision="fp32_refined") as s:
            _, _, info = s.solve([1.0, 0.5], tol=1e-8, method="cg", max_iter=2000)
        assert info["status"] == "FH_OK"
        eta.append(info["eta_r"] / u)
    assert 0.5 <= eta[1] / eta[0] <= 2.0, eta


def test_batch_with_small_loads():
    cuda_or_skip()
    from paper_1004_1122_gb300 import fh

    rng = np.random.default_rng(6)
    cells = [(rng.random((n, n)) < 0.35).astype(np.uint8) for n in (27, 81, 81, 243)]
    tab = [micro.isotropic_table([1.0, 40.0], 2)] * len(cells)
    with fh.Batch(cells, tab, nloads=2, precision="fp32_refined") as b:
        ref, st, _, _ = b.solve(np.eye(2), tol=1e-8, method="cg", max_iter=2000)
        assert np.all(st == 0)
        # each load of its own size
        E = np.diag([1e-13, 1e-3])
        got, st, _, _ = b.solve(E, tol=1e-8, method="cg", max_iter=2000)
    assert np.all(st == 0), st
    assert np.max(np.abs(got / np.array([1e-13, 1e-3]) - ref)) <= 1e-6 * np.max(np.abs(ref))
