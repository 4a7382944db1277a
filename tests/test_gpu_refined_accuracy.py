"""The float32 rounding in refined CG solves, whose iteration runs in the
frequency domain, is no larger than in the same solves with the iteration on
fields.

BiCG of a symmetric system makes the steps of CG (isotropic media), and its
float32 iteration runs on the fields with the same refinement around it.  The
last inner solve stops where its recursive residual says so; the true residual
of the solution is that and, orthogonal to it, the rounding gathered on the way.
The rounding part is compared, because where within its last step's decrease a
recursion stops is chance.  Geometric mean over a set of cells: no larger than
BiCG's.
"""
import numpy as np
import pytest

from paper_1004_1122_gb300 import microstructure as micro

from gpu_util import cuda_or_skip

pytestmark = pytest.mark.gpu

TOL = 1e-8
# ends with the first inner solve, at the residual it hands over in every solve
# to a smaller tolerance
FIRST = 1.5e-3


def _balls(N, rng):
    d = len(N)
    at = np.stack(np.meshgrid(*[np.arange(n) for n in N], indexing="ij"))
    period = np.array(N).reshape((d,) + (1,) * d)
    phase = np.zeros(N, np.uint8)
    for _ in range(40 if d == 2 else 25):  # overlapping, periodic
        dist = np.abs(at - rng.random(d).reshape(period.shape) * period)
        dist = np.minimum(dist, period - dist)
        phase |= ((dist ** 2).sum(axis=0) <= (rng.uniform(0.05, 0.14) * min(N)) ** 2).astype(np.uint8)
    return phase


@pytest.mark.parametrize("contrast", [30.0, 100.0, 300.0])
def test_rounding_against_the_iteration_on_fields(contrast):
    cuda_or_skip()
    from paper_1004_1122_gb300 import fh

    ratios = []
    for N in [(147, 189), (315, 105), (135, 225), (96, 150), (45, 63, 35), (36, 48, 40)]:
        d = len(N)
        phase = _balls(N, np.random.default_rng(sum(N)))
        E = np.arange(1.0, d + 1.0) / d
        rounding = {}
        with fh.Solver(phase, micro.isotropic_table([1.0, contrast], d), precision="fp32_refined") as s:
            for method in ("cg", "bicg"):
                _, _, one = s.solve(E, tol=FIRST, method=method, max_iter=20000)
                _, _, two = s.solve(E, tol=TOL, method=method, max_iter=20000)
                assert one["status"] == two["status"] == "FH_OK"
                assert one["outer_iters"] == 1 and two["outer_iters"] == 2, (N, method)
                recursive = two["rel_res"] * one["rel_res_true"]
                assert two["rel_res_true"] > recursive
                rounding[method] = np.sqrt(two["rel_res_true"] ** 2 - recursive ** 2)
        ratios.append(rounding["cg"] / rounding["bicg"])
    assert np.exp(np.mean(np.log(ratios))) <= 1.0, ratios
