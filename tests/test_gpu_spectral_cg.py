"""The frequency-domain CG iteration of refined solves against the oracle's CG.

With a loose tolerance a refined solve from e = E is one float32 CG run, and
its residual history is comparable step by step with the oracle's float64 CG
(same recurrences in another basis).  Derivation of the bounds: float32 sums
and transforms perturb each residual norm by O(2^-24 log2 |N|) of the initial
one, amplified along the iteration by at most the contrast, so the leading
entries (down to 1e-3 of |e0|) agree within 1e-4 |e0| + 2 % of their value.
Solutions at tolerance 1e-9 agree with the oracle's to kappa * 1e-9 <= 1e-6.

Grids: compile-time plans of one, two and three stages, run-time plans, the
small-radix plans of small grids, extended radices, even axes, single lines
and odd line counts (unpaired lines in 3-D), anisotropic L and L0, cells that
are not cubes, several loads and several cells per launch.
"""
import numpy as np
import pytest

import oracle
from paper_1004_1122_gb300 import microstructure as micro

from gpu_util import cuda_or_skip, spd

pytestmark = pytest.mark.gpu

GRIDS = [(75, 81), (135, 225), (243, 125), (405, 375), (3, 1125), (1215, 9), (105, 189), (49, 35), (21, 3),
         (17, 85), (16, 30), (27, 27, 27), (25, 75, 81), (3, 5, 7), (9, 21, 15), (135, 3, 25), (17, 9, 13), (6, 8, 10)]


def _problem(N, aniso):
    d = len(N)
    rng = np.random.default_rng(sum(N) + 7 * d)
    phase = (rng.random(N) < 0.35).astype(np.uint8)
    if not aniso:
        L = micro.isotropic_table([1.0, 30.0], d)
        return phase, L, oracle.reference_medium(L), np.ones(d)
    L = np.stack([spd(rng, d, 0.5, 2.0), spd(rng, d, 3.0, 9.0)])
    # a slightly anisotropic reference medium: CG on I + B needs it near isotropic
    L0 = 4.0 * np.eye(d) + 0.1 * spd(rng, d, 0.5, 2.0)
    return phase, L, L0, rng.uniform(0.5, 2.0, size=d)


@pytest.mark.parametrize("N", GRIDS)
@pytest.mark.parametrize("aniso", [False, True])
def test_refined_cg_follows_the_oracle(N, aniso):
    torch = cuda_or_skip()
    from paper_1004_1122_gb300 import fh

    phase, L, L0, Y = _problem(N, aniso)
    d = len(N)
    E = np.arange(1.0, d + 1.0) / d
    with fh.Solver(phase, L, L0=L0, Y=Y, precision="fp32_refined") as s:
        _, _, first = s.solve(E, tol=5e-3, method="cg", history=64, max_iter=64)
        x, col, info = s.solve(E, tol=1e-9, method="cg", max_iter=20000)
    assert info["status"] == "FH_OK", info
    xo, io = oracle.cg(phase, L, L0, E, Y=Y, tol=1e-12, max_iter=5000)
    h = first["history"]
    n = min(len(h), len(io["history"]))
    assert n > 1
    ref = np.asarray(io["history"][:n])
    if not aniso:  # the theory of CG on I + B covers isotropic L0 only
        assert np.all(np.abs(h[:n] - ref) <= 1e-4 + 0.02 * ref), (h[:n], ref)
    assert np.linalg.norm(x.cpu().numpy() - xo) <= 1e-6 * np.linalg.norm(xo)


@pytest.mark.parametrize("N", [(81, 135), (63, 21), (27, 45, 75), (15, 9, 21)])
def test_all_loads_match_single_loads(N):
    torch = cuda_or_skip()
    from paper_1004_1122_gb300 import fh

    phase, L, L0, Y = _problem(N, False)
    with fh.Solver(phase, L, L0=L0, Y=Y, precision="fp32_refined") as s:
        Le, infos = s.solve_all(tol=1e-9)
        cols = [s.solve(e, tol=1e-9, want_field=False)[1] for e in np.eye(len(N))]
    assert all(i["status"] == "FH_OK" for i in infos)
    assert np.max(np.abs(Le - np.stack(cols, axis=1))) <= 1e-7 * np.max(np.abs(Le))


@pytest.mark.parametrize("N", [(75, 81), (405, 225), (135, 3), (25, 75, 81), (81, 27, 135), (3, 135, 75), (5, 7, 3)])
@pytest.mark.parametrize("transpose", [False, True])
def test_float32_product_in_place(N, transpose):
    """The operator's product on the same passes.  Bound: 64 u (1 + max|dL|)
    max|e| of the FFT stages, times 4 for the packed line transforms."""
    torch = cuda_or_skip()
    from paper_1004_1122_gb300 import fh

    phase, L, L0, Y = _problem(N, True)
    e = np.random.default_rng(1).normal(size=(len(N),) + N).astype(np.float32)
    ref = (oracle.apply_AT if transpose else oracle.apply_A)(e.astype(np.float64), phase, L, L0, Y)
    with fh.Solver(phase, L, L0=L0, Y=Y, precision="fp32") as s:
        x = torch.from_numpy(e).cuda()
        got = s.apply(x, transpose=transpose).double().cpu().numpy()
        s.apply(x, out=x, transpose=transpose)
    tol = 4 * 64 * 2.0 ** -24 * (1.0 + np.max(np.abs(L - L0[None]))) * np.max(np.abs(e))
    assert np.max(np.abs(got - ref)) <= tol
    assert np.array_equal(x.double().cpu().numpy(), got)
