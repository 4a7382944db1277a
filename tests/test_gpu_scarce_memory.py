"""Contexts whose frequency-layout buffers do not fit the memory that is left run
the passes on fields: what fits without those buffers is not refused.

The memory a context takes is measured first; then all but that much less 60 MB
(the 3-D frequency-layout passes take 115 MB of it on this grid) is held while
another is created.  Product bound as for the float32 products elsewhere: 64 u
(1 + max|dL|) max|e|, times 4 for the packed line transforms, each way; solutions
at tolerance 1e-8 agree to 2 kappa 1e-8.
"""
import numpy as np
import pytest

from paper_1004_1122_gb300 import microstructure as micro

from gpu_util import cuda_or_skip

pytestmark = pytest.mark.gpu

N = (243, 243, 243)
KEEP = 60 << 20


def _tight(torch, fh, args, kw, less=KEEP):
    """A context created in the memory an ordinary one takes, less `less` bytes."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    with fh.Solver(*args, **kw):
        torch.cuda.synchronize()
        took = before - torch.cuda.mem_get_info()[0]
    free = torch.cuda.mem_get_info()[0]
    junk = torch.empty(free - took + less, dtype=torch.uint8, device="cuda")
    try:
        return fh.Solver(*args, **kw)
    finally:
        del junk
        torch.cuda.empty_cache()


@pytest.mark.parametrize("precision", ["fp32", "fp32_refined"])
def test_a_context_without_the_frequency_buffers(precision):
    torch = cuda_or_skip()
    from paper_1004_1122_gb300 import fh

    phase = (np.random.default_rng(2).random(N) < 0.3).astype(np.uint8)
    args, kw = (phase, micro.isotropic_table([1.0, 20.0], 3)), {"precision": precision}
    g = torch.Generator(device="cuda").manual_seed(1)
    e = torch.randn((3,) + N, generator=g, device="cuda")
    with fh.Solver(*args, **kw) as s:
        ref = [s.apply(e, transpose=t).clone() for t in (False, True)]
        if precision == "fp32_refined":
            x = s.solve([1.0, 0.5, 0.25], tol=1e-8)[0].clone()
    with _tight(torch, fh, args, kw) as s:
        got = [s.apply(e, transpose=t) for t in (False, True)]
        tol = 2 * 4 * 64 * 2.0 ** -24 * (1.0 + 9.5) * float(e.abs().max())
        for a, b in zip(ref, got):
            assert float((a - b).abs().max()) <= tol
        if precision == "fp32_refined":
            y, _, info = s.solve([1.0, 0.5, 0.25], tol=1e-8)
            assert info["status"] == "FH_OK"
            assert float((y - x).norm()) <= 2 * 20 * 1e-8 * float(x.norm())


def test_a_context_without_the_second_direction_buffer():
    """Refined contexts allocate CG's second direction (12 bytes per node) with
    the others; methods that need none run where it does not fit."""
    torch = cuda_or_skip()
    from paper_1004_1122_gb300 import fh

    phase = (np.random.default_rng(2).random(N) < 0.3).astype(np.uint8)
    args, kw = (phase, micro.isotropic_table([1.0, 4.0], 3)), {"precision": "fp32_refined"}
    with _tight(torch, fh, args, kw, less=220 << 20) as s:
        _, _, info = s.solve([1.0, 0.5, 0.25], tol=1e-6, method="fixed_point")
    assert info["status"] == "FH_OK"
