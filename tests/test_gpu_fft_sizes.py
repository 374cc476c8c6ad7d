"""The FFT Poisson potential at grid sizes that take every pair of stages (4x4, 4x2, 4x3, 2x3, 2x5, 3x3,
3x5), single stages of every radix, both layouts of the lines (n a multiple of 8 or not), the smallest
and the largest grid, and an odd number of states (an unpaired last one). Tolerances, relative to the
largest entry: float64 1e-10, float32 3e-5 (transforms of at most 2^24 points, roundoff 6e-8 a stage and
at most 24 stages, with margin)."""
import numpy as np
import pytest

from oracle import hartree as ohartree
from oracle import xc as oxc
from paper_1507_08157_gb300 import synthetic as sy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n,k", [(8, 3), (9, 1), (10, 2), (12, 1), (15, 3), (16, 1), (18, 1), (25, 1), (27, 2), (40, 3), (50, 1),
                                 (60, 2), (64, 1), (81, 1), (90, 1), (96, 2), (100, 1), (120, 1), (125, 1), (256, 1)])
def test_potential_at_grid_sizes(n, k, prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_08157_gb300 import build, tddft
    build.build()
    s = sy.generate(sy.Recipe(natoms=1, cell_ang=8.0, ngrid=n, radius_ang=2.0, seed=3))
    ctx = tddft.Context(s, precision=prec, precond="none")
    rho = np.random.default_rng(n).standard_normal((k, n, n, n))
    got = ctx.response_potential(rho)
    ref = np.stack([ohartree.hartree(r, s.cell) for r in rho]) + oxc.fxc_lda(s.n0)[None] * rho
    assert np.max(np.abs(got - ref)) <= {"fp64": 1e-10, "mixed": 3e-5}[prec] * np.max(np.abs(ref))
