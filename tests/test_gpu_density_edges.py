"""The tensor-core response density at the edges of its items, against the FP64 oracle: chi lists on
both sides of 128 (whole tile or two halves) and 256 (one chunk of chi or several that add to rho),
phi lists on both sides of 64 and 128, lists whose phi stay in float32, one state, an odd and an
even count. Small cells in which every function touches most tiles, on a 30^3 grid (tiles of 8
leave a ragged tail of 6). float16 operands with float32 accumulation: 2e-3 of the largest entry,
as in the other tensor-core density tests."""
import numpy as np
import pytest

from oracle import operator as oop
from paper_1507_08157_gb300 import synthetic as sy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("natoms,nchi,k", [(14, 9, 3), (15, 9, 1), (17, 9, 4), (28, 9, 2), (29, 9, 3), (33, 4, 5),
                                           (40, 4, 2), (64, 4, 1), (66, 4, 3)])
def test_density_matches_oracle_at_list_edges(natoms, nchi, k):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_08157_gb300 import build, tddft
    build.build()
    s = sy.generate(sy.Recipe(natoms=natoms, cell_ang=9.4, ngrid=30, nchi=nchi, radius_ang=4.0, min_sep_ang=1.0,
                              seed=100 + natoms))
    ctx = tddft.Context(s, precision="mixed", precond="none")
    P = sy.random_kernels(s, k, 7)[1]
    P[-1] *= 1e-3                      # states of different scales share a pair
    rho, ref = ctx.response_density(P), oop.Operator(s).response_density(P)
    for q in range(k):
        assert np.max(np.abs(rho[q] - ref[q])) <= 2e-3 * np.max(np.abs(ref[q])), q
