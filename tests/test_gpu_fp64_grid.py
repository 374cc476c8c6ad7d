"""The float64 grid contractions by exact splitting on the tensor cores, against the FP64 oracle, at the
edges of their blocks: chi lists on both sides of 64, 128 and 448 (one accumulation or two), phi lists
on both sides of 32 and no multiple of four per atom (density on the CUDA cores), one state and
several, states of very different scales and a state of zeros, ragged grid (30^3).

Tolerance: 1e-13 of a state's largest entry. Each of the at most ~5e4 terms of an entry (512 points of
about 60 tiles, or 459 x 204 pairs of functions) carries a rounding error of 2^-53 of its own size in
either computation; adding in quadrature, 2 sqrt(5e4) 2^-53 = 5e-14 of the terms' size, which the
largest entry is not below."""
import numpy as np
import pytest

from oracle import grid as ogrid
from paper_1507_08157_gb300 import synthetic as sy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("natoms,nchi,nphi,k", [(7, 9, 4, 1), (8, 9, 4, 3), (14, 9, 4, 2), (15, 9, 4, 3), (9, 4, 4, 1),
                                                (9, 4, 3, 2), (51, 9, 4, 2)])
def test_float64_grid_contractions_match_oracle(natoms, nchi, nphi, k):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_08157_gb300 import build, tddft
    build.build()
    s = sy.generate(sy.Recipe(natoms=natoms, cell_ang=9.4, ngrid=30, nchi=nchi, nphi=nphi, radius_ang=4.0,
                              min_sep_ang=1.0, seed=300 + natoms))
    ctx = tddft.Context(s, precision="fp64", precond="none")
    chi, phi = ogrid.BoxedSet(s.chi, s.n), ogrid.BoxedSet(s.phi, s.n)
    P = sy.random_kernels(s, k, 11)[0]
    V = np.random.default_rng(natoms).standard_normal((k, s.n, s.n, s.n))
    P[-1] *= 1e-30
    V[-1] *= 1e+25
    if k == 3:
        P[1], V[1] = 0.0, 0.0
    rho, ref = ctx.response_density(P), ogrid.response_density(chi, phi, P)
    out, oref = ctx.potential_integrals(V), ogrid.potential_integrals(chi, phi, V, s.dV)
    for q in range(k):
        assert np.max(np.abs(rho[q] - ref[q])) <= 1e-13 * np.max(np.abs(ref[q])), q
        assert np.max(np.abs(out[q] - oref[q])) <= 1e-13 * np.max(np.abs(oref[q])), q
