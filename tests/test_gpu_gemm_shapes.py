"""Products of a variable matrix with a constant one on the tensor cores (three-term TF32 split), through
the start of a solver state: P = P^c S L S P^v and its orthonormalisation, against the oracle. Sizes take
every tile width (32, 64, 112, 128), edges of one row or four past a tile of lanes, several tiles per
block, a single slice of K, and rows that do not start on 16 bytes (nphi = 3 at 30 atoms: copied
operands). Tolerance of the largest entry: 3e-5 for float32 products (roundoff 6e-8 times ~1000-term
sums, four in a row, with margin) times the condition of the Gram matrix, which the error of a
Gram-Schmidt coefficient carries."""
import numpy as np
import pytest

from oracle import operator as oop, solver as osolver
from paper_1507_08157_gb300 import synthetic as sy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("natoms,nchi,nphi,k", [(28, 4, 4, 1), (33, 4, 4, 2), (16, 9, 4, 1), (15, 9, 4, 3), (30, 9, 3, 2),
                                                (56, 4, 4, 3), (56, 4, 4, 16), (60, 4, 4, 16), (47, 9, 4, 5)])
def test_constant_products_match_oracle(natoms, nchi, nphi, k):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_08157_gb300 import build, tddft
    build.build()
    s = sy.generate(sy.Recipe(natoms=natoms, cell_ang=10.4, ngrid=30, nchi=nchi, nphi=nphi, radius_ang=4.0,
                              min_sep_ang=0.9, seed=500 + natoms))
    Y0 = sy.initial_guess(s, k, 3)
    got = tddft.Context(s, precision="mixed", precond="none").state(Y0).get()["Pp"]
    op = oop.Operator(s)
    P = np.array([op.project(Y) for Y in Y0])
    M = np.array([[op.inner(x, y) for y in P] for x in P])
    ref = np.einsum("ij,jab->iab", osolver.gram_schmidt_coefficients(0.5 * (M + M.T), list(range(k))), P)
    assert np.max(np.abs(got - ref)) <= 3e-5 * np.linalg.cond(M) * np.max(np.abs(ref))
