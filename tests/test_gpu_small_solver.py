"""FP64 solver steps against the oracle on both sides of the sizes at which the small-system kernels
give way: the inner CG in one block (up to 20 atoms with 4 functions each, rc rv (rc + rv) = 128000 of
131072; 21 atoms are past it), traces by one warp per pair (kernels of up to 8192 elements; 153 x 68 is
past it), products with edges of 10 to 153 in 16, 32 and 64 wide tiles; one state and an odd number.
The k x k algebra of a step (start, Ritz values, line step, Gram-Schmidt) at block sizes of one to
eight warps: k = 4 to 16, the start and one step; traces of rows past 8192 elements in both pair
tiles and, at an odd length, without 16-byte loads.
Tolerances as derived for the step parity at three atoms: pairs 1e-7 of their scale after each step
(the preconditioner's relative residual 1e-4 multiplies rounding of its own), energies 1e-10."""
import numpy as np
import pytest

from oracle import operator as oop, solver as osolver
from paper_1507_08157_gb300 import synthetic as sy

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


@pytest.mark.parametrize("natoms,nchi,k", [(5, 4, 1), (12, 4, 3), (20, 4, 2), (21, 4, 1), (17, 9, 2)])
def test_small_fp64_solver_steps_match_oracle(natoms, nchi, k):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_08157_gb300 import build, tddft
    build.build()
    s = sy.generate(sy.Recipe(natoms=natoms, cell_ang=9.4, ngrid=30, nchi=nchi, radius_ang=4.0, min_sep_ang=1.0,
                              seed=40 + natoms))
    Y0 = sy.initial_guess(s, k, 3)
    ref = osolver.PCG(oop.Operator(s), Y0)
    st = tddft.Context(s, precision="fp64").state(Y0)
    for _ in range(2):
        om_r, res_r = ref.step()
        om_g, res_g = st.step()
        assert np.max(np.abs(om_g - om_r)) < 1e-10
        assert np.max(np.abs(res_g - res_r) / res_r) < 1e-6
        got = st.get()
        assert _rel(got["Pp"], ref.Pp) < 1e-7 and _rel(got["Pq"], ref.Pq) < 1e-7


@pytest.mark.parametrize("natoms,nchi,nphi,k", [(12, 4, 4, 4), (12, 4, 4, 6), (12, 4, 4, 7), (12, 4, 4, 10), (12, 4, 4, 11),
                                                (12, 4, 4, 16), (17, 9, 4, 5), (17, 9, 4, 11), (17, 9, 4, 16), (19, 9, 3, 3)])
def test_small_algebra_matches_oracle_for_every_block_size(natoms, nchi, nphi, k):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_08157_gb300 import build, tddft
    build.build()
    s = sy.generate(sy.Recipe(natoms=natoms, cell_ang=9.4, ngrid=30, nchi=nchi, nphi=nphi, radius_ang=4.0,
                              min_sep_ang=1.0, seed=40 + natoms))
    Y0 = sy.initial_guess(s, k, 3)
    ref = osolver.PCG(oop.Operator(s), Y0)
    st = tddft.Context(s, precision="fp64").state(Y0)
    got = st.get()
    assert _rel(got["Pp"], ref.Pp) < 1e-9 and _rel(got["Pq"], ref.Pq) < 1e-9
    om_r, res_r = ref.step()
    om_g, res_g = st.step()
    assert np.max(np.abs(om_g - om_r)) < 1e-10
    assert np.max(np.abs(res_g - res_r) / res_r) < 1e-6
    got = st.get()
    assert _rel(got["Pp"], ref.Pp) < 1e-7 and _rel(got["Pq"], ref.Pq) < 1e-7
