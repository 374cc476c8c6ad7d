"""The tensor-core potential integrals at the edges of their items, against the FP64 oracle: chi lists on
both sides of 128, phi lists on both sides of 48 and 96, one state, odd and even counts, states of
different scales in one pair, and phi lists that are no whole quads (the kernel for other lists).
Small cells in which every function touches most tiles, on a 30^3 grid (tiles of 8 leave a ragged
tail of 6). float16 operands with float32 accumulation: 2e-3 of the largest entry, as in the other
tensor-core integrals tests."""
import numpy as np
import pytest

from oracle import grid as ogrid
from paper_1507_08157_gb300 import synthetic as sy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("natoms,nchi,nphi,k", [(12, 9, 4, 1), (13, 9, 4, 2), (14, 9, 4, 3), (15, 9, 4, 5), (24, 4, 4, 4),
                                                (25, 4, 4, 1), (33, 4, 4, 3), (9, 4, 1, 2)])
def test_integrals_match_oracle_at_list_edges(natoms, nchi, nphi, k):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_08157_gb300 import build, tddft
    build.build()
    s = sy.generate(sy.Recipe(natoms=natoms, cell_ang=9.4, ngrid=30, nchi=nchi, nphi=nphi, radius_ang=4.0,
                              min_sep_ang=1.0, seed=200 + natoms))
    ctx = tddft.Context(s, precision="mixed", precond="none")
    V = np.random.default_rng(natoms).standard_normal((k, s.n, s.n, s.n))
    V[-1] *= 1e-3
    got = ctx.potential_integrals(V)
    ref = ogrid.potential_integrals(ogrid.BoxedSet(s.chi, s.n), ogrid.BoxedSet(s.phi, s.n), V, s.dV)
    for q in range(k):
        assert np.max(np.abs(got[q] - ref[q])) <= 2e-3 * np.max(np.abs(ref[q])), q


@pytest.mark.parametrize("ngrid,k", [(96, 1), (108, 1), (108, 2)])
def test_single_state_on_few_and_many_tiles(ngrid, k):
    # one state takes the kernel by units from 2049 tiles on (13^3 at 108), the item kernel below
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_08157_gb300 import build, tddft
    build.build()
    s = sy.generate(sy.Recipe(natoms=10, cell_ang=ngrid / 4.0, ngrid=ngrid, nchi=9, radius_ang=3.0, min_sep_ang=1.0, seed=3))
    ctx = tddft.Context(s, precision="mixed", precond="none")
    V = np.random.default_rng(k).standard_normal((k, s.n, s.n, s.n))
    got = ctx.potential_integrals(V)
    ref = ogrid.potential_integrals(ogrid.BoxedSet(s.chi, s.n), ogrid.BoxedSet(s.phi, s.n), V, s.dV)
    assert np.max(np.abs(got - ref)) <= 2e-3 * np.max(np.abs(ref))
