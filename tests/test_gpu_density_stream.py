"""The response density of one state on dense tiles (chi streamed in units of at most 320 chi and 128 phi)
at the edges of its units, against the FP64 oracle: chi lists on both sides of 320 and in two units, phi
lists on both sides of 256; lists short enough for the per-tile kernel, which keep the items; the tuner's choice between it and the density items, for one state and
for several. Small cells in which every function touches most tiles, ragged 30^3 grid. float16 operands
with float32 accumulation: 2e-3 of the largest entry, as in the other tensor-core density tests."""
import numpy as np
import pytest

from oracle import operator as oop
from paper_1507_08157_gb300 import synthetic as sy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("natoms,nchi", [(66, 4), (80, 4), (81, 4), (96, 4), (97, 4), (71, 9), (72, 9)])
def test_single_state_density_at_unit_edges(natoms, nchi):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_08157_gb300 import build, tddft
    build.build()
    s = sy.generate(sy.Recipe(natoms=natoms, cell_ang=9.4, ngrid=30, nchi=nchi, radius_ang=4.0, min_sep_ang=0.8,
                              seed=500 + natoms))
    ctx = tddft.Context(s, precision="mixed", precond="none")
    P = sy.random_kernels(s, 2, 7)[1]
    ref = oop.Operator(s).response_density(P)

    def check():
        for k in (1, 2):
            rho = ctx.response_density(P[:k])
            for q in range(k):
                assert np.max(np.abs(rho[q] - ref[q])) <= 2e-3 * np.max(np.abs(ref[q])), (k, q)

    check()
    rows = [r for r in ctx.autotune(1) if r["stage"] == "response_density"]
    short = any(r["kind"] == "per-tile" for r in rows)
    assert {r["chi_chunk"] for r in rows} == ({0, 128, 256} if short else {128, 256, 320})
    assert short == (natoms == 66) and sum(r["chosen"] for r in rows) == 1
    check()
