"""tddft_autotune where a context was made with other kernels than the tuner may choose: a truncated
(sparse) context that was created on the per-tile density kernel has scratch for the density units
which the tuner times and can install, and still matches the truncated oracle afterwards; and for one
state, whose integrals may run on units or on items, both are timed and either can be kept.

Tolerance: 2e-3 of the largest entry, as in the other tests of the float16 grid contractions."""
import numpy as np
import pytest

from oracle import grid as ogrid
from oracle import sparse as osp
from paper_1507_08157_gb300 import synthetic as sy

pytestmark = pytest.mark.gpu

TOL = 2e-3


@pytest.fixture(scope="module")
def tddft():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_08157_gb300 import build, tddft as td
    build.build()
    td.load()
    return td


@pytest.mark.parametrize("var", ["TDDFT_NO_PERSISTENT_DENSITY", "TDDFT_NO_QUAD_GATHER", "TDDFT_NO_DENSITY_UNITS"])
def test_sparse_context_made_without_units_can_be_tuned(tddft, monkeypatch, var):
    monkeypatch.setenv(var, "1")
    s = sy.generate(sy.Recipe(natoms=12, cell_ang=14.0, ngrid=40, nchi=9, radius_ang=3.5, kernel_cutoff_ang=6.0,
                              density_kernel_cutoff_ang=6.0, seed=43))
    ctx = tddft.Context(s, sparse=True, precision="mixed", precond="none")
    rows = [r for r in ctx.autotune(3) if r["stage"] == "response_density"]
    assert {r["kind"] for r in rows} == {"per-tile", "units"}
    P = sy.random_kernels(s, 3, 5)[0]
    op = osp.TruncatedOperator(s)
    rho = ctx.response_density(ctx.to_pattern(P))
    ref = op.response_density(P * op.mask)
    for q in range(3):
        assert np.max(np.abs(rho[q] - ref[q])) <= TOL * np.max(np.abs(ref[q])), q


@pytest.mark.parametrize("ngrid", [40, 108])     # 125 and 2744 tiles: one state on items, on units
def test_one_state_is_tuned_on_both_integrals_kernels(tddft, ngrid):
    s = sy.generate(sy.Recipe(natoms=12, cell_ang=0.35 * ngrid, ngrid=ngrid, nchi=9, radius_ang=3.0, cluster_ang=6.0,
                              seed=45))
    ctx = tddft.Context(s, precision="mixed", precond="none")
    V = np.random.default_rng(4).standard_normal((3, s.n, s.n, s.n))
    ref = ogrid.potential_integrals(ogrid.BoxedSet(s.chi, s.n), ogrid.BoxedSet(s.phi, s.n), V, s.dV)

    def check():
        for k in (1, 3):
            out = ctx.potential_integrals(V[:k])
            for q in range(k):
                assert np.max(np.abs(out[q] - ref[q])) <= TOL * np.max(np.abs(ref[q])), (k, q)

    check()
    rows = [r for r in ctx.autotune(1) if r["stage"] == "potential_integrals"]
    assert {(128, 48), (128, 32)} < {(r["chi_chunk"], r["phi_chunk"]) for r in rows}
    assert {r["chi_chunk"] for r in rows} == {128, 256, 384}
    assert sum(r["chosen"] for r in rows) == 1 and min(rows, key=lambda r: r["ms"])["chosen"]
    check()
    rows = [r for r in ctx.autotune(3) if r["stage"] == "potential_integrals"]
    assert {r["chi_chunk"] for r in rows} == {128}
    check()
