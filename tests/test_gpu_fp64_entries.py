"""The float64 grid contractions entry by entry: every grid point of the response density keeps the
accuracy of a float64 sum of its own terms, whatever the sizes of other points, functions and blocks of
P, and a NaN or infinity spoils the tiles it reaches and nothing else.

Density tolerance: a float64 sum of at most N_chi products per phi and N_phi phi has an error of at most
(N_chi + N_phi) 2^-53 of the sum of its terms' sizes, the reference and the library one each."""
import dataclasses

import numpy as np
import pytest

from oracle import grid as ogrid
from paper_1507_08157_gb300 import synthetic as sy

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tddft():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_08157_gb300 import build, tddft as td
    build.build()
    td.load()
    return td


def _sets(s):
    sizes = [dataclasses.replace(f, val=np.abs(f.val)) for f in (s.chi, s.phi)]
    return [ogrid.BoxedSet(f, s.n) for f in (s.chi, s.phi, *sizes)]


def _kernels(s, kind):
    P = sy.random_kernels(s, 2, 11)[0]
    rng = np.random.default_rng(5)
    na, nc, nv = s.natoms, P.shape[1] // s.natoms, P.shape[2] // s.natoms
    block = 10.0 ** -np.array([0, 6, 12])[np.arange(na) % 3]
    if kind == "rows":
        P *= np.repeat(block, nc)[:, None]
    elif kind == "columns":
        P *= np.repeat(block, nv)[None, :]
    elif kind == "both":
        P *= np.repeat(block, nc)[:, None] * np.repeat(block, nv)[None, :]
    elif kind == "spread":
        P *= 10.0 ** rng.uniform(-12, 0, P.shape)
    elif kind == "wide":             # scales too far apart for one tile's columns
        P *= np.repeat(10.0 ** -np.array([0, 290])[np.arange(na) % 2], nv)[None, :]
    elif kind == "zeros":
        P[:, : nc] = 0.0
        P[:, :, 1] = 0.0
        P[1] = 0.0
    return P


@pytest.mark.parametrize("radius", [2.5, 6.0])
@pytest.mark.parametrize("kind", ["plain", "rows", "columns", "both", "spread", "wide", "zeros"])
def test_density_keeps_float64_accuracy_at_every_point(tddft, kind, radius):
    s = sy.generate(sy.Recipe(natoms=9, cell_ang=14.0, ngrid=45, nchi=9, radius_ang=radius, seed=57))
    chi, phi, achi, aphi = _sets(s)
    P = _kernels(s, kind)
    rho = tddft.Context(s, precision="fp64", precond="none").response_density(P)
    ref, size = ogrid.response_density(chi, phi, P), ogrid.response_density(achi, aphi, np.abs(P))
    tol = 2 * (P.shape[1] + P.shape[2]) * 2.0 ** -53
    assert np.all(np.abs(rho - ref) <= tol * size + 1e-300)


def _tiles_of(s, fs, f):
    """Tiles that the box of function f reaches, [nt, nt, nt]."""
    nt = -(-s.n // 8)
    on = []
    for ax in range(3):
        m = np.zeros(nt, dtype=bool)
        m[((fs.box[f, ax] + np.arange(fs.box[f, 3 + ax])) % s.n) // 8] = True
        on.append(m)
    return on[0][:, None, None] & on[1][None, :, None] & on[2][None, None, :]


def _points(s, tiles):
    return np.repeat(np.repeat(np.repeat(tiles, 8, 0), 8, 1), 8, 2)[: s.n, : s.n, : s.n]


@pytest.fixture(scope="module")
def spread9():
    return sy.generate(sy.Recipe(natoms=9, cell_ang=14.0, ngrid=45, nchi=9, radius_ang=2.0, seed=57))


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed", 2e-3)])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_density_of_a_bad_kernel_entry_is_bad_where_it_reaches(tddft, spread9, bad, precision, tol):
    s = spread9
    chi, phi, _, _ = _sets(s)
    P = sy.random_kernels(s, 3, 12)[0]
    a, b = 13, 5
    P[:, a, b] = 0.0
    ref = ogrid.response_density(chi, phi, P)
    P[1, a, b] = bad
    rho = tddft.Context(s, precision=precision, precond="none").response_density(P)
    reach = _points(s, _tiles_of(s, s.chi, a) & _tiles_of(s, s.phi, b))
    assert 0 < reach.sum() < reach.size
    hit = np.abs(ogrid.full_grid(s.chi, s.n)[a] * ogrid.full_grid(s.phi, s.n)[b]) > 0.0
    assert not np.any(np.isfinite(rho[1][hit])) and np.all(reach[hit])
    for q in range(3):
        keep = ~reach if q == 1 else np.ones_like(reach)
        assert np.max(np.abs(rho[q] - ref[q])[keep]) <= tol * np.max(np.abs(ref[q])), q


def _potentials(s, kind):
    rng = np.random.default_rng(6)
    V = rng.standard_normal((2, s.n, s.n, s.n))
    if kind == "peak":
        V[0, s.n // 2, s.n // 2, s.n // 2] = 1e12
        V[1, 3, 4, 5] = -1e30
    elif kind == "gaussian":
        x = (np.arange(s.n) - s.n / 2) * s.h
        V[:] = np.exp(-0.25 * sum(np.meshgrid(x ** 2, x ** 2, x ** 2, indexing="ij")))
    elif kind == "spread":
        V *= 10.0 ** rng.uniform(-12, 0, V.shape)
    elif kind == "zeros":
        V[0, : s.n // 2] = 0.0
        V[1] = 0.0
    return V


def _tile_scales(s, V):
    """Sum over tiles of max |chi_a| max |V phi_b|, [a, b]."""
    nt = -(-s.n // 8)

    def tops(full):
        pad = np.zeros((full.shape[0],) + (nt * 8,) * 3)
        pad[:, : s.n, : s.n, : s.n] = np.abs(full)
        return pad.reshape(-1, nt, 8, nt, 8, nt, 8).max(axis=(2, 4, 6)).reshape(full.shape[0], -1)

    return tops(ogrid.full_grid(s.chi, s.n)) @ tops(ogrid.full_grid(s.phi, s.n) * V).T


@pytest.mark.parametrize("radius", [2.5, 6.0])
@pytest.mark.parametrize("kind", ["plain", "peak", "gaussian", "spread", "zeros"])
def test_integrals_keep_their_tiles_accuracy(tddft, kind, radius):
    """Bound per entry: 2^-47 of the tiles' scales (per product 2^-60 for the digit products left out and
    2^-62 for the digits' rounding, of scales at most 8 times the largest values, 512 of them) and, of the
    sum of the terms' sizes, the rounding of float64 sums of at most 45^3 terms added in quadrature,
    8 sqrt(45^3) 2^-53 < 1e-12."""
    s = sy.generate(sy.Recipe(natoms=9, cell_ang=14.0, ngrid=45, nchi=9, radius_ang=radius, seed=57))
    chi, phi, achi, aphi = _sets(s)
    V = _potentials(s, kind)
    out = tddft.Context(s, precision="fp64", precond="none").potential_integrals(V)
    ref = ogrid.potential_integrals(chi, phi, V, s.dV)
    size = ogrid.potential_integrals(achi, aphi, np.abs(V), s.dV)
    for q in range(2):
        assert np.all(np.abs(out[q] - ref[q]) <= 2.0 ** -47 * s.dV * _tile_scales(s, V[q]) + 1e-12 * size[q] + 1e-300), q
        assert np.max(np.abs(out[q] - ref[q])) <= 1e-13 * np.max(size[q]), q


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed", 2e-3)])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_integrals_of_a_bad_potential_are_bad_where_it_reaches(tddft, spread9, bad, precision, tol):
    s = spread9
    chi, phi, _, _ = _sets(s)
    V = np.random.default_rng(8).standard_normal((3, s.n, s.n, s.n))
    ref = ogrid.potential_integrals(chi, phi, V, s.dV)
    i = 9
    p = tuple((s.phi.box[i, :3] + s.phi.box[i, 3:] // 2) % s.n)     # the centre of an atom's functions
    V[1][p] = bad
    out = tddft.Context(s, precision=precision, precond="none").potential_integrals(V)
    t = tuple(x // 8 for x in p)
    reach = np.outer(*[[_tiles_of(s, f, j)[t] for j in range(f.nfun)] for f in (s.chi, s.phi)])
    assert 0 < reach.sum() < reach.size
    hit = np.outer(np.abs(ogrid.values_at(chi, p)) > 0, np.abs(ogrid.values_at(phi, p)) > 0)
    assert hit.any() and not np.any(np.isfinite(out[1][hit])) and np.all(reach[hit])
    for q in range(3):
        keep = ~reach if q == 1 else np.ones_like(reach)
        assert np.max(np.abs(out[q] - ref[q])[keep]) <= tol * np.max(np.abs(ref[q])), q
