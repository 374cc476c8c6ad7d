"""Solver states on memory that a destroyed state gave back: the results of fresh memory, with larger and
smaller states in between, with two states alive at once (one of them on memory of its own), and a state
that outlives every Python reference to its context. FP64; the potential integrals add tiles in
any order, so that runs agree to the bound of the step parity: energies 1e-10, pairs 1e-7 of scale."""
import numpy as np
import pytest

from paper_1507_08157_gb300 import synthetic as sy

pytestmark = pytest.mark.gpu


def test_states_on_reused_memory_match_fresh_ones():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1507_08157_gb300 import build, tddft
    build.build()
    s = sy.generate(sy.Recipe(natoms=6, cell_ang=9.4, ngrid=30, nchi=4, radius_ang=4.0, min_sep_ang=1.0, seed=46))
    guess = {k: sy.initial_guess(s, k, 3) for k in (1, 2, 5)}

    def run(st):
        om = [st.step()[0] for _ in range(2)]
        got = st.get()
        return om, [got["Pp"], got["fq"]]

    def same(a, b):
        assert np.max(np.abs(np.array(a[0]) - np.array(b[0]))) < 1e-10
        for x, y in zip(a[1], b[1]):
            assert np.max(np.abs(x - y)) < 1e-7 * np.max(np.abs(y))

    fresh = {k: run(tddft.Context(s, precision="fp64").state(guess[k])) for k in guess}
    ctx = tddft.Context(s, precision="fp64")
    for k in (2, 5, 2, 1, 1, 5):
        st = ctx.state(guess[k])
        same(run(st), fresh[k])
        del st
    one = ctx.state(guess[2])
    two = ctx.state(guess[2])
    del ctx
    same(run(one), fresh[2])
    same(run(two), fresh[2])
