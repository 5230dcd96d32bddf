"""The general solver's X step (csrc/ve_fxsign.cu) where its iteration can go wrong: sizes that do
not fill 16 x 16 blocks or 32 x 32 tiles, a dominant eigenvalue, eigenvalues far below the first
pass's range, exact zeros and extreme scales.  One sweep from a state with a chosen X against the
oracle's eigendecomposition."""
import numpy as np
import pytest

from oracle import alg5
from oracle import models as mo
from paper_2106_02682_gb300 import synth

pytestmark = pytest.mark.gpu


def _x(kind, n, rng):
    Q, _ = np.linalg.qr(rng.normal(size=(n, n)))
    if kind == "dominant":
        lam = np.r_[1e4, rng.normal(size=n - 1)]
    elif kind == "tiny":       # below 3e-6 and 1e-11 of the norm
        lam = np.r_[rng.normal(size=n // 2), 1e-7 * rng.normal(size=n // 4), 1e-12 * rng.normal(size=n - n // 2 - n // 4)]
    elif kind == "rank1":
        lam = np.r_[-3.0, np.zeros(n - 1)]
    elif kind == "large":
        lam = 1e60 * rng.normal(size=n)
    else:
        lam = np.repeat([1.0, -1.0], n // 2)[:n]
    X = (Q * lam) @ Q.T
    return 0.5 * (X + X.T)


@pytest.mark.parametrize("kind", ["dominant", "tiny", "rank1", "large", "signs"])
@pytest.mark.parametrize("spins,L", [(2, 1), (5, 1), (9, 3), (52, 1), (58, 2)])
def test_one_sweep_matches_the_oracle(spins, L, kind):
    from paper_2106_02682_gb300 import ve
    terms = synth.disordered_chain(spins, "xxz", seed=spins)
    bonds = [(int(s), int(t), B) for (s, t), B in zip(terms['bond_sites'], terms['bond_ops'])]
    blocks = mo.general_blocks(spins, L, terms['onsite'], bonds)
    # a weak global step leaves Y = X - eps G with X's spectrum
    eps = 1e-14
    pb, s5 = alg5.GeneralProblem(blocks, eps=eps), alg5.general_setup(blocks)
    st = alg5.initial_state(pb, s5)
    n = pb.N * pb.D
    st['X'] = _x(kind, n, np.random.default_rng(n))
    scale = np.max(np.abs(st['X']))
    h = ve.ve_general_create(terms, L, ve.ve_default_options(eps=eps))
    try:
        ve.ve_general_set_state(h, alg5.pack_state(pb, s5, st))
        ve.ve_general_iterate(h, 1)
        got = ve.ve_general_get_state(h)[-n * n:].reshape(n, n)
        again = ve.ve_general_get_state(h)
    finally:
        ve.ve_general_destroy(h)
    alg5.iterate(pb, s5, st)
    # both backward errors grow like n u ||Y||; 1e-10 is the solver's bar at n = 64
    assert np.max(np.abs(got - st['X'])) <= 1e-10 * max(1.0, n / 64) * scale
    assert np.array_equal(got, got.T)
    assert np.array_equal(again[-n * n:].reshape(n, n), got)


def test_bound_after_a_bound_of_a_nonfinite_state():
    """The bound's eigensolve of X starts from the last bound's eigenvectors, but not from those of a
    state that was not finite."""
    from paper_2106_02682_gb300 import ve
    terms = synth.disordered_chain(6, "tfim", seed=3)
    h = ve.ve_general_create(terms, 1, ve.ve_default_options())
    try:
        ve.ve_general_iterate(h, 5)
        good = ve.ve_general_get_state(h)
        want = ve.ve_general_bound(h).bound_per_spin
        bad = good.copy()
        bad[-1] = np.nan  # an entry of X
        ve.ve_general_set_state(h, bad)
        with pytest.raises(ve.VEError):
            ve.ve_general_bound(h)
        ve.ve_general_set_state(h, good)
        got = ve.ve_general_bound(h)
    finally:
        ve.ve_general_destroy(h)
    # the pair and cluster minima do not depend on X; its own enters with N m max(0, -lmin(X))
    assert abs(got.bound_per_spin - want) <= 1e-11
