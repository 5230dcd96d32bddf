"""The general solver's X step on matrices of up to 16 rows (csrc/ve_fxsign.cu, k_fx_small): one warp
for a matrix that does not fill its 16 x 16 tile, against numpy at the spectra where its rules change."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _spectrum(kind, n, rng):
    if kind == "psd":
        return rng.uniform(0.1, 1.0, n)
    if kind == "nsd":
        return -rng.uniform(0.1, 1.0, n)
    if kind == "rank1":
        return np.r_[-3.0, np.zeros(n - 1)]
    if kind == "near_zero":
        return np.r_[1.0, -1.0, 10.0 ** -rng.uniform(3, 15, n - 2) * rng.choice([-1, 1], n - 2)]
    if kind == "dominant":
        return np.r_[-200.0, rng.uniform(-1.0, 1.0, n - 1)]
    return rng.uniform(-1.0, 1.0, n)


@pytest.mark.parametrize("kind", ["random", "psd", "nsd", "rank1", "near_zero", "dominant", "zero", "nan"])
@pytest.mark.parametrize("spins", [2, 3, 4, 5])
def test_one_sweep(spins, kind):
    """A global step so weak that Y = X; 5 spins (20 rows) take the products."""
    from paper_2106_02682_gb300 import synth, ve
    n = 4 * spins
    rng = np.random.default_rng(spins)
    Q, _ = np.linalg.qr(rng.normal(size=(n, n)))
    lam = np.zeros(n) if kind == "zero" else _spectrum(kind, n, rng)
    X = (Q * lam) @ Q.T
    X = 0.5 * (X + X.T)
    if kind == "nan":
        X[1, 2] = np.nan
    h = ve.ve_general_create(synth.disordered_chain(spins, "xxz", seed=spins), 1, ve.ve_default_options(eps=1e-300))
    try:
        state = ve.ve_general_get_state(h)
        state[-n * n:] = X.ravel()
        ve.ve_general_set_state(h, state)
        try:
            ve.ve_general_iterate(h, 1)
        except ve.VEError:
            assert kind == "nan"
        got = ve.ve_general_get_state(h)[-n * n:].reshape(n, n)
    finally:
        ve.ve_general_destroy(h)
    if kind == "nan":
        assert np.all(np.isnan(got))
        return
    w, V = np.linalg.eigh(X)
    assert np.array_equal(got, got.T)
    # rounding, and Y = X - eps G with |G| <= 1
    assert np.max(np.abs(got - (V * np.maximum(w, 0.0)) @ V.T)) <= 64 * n * U * np.max(np.abs(lam)) + n * 1e-300
