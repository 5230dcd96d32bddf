"""The general solver's X step (csrc/ve_fxsign.cu) to float64 accuracy, and bit for bit from run to run
(its launches overlap): sizes that do not fill 16 x 16 blocks or 32 x 32 tiles, spectra with a dominant
eigenvalue, eigenvalues far below the first pass's range, exact zeros."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _spectrum(kind, n, rng):
    if kind == "dominant":
        return np.r_[1e4, rng.normal(size=n - 1)]
    if kind == "tiny":       # below 3e-6 and 1e-11 of the norm
        k = n // 4
        return np.r_[rng.normal(size=n - 2 * k), 1e-7 * rng.normal(size=k), 1e-12 * rng.normal(size=k)]
    if kind == "rank1":
        return np.r_[-3.0, np.zeros(n - 1)]
    return np.repeat([1.0, -1.0], n // 2)[:n]


@pytest.mark.parametrize("kind", ["dominant", "tiny", "rank1", "signs"])
@pytest.mark.parametrize("spins,L", [(2, 1), (5, 1), (9, 3), (52, 1), (58, 2)])
def test_float64_accuracy_and_reproducibility(spins, L, kind):
    from paper_2106_02682_gb300 import synth, ve
    terms = synth.disordered_chain(spins, "xxz", seed=spins)
    # so weak a global step that Y = X to rounding
    handles = [ve.ve_general_create(terms, L, ve.ve_default_options(eps=1e-300)) for _ in range(2)]
    try:
        N, _, D, _ = ve.ve_general_dims(handles[0])
        n = N * D
        rng = np.random.default_rng(n)
        Q, _ = np.linalg.qr(rng.normal(size=(n, n)))
        lam = _spectrum(kind, n, rng)
        X = (Q * lam) @ Q.T
        X = 0.5 * (X + X.T)
        state = ve.ve_general_get_state(handles[0])
        state[-n * n:] = X.ravel()
        out = []
        for h in handles:
            for _ in range(2):  # again on the same handle, and on a fresh one
                ve.ve_general_set_state(h, state)
                ve.ve_general_iterate(h, 1)
                out.append(ve.ve_general_get_state(h)[-n * n:].reshape(n, n))
    finally:
        for h in handles:
            ve.ve_general_destroy(h)
    w, V = np.linalg.eigh(X)
    norm = np.max(np.abs(lam))
    assert np.max(np.abs(out[0] - (V * np.maximum(w, 0.0)) @ V.T)) <= 64 * n * U * norm
    # no eigenvalue is left behind, the smallest included: rounding of the entries
    assert np.linalg.eigvalsh(out[0]).min() >= -4 * n * U * np.max(np.abs(X))
    for other in out[1:]:
        assert np.array_equal(out[0], other)
