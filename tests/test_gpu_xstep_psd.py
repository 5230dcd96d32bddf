"""The X step leaves X positive semidefinite to the rounding of X itself, however large the negative
eigenvalues are that it removes (eps G has one of the order of the cluster count).  The certificate
charges every unit of -lmin(X) with N m units of energy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.mark.parametrize("sweeps", [1, 15])
@pytest.mark.parametrize("spins,L,kind", [(5, 1, "tfim"), (16, 1, "tfim"), (16, 1, "xxz"), (64, 1, "tfim"), (32, 2, "tfim")])
def test_dense_x_step(spins, L, kind, sweeps):
    from paper_2106_02682_gb300 import synth, ve
    h = ve.ve_general_create(synth.disordered_chain(spins, kind, seed=spins), L)
    try:
        N, _, D, _ = ve.ve_general_dims(h)
        n = N * D
        ve.ve_general_iterate(h, sweeps)
        X = ve.ve_general_get_state(h)[-n * n:].reshape(n, n)
    finally:
        ve.ve_general_destroy(h)
    # entries of Y = X - eps G, eps = 2, |G| <= 1 (marginals): rounding of every entry, n u in the norm
    assert np.linalg.eigvalsh(X).min() >= -n * U * (np.max(np.abs(X)) + 2.0)
