"""lmin(X) in the general solver's certificate: zero to rounding after an X step (csrc/ve_fxsign.cu,
fxsign_lmin), by an eigensolve for any other X; against numpy on the same X."""
import time

import numpy as np
import pytest

from paper_2106_02682_gb300 import synth

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _x(ve, h):
    N, _, D, _ = ve.ve_general_dims(h)
    n = N * D
    return ve.ve_general_get_state(h)[-n * n:].reshape(n, n)


@pytest.mark.parametrize("spins,L,kind", [(2, 1, "tfim"), (3, 1, "xxz"), (4, 1, "tfim"), (5, 1, "tfim"), (16, 1, "xxz"),
                                          (64, 1, "tfim"), (20, 2, "tfim"), (9, 3, "xxz")])
def test_after_sweeps(spins, L, kind):
    from paper_2106_02682_gb300 import ve
    h = ve.ve_general_create(synth.disordered_chain(spins, kind, seed=spins), L)
    try:
        for sweeps in (1, 14):
            ve.ve_general_iterate(h, sweeps)
            c = ve.ve_general_bound(h)
            X = _x(ve, h)
            w = np.linalg.eigvalsh(X)
            n = len(w)
            # a lower bound to rounding, as close as an eigensolve that stops at n u ||X||
            assert w[0] - n * U * w[-1] <= c.x_min_eig <= w[0] + 8 * U * w[-1]
            assert c.x_neg_correction == ve.ve_general_dims(h)[0] * ve.ve_general_dims(h)[1] * max(0.0, -c.x_min_eig)
    finally:
        ve.ve_general_destroy(h)


@pytest.mark.parametrize("spins", [3, 5, 16, 40])
@pytest.mark.parametrize("low", [0.3, 1e-7, 1e-11, 0.0, -1e-9, -0.2])
def test_any_x(spins, low):
    """X set with a given smallest eigenvalue: definite, nearly singular, singular, indefinite."""
    from paper_2106_02682_gb300 import ve
    n = 4 * spins
    rng = np.random.default_rng(spins)
    Q, _ = np.linalg.qr(rng.normal(size=(n, n)))
    X = (Q * np.r_[low, low + rng.uniform(0.5, 2.0, n - 1)]) @ Q.T
    X = 0.5 * (X + X.T)
    h = ve.ve_general_create(synth.disordered_chain(spins, "tfim", seed=spins), 1)
    try:
        ve.ve_general_iterate(h, 2)
        state = ve.ve_general_get_state(h)
        state[-n * n:] = X.ravel()
        ve.ve_general_set_state(h, state)
        c = ve.ve_general_bound(h)
    finally:
        ve.ve_general_destroy(h)
    w = np.linalg.eigvalsh(X)
    # the eigensolve's stop (n u ||X||_F) and its rounding
    assert abs(c.x_min_eig - w[0]) <= 4 * n * U * np.linalg.norm(X)


def test_first_bound_is_not_a_cold_eigensolve():
    """128 spins, X of 512 x 512: a cold eigensolve takes 40 to 80 ms, the bound about 1 ms."""
    from paper_2106_02682_gb300 import ve
    terms = synth.disordered_chain(128, "tfim", seed=1)
    times = []
    for _ in range(3):
        h = ve.ve_general_create(terms, 1)
        try:
            ve.ve_general_iterate(h, 20)
            t = time.perf_counter()
            ve.ve_general_bound(h)
            times.append(time.perf_counter() - t)
        finally:
            ve.ve_general_destroy(h)
    assert min(times) < 0.015
