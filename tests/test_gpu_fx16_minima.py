"""The smallest eigenvalues of 16 x 16 blocks in the certificate (csrc/ve_fx16.cuh, lowest): lower bounds
up to rounding, and close, through lmin(X) of ve_bound on states with a chosen X."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _spectrum(kind, rng):
    if kind == "clustered":
        return np.repeat([1.0, 0.25, -0.5, -1.0], 4)
    if kind == "graded":
        return 10.0 ** -np.arange(16.0) * rng.choice([-1, 1], 16)
    if kind == "near_zero":
        return np.r_[1.0, 10.0 ** -rng.uniform(3, 15, 15) * rng.choice([-1, 1], 15)]
    if kind == "equal":
        return np.full(16, 0.7)
    return rng.normal(size=16)


@pytest.mark.parametrize("exponent", [-300, 0, 300])
@pytest.mark.parametrize("kind", ["random", "clustered", "graded", "near_zero", "equal"])
@pytest.mark.parametrize("N", [2, 7])
def test_minima_are_lower_bounds(N, kind, exponent):
    from paper_2106_02682_gb300 import ve
    rng = np.random.default_rng(N)
    C = np.zeros((N, 16, 16), complex)
    for k in range(N // 2 + 1):
        G = rng.normal(size=(16, 16)) + (0 if 2 * k % N == 0 else 1j) * rng.normal(size=(16, 16))
        Q, _ = np.linalg.qr(G)
        C[k] = (Q * _spectrum(kind, rng)) @ Q.conj().T
        C[k] = 0.5 * (C[k] + C[k].conj().T)
        C[-k % N] = C[k].conj()
    X = np.fft.ifft(C, axis=0).real.copy()
    h = ve.ve_create((2 * N,), (2,), ve.ve_ham_tfim(1, 1.0, 1.0), ve.ve_default_options())
    try:
        state = ve.ve_get_state(h)
        state[-X.size:] = np.ldexp(X, exponent).ravel()
        ve.ve_set_state(h, state)
        got = np.ldexp(ve.ve_bound(h).x_min_eig, -exponent)
    finally:
        ve.ve_destroy(h)
    Ck = np.fft.fft(X, axis=0)
    w = np.linalg.eigvalsh(0.5 * (Ck + np.conj(np.swapaxes(Ck, 1, 2))))
    norm = np.max(np.abs(w))
    # rounding of the DFT, of the entries (53 bits of the largest) and of both products, as a norm; the
    # off-diagonal that is taken off is at most n u ||A||_F
    assert w.min() - 8 * 16 * U * norm <= got <= w.min() + 2 * 16 * U * norm
