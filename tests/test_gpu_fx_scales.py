"""The fixed-point projections (csrc/ve_fx16.cuh, ve_fx64.cuh, ve_fxsign.cu) on matrices so large or
so small that squares of their entries overflow or vanish, or that results are subnormal.  A power
of two as the scale changes nothing but exponents, so the reference is that of the unscaled matrix."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U = 2.0 ** -53
SCALES = [-1018, -560, 530, 1000]


def _psd(C):
    w, V = np.linalg.eigh(C)
    return (V * np.maximum(w, 0.0)[..., None, :]) @ np.conj(np.swapaxes(V, -1, -2))


def _x_step(ve, X, M, D, precision):
    import torch
    x = torch.from_numpy(X).cuda()
    ws = torch.empty(ve.ve_circulant_workspace_size(M, D), dtype=torch.uint8, device="cuda")
    ve.ve_circulant_project(x.data_ptr(), x.data_ptr(), M, D, ws.data_ptr(), ws.numel(), precision)
    torch.cuda.synchronize()
    return x.cpu().numpy()


def _block_row(N, D, seed):
    """First block row whose blocks C_k (norm below 1) have eigenvalues of both signs."""
    rng = np.random.default_rng(seed)
    C = np.zeros((N, D, D), complex)
    for k in range(N // 2 + 1):
        G = rng.normal(size=(D, D)) + (0 if 2 * k % N == 0 else 1j) * rng.normal(size=(D, D))
        Q, _ = np.linalg.qr(G)
        C[k] = (Q * rng.uniform(-1.0, 1.0, D)) @ Q.conj().T
        C[k] = 0.5 * (C[k] + C[k].conj().T)
        C[-k % N] = C[k].conj()
    return np.fft.ifft(C, axis=0).real.copy()


def _check_x_step(D, exponent):
    from paper_2106_02682_gb300 import ve
    X = _block_row(5, D, D)
    ref = np.fft.ifft(_psd(np.fft.fft(X, axis=0)), axis=0).real
    for precision in (ve.VE_PREC_FP64, ve.VE_PREC_DF64):
        got = np.ldexp(_x_step(ve, np.ldexp(X, exponent), (5,), D, precision), -exponent)
        # 64 n u covers the DFT, the eigenvectors or the sign, the products and the subnormal spacing
        # (2^-1074: u / 8 at the smallest scale)
        assert np.max(np.abs(got - ref)) <= 64 * D * U


@pytest.mark.parametrize("exponent", SCALES)
def test_x_step_16(exponent):
    _check_x_step(16, exponent)


@pytest.mark.parametrize("exponent", SCALES)
def test_x_step_64(exponent):
    _check_x_step(64, exponent)


@pytest.mark.parametrize("exponent", [-1018, -560, 530])
@pytest.mark.parametrize("spins", [5, 26])
def test_dense_x_step(spins, exponent):
    """One sweep of the general solver, its global step so weak that Y = X to rounding."""
    from paper_2106_02682_gb300 import synth, ve
    n = 4 * spins
    rng = np.random.default_rng(spins)
    Q, _ = np.linalg.qr(rng.normal(size=(n, n)))
    X = (Q * rng.uniform(-1.0, 1.0, n)) @ Q.T
    X = 0.5 * (X + X.T)
    h = ve.ve_general_create(synth.disordered_chain(spins, "xxz", seed=spins), 1, ve.ve_default_options(eps=1e-323))
    try:
        state = ve.ve_general_get_state(h)
        state[-n * n:] = np.ldexp(X, exponent).ravel()
        ve.ve_general_set_state(h, state)
        try:
            ve.ve_general_iterate(h, 1)
        except ve.VEError:
            assert exponent > 500  # the feasibility error is a sum of squares
        got = np.ldexp(ve.ve_general_get_state(h)[-n * n:].reshape(n, n), -exponent)
    finally:
        ve.ve_general_destroy(h)
    assert np.max(np.abs(got - _psd(X))) <= 64 * n * U
