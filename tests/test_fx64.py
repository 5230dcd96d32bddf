"""The fixed-point 64 x 64 projections (csrc/ve_fx64.cuh) against numpy through the X step of small
block-circulant matrices: spectra at the ends of the sign iteration's range, and scales."""
import numpy as np
import pytest

U = 2.0 ** -53


def _spectrum(kind, rng):
    n = 64
    lam = rng.normal(size=n)
    if kind == "psd":
        lam = np.abs(lam) + 0.1
    elif kind == "clustered":
        lam = np.repeat([1.0, 0.25, -0.5, -1.0], n // 4)
    elif kind == "rank2":
        lam = np.r_[1.0, -1.0, np.zeros(n - 2)]
    elif kind == "near_zero":
        lam = np.r_[1.0, -1.0, 10.0 ** -rng.uniform(3, 15, n - 2) * rng.choice([-1, 1], n - 2)]
    elif kind == "zero":
        lam = np.zeros(n)
    return lam


def _psd(C):
    w, V = np.linalg.eigh(C)
    return (V * np.maximum(w, 0.0)[..., None, :]) @ np.conj(np.swapaxes(V, -1, -2))


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [1.0, 3e-120, 7e90])
@pytest.mark.parametrize("kind", ["random", "psd", "clustered", "rank2", "near_zero", "zero"])
@pytest.mark.parametrize("N", [2, 5])
def test_x_step_matches_numpy(N, kind, scale):
    """Real blocks at k = -k, complex ones elsewhere.  Both sides' errors are a few n u max|C|."""
    torch = pytest.importorskip("torch")
    from paper_2106_02682_gb300 import ve
    rng = np.random.default_rng(64 + N)
    C = np.zeros((N, 64, 64), complex)
    for k in range(N // 2 + 1):
        G = rng.normal(size=(64, 64)) + (0 if 2 * k % N == 0 else 1j) * rng.normal(size=(64, 64))
        Q, _ = np.linalg.qr(G)
        C[k] = scale * (Q * _spectrum(kind, rng)) @ Q.conj().T
        C[k] = 0.5 * (C[k] + C[k].conj().T)
        C[-k % N] = C[k].conj()
    X = np.fft.ifft(C, axis=0).real.copy()
    ref = np.fft.ifft(_psd(np.fft.fft(X, axis=0)), axis=0).real
    for precision in (ve.VE_PREC_FP64, ve.VE_PREC_DF64):
        x = torch.from_numpy(X).cuda()
        ws = torch.empty(ve.ve_circulant_workspace_size((N,), 64), dtype=torch.uint8, device="cuda")
        ve.ve_circulant_project(x.data_ptr(), x.data_ptr(), (N,), 64, ws.data_ptr(), ws.numel(), precision)
        torch.cuda.synchronize()
        # eigenvalues of 64 x 64 blocks of norm s: |C| <= s; 64 n u covers the DFT and the products
        assert np.max(np.abs(x.cpu().numpy() - ref)) <= 64 * 64 * U * max(scale, 1e-300)


@pytest.mark.gpu
def test_non_finite_blocks_come_back_as_nan():
    torch = pytest.importorskip("torch")
    from paper_2106_02682_gb300 import ve
    X = np.random.default_rng(0).normal(size=(3, 64, 64))
    X[1, 2, 5] = np.nan
    x = torch.from_numpy(X).cuda()
    ws = torch.empty(ve.ve_circulant_workspace_size((3,), 64), dtype=torch.uint8, device="cuda")
    ve.ve_circulant_project(x.data_ptr(), x.data_ptr(), (3,), 64, ws.data_ptr(), ws.numel())
    torch.cuda.synchronize()
    assert np.all(np.isnan(x.cpu().numpy()))
