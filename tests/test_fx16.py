"""The fixed-point 16 x 16 projections (csrc/ve_fx16.cuh): the first-order remainder that ends them
(CPU), and the kernel against numpy through the X step of small block-circulant matrices, at the
spectra and scales where its stopping rules, shortcuts and exponents change (GPU)."""
import numpy as np
import pytest

U = 2.0 ** -53


def _first_order(lam, E):
    s = lam >= 0
    cross = s[:, None] != s[None, :]
    lp = np.where(s[:, None], lam[:, None], lam[None, :])
    lm = np.where(s[:, None], lam[None, :], lam[:, None])
    L = np.where(cross, lp / np.where(cross, lp - lm, 1.0), np.where(s[:, None] & s[None, :], 1.0, 0.0))
    return L * E + np.diag(np.maximum(lam, 0.0)), np.where(cross, E, 0.0)


@pytest.mark.parametrize("clustered", [False, True])
@pytest.mark.parametrize("complex_", [False, True])
def test_remainder_needs_the_two_signs_to_mix(complex_, clustered):
    """||f(Lambda + E) - (f(Lambda) + L o E)|| <= 0.25 ||B|| ||E|| / d for ||E|| <= d / 4, B the part of
    E between diagonal entries of opposite sign, d the diagonal's distance from zero."""
    rng = np.random.default_rng(20210604 + 2 * complex_ + clustered)
    n = 16
    for _ in range(400):
        lam = rng.uniform(0.02, 1.0, n) * 10.0 ** rng.uniform(-2, 0, n)
        if clustered:
            lam = np.repeat(lam[:4], 4)
        lam *= rng.choice([-1.0, 1.0], n)
        d = np.min(np.abs(lam))
        E = rng.normal(size=(n, n)) + (1j * rng.normal(size=(n, n)) if complex_ else 0.0)
        E = 0.5 * (E + E.conj().T)
        np.fill_diagonal(E, 0.0)
        s = lam >= 0
        E = np.where(s[:, None] != s[None, :], E * 10.0 ** rng.uniform(-6, 0), E)
        E *= d * rng.uniform(0.01, 0.25) / np.linalg.norm(E)
        w, V = np.linalg.eigh(np.diag(lam) + E)
        M, B = _first_order(lam, E)
        R = np.linalg.norm((V * np.maximum(w, 0.0)) @ V.conj().T - M)
        assert R <= 0.25 * np.linalg.norm(B) * np.linalg.norm(E) / d + 20 * n * U


def _spectrum(kind, rng):
    lam = rng.normal(size=16)
    if kind == "psd":
        lam = np.abs(lam) + 0.1
    elif kind == "nsd":
        lam = -np.abs(lam) - 0.1
    elif kind == "clustered":
        lam = np.repeat([1.0, 0.25, -0.5, -1.0], 4)
    elif kind == "rank2":
        lam = np.r_[1.0, -1.0, np.zeros(14)]
    elif kind == "near_zero":
        lam = np.r_[1.0, -1.0, 10.0 ** -rng.uniform(3, 15, 14) * rng.choice([-1, 1], 14)]
    elif kind == "graded":
        lam = 10.0 ** -np.arange(16.0) * rng.choice([-1, 1], 16)
    elif kind == "zero":
        lam = np.zeros(16)
    return lam


def _psd(C):
    w, V = np.linalg.eigh(C)
    return (V * np.maximum(w, 0.0)[..., None, :]) @ np.conj(np.swapaxes(V, -1, -2))


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [1.0, 3e-120, 7e90])
@pytest.mark.parametrize("kind", ["random", "psd", "nsd", "clustered", "rank2", "near_zero", "graded", "zero"])
@pytest.mark.parametrize("N", [2, 3, 7])
def test_x_step_matches_numpy(N, kind, scale):
    """Blocks C_k of the given spectrum (real for k = -k, else complex), N not a power of two among
    them.  Both sides' errors are a few n u max|C|: 64 n u covers the DFT, V and both products."""
    torch = pytest.importorskip("torch")
    from paper_2106_02682_gb300 import ve
    rng = np.random.default_rng(N)
    C = np.zeros((N, 16, 16), complex)
    for k in range(N // 2 + 1):
        G = rng.normal(size=(16, 16)) + (0 if 2 * k % N == 0 else 1j) * rng.normal(size=(16, 16))
        Q, _ = np.linalg.qr(G)
        C[k] = scale * (Q * _spectrum(kind, rng)) @ Q.conj().T
        C[k] = 0.5 * (C[k] + C[k].conj().T)
        C[-k % N] = C[k].conj()
    X = np.fft.ifft(C, axis=0).real.copy()
    for precision in (ve.VE_PREC_FP64, ve.VE_PREC_DF64):
        x = torch.from_numpy(X).cuda()
        y = torch.empty_like(x)
        ws = torch.empty(ve.ve_circulant_workspace_size((N,), 16), dtype=torch.uint8, device="cuda")
        ve.ve_circulant_project(x.data_ptr(), y.data_ptr(), (N,), 16, ws.data_ptr(), ws.numel(), precision)
        torch.cuda.synchronize()
        ref = np.fft.ifft(_psd(np.fft.fft(X, axis=0)), axis=0).real
        assert np.max(np.abs(y.cpu().numpy() - ref)) <= 64 * 16 * U * max(np.max(np.abs(C)), 1e-300)


@pytest.mark.gpu
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_blocks_come_back_as_nan(bad):
    torch = pytest.importorskip("torch")
    from paper_2106_02682_gb300 import ve
    X = np.random.default_rng(0).normal(size=(3, 16, 16))
    X[1, 2, 5] = bad
    x = torch.from_numpy(X).cuda()
    ws = torch.empty(ve.ve_circulant_workspace_size((3,), 16), dtype=torch.uint8, device="cuda")
    ve.ve_circulant_project(x.data_ptr(), x.data_ptr(), (3,), 16, ws.data_ptr(), ws.numel())
    torch.cuda.synchronize()
    assert np.all(np.isnan(x.cpu().numpy()))
