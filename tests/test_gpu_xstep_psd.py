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


@pytest.mark.parametrize("D", [16, 64])
@pytest.mark.parametrize("N", [2, 5])
def test_wavevector_blocks(N, D):
    """Blocks with one eigenvalue of -200, along a vector spread over the entries, the others in [-1, 1]."""
    import torch
    from paper_2106_02682_gb300 import ve
    rng = np.random.default_rng(N + D)
    C = np.zeros((N, D, D), complex)
    for k in range(N // 2 + 1):
        G = rng.normal(size=(D, D)) + (0 if 2 * k % N == 0 else 1j) * rng.normal(size=(D, D))
        G[:, 0] /= np.abs(G[:, 0])
        Q, _ = np.linalg.qr(G)
        C[k] = (Q * np.r_[-200.0, rng.uniform(-1.0, 1.0, D - 1)]) @ Q.conj().T
        C[k] = 0.5 * (C[k] + C[k].conj().T)
        C[-k % N] = C[k].conj()
    X = np.fft.ifft(C, axis=0).real.copy()
    x = torch.from_numpy(X).cuda()
    ws = torch.empty(ve.ve_circulant_workspace_size((N,), D), dtype=torch.uint8, device="cuda")
    ve.ve_circulant_project(x.data_ptr(), x.data_ptr(), (N,), D, ws.data_ptr(), ws.numel())
    torch.cuda.synchronize()
    Y = np.fft.fft(x.cpu().numpy(), axis=0)
    low = np.linalg.eigvalsh(0.5 * (Y + np.conj(np.swapaxes(Y, 1, 2)))).min()
    # rounding of every entry of C_k (the projection), and of the result (both transforms)
    assert low >= -D * U * (np.max(np.abs(C)) + 4.0)
