"""The first-order reconstruction of the 16 x 16 fixed-point projections (csrc/ve_fx16.cuh): the
entries between eigenvalues of opposite sign, to float64 accuracy.  Direct sums of 2 x 2 blocks
[[a, e], [e, -b]] have the closed form f = (A + |A|) / 2, |A| = (A^2 + (a b + e^2) I) / (2 R),
R = sqrt(((a + b) / 2)^2 + e^2); with e inside the first-order rule the projection reconstructs from
V = I at once, and the off-diagonal entry is e times the divided difference."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.mark.parametrize("complex_", [False, True])
@pytest.mark.parametrize("seed", range(8))
def test_entries_between_the_signs(seed, complex_):
    import torch
    from paper_2106_02682_gb300 import ve
    D, N = 16, 4
    rng = np.random.default_rng(seed)
    C, want = np.zeros((N, D, D), complex), np.zeros((N, D, D), complex)
    for k in range(N // 2 + 1):
        a, b = rng.uniform(0.75, 1.0, 8), rng.uniform(0.75, 1.0, 8)
        e = np.zeros(8, complex)
        # 2 |e|^2 <= 16 u ||A||_F d with ||A||_F >= 3, d >= 0.75: |e| <= 4.4e-8
        e[rng.integers(8)] = 4e-8 * (np.exp(2j * np.pi * rng.uniform()) if complex_ and k == 1 else 1.0)
        R = np.sqrt((0.5 * (a + b)) ** 2 + np.abs(e) ** 2)
        w = 0.5 * (1.0 + 0.5 * (a - b) / R)
        i, j = np.arange(8), np.arange(8) + 8
        C[k, i, i], C[k, j, j], C[k, i, j], C[k, j, i] = a, -b, e, e.conj()
        want[k, i, j], want[k, j, i] = e * w, e.conj() * w
        C[-k % N], want[-k % N] = C[k].conj(), want[k].conj()
    X = np.fft.ifft(C, axis=0).real.copy()
    x = torch.from_numpy(X).cuda()
    ws = torch.empty(ve.ve_circulant_workspace_size((N,), D), dtype=torch.uint8, device="cuda")
    ve.ve_circulant_project(x.data_ptr(), x.data_ptr(), (N,), D, ws.data_ptr(), ws.numel())
    torch.cuda.synchronize()
    Y = np.fft.fft(x.cpu().numpy(), axis=0)
    off = np.abs(Y - want)[:, :8, 8:]
    # of max|C| = 1: quantisation u / 2, the weighted entry u / 2, both products and the packing u / 4
    # each; the DFT's own rounding acts on entries of 1e-8 alone
    assert off.max() <= 2 * U
