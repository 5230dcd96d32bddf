"""Definite blocks come back from the 16 x 16 fixed-point X step (csrc/ve_fft.cu, k_xproj16) as their
Hermitian part, as the others do: rounding that breaks X_{-delta} = X_delta^T must not pass through."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.mark.parametrize("M", [(2,), (8,), (9,), (4, 6)])
@pytest.mark.parametrize("D", [4, 16, 64])
def test_definite_blocks_are_made_hermitian(D, M):
    import torch
    from paper_2106_02682_gb300 import synth, ve
    N = int(np.prod(M))
    rng = np.random.default_rng(N)
    X = 0.1 * synth.circulant_first_row(M, D, seed=N)
    X[0] += 5.0 * np.eye(D)
    skew = 1e-9 * rng.normal(size=X.shape)
    skew -= np.swapaxes(skew[synth.neg_linear_index(M)], 1, 2)
    C = np.fft.fftn(X.reshape(M + (D, D)), axes=tuple(range(len(M)))).reshape(N, D, D)
    assert np.linalg.eigvalsh(C).min() > 0.1
    for precision in (ve.VE_PREC_FP64, ve.VE_PREC_DF64):
        x = torch.from_numpy(X + skew).cuda()
        y = torch.empty_like(x)
        ws = torch.empty(ve.ve_circulant_workspace_size(M, D), dtype=torch.uint8, device="cuda")
        ve.ve_circulant_project(x.data_ptr(), y.data_ptr(), M, D, ws.data_ptr(), ws.numel(), precision)
        torch.cuda.synchronize()
        # rounding of the DFT and the projection: 64 n u max|C| (double-float D = 4: 2^-48)
        u = 2.0 ** -48 if D == 4 and precision == ve.VE_PREC_DF64 else U
        assert np.max(np.abs(y.cpu().numpy() - X)) <= 64 * D * u * np.max(np.abs(C))
