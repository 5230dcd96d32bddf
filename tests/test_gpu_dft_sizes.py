"""The block DFT's lengths (csrc/ve_fft.cu) one by one, 1 .. 64 along either axis of a lattice and as
the factors of a chain, through the X step of a positive block row, which the projection returns
unchanged: what is left is the forward and the inverse transform."""
import numpy as np
import pytest

from paper_2106_02682_gb300 import synth

pytestmark = pytest.mark.gpu


def _run(ve, X, M, precision):
    import torch
    x = torch.from_numpy(X).cuda()
    y = torch.empty_like(x)
    D = X.shape[1]
    ws = torch.empty(ve.ve_circulant_workspace_size(M, D), dtype=torch.uint8, device="cuda")
    ve.ve_circulant_project(x.data_ptr(), y.data_ptr(), M, D, ws.data_ptr(), ws.numel(), precision)
    torch.cuda.synchronize()
    return y.cpu().numpy()


@pytest.mark.parametrize("M", [(n, 3) for n in range(1, 65)] + [(2, n) for n in range(1, 65)] +
                         [(n,) for n in (2, 3, 31, 61, 66, 170, 183, 244, 962, 3721, 4096)])
def test_transforms_of_every_length(M):
    from paper_2106_02682_gb300 import ve
    N = int(np.prod(M))
    X = synth.circulant_first_row(M, 4, seed=N) * 0.1
    X[0] += 10.0 * np.eye(4)   # every wavevector block positive definite
    # a transform's error is a few u log2(N) ||x||, the projection's a few u of blocks of norm 10
    assert np.max(np.abs(_run(ve, X, M, ve.VE_PREC_FP64) - X)) <= 2e-13
    assert np.max(np.abs(_run(ve, X, M, ve.VE_PREC_MIXED) - X)) <= 1e-4
