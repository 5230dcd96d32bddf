"""Power-of-two transforms on either side of the rule that gives small passes four points a thread
(csrc/ve_fft.cu, k_fft_quad): through the X step of a positive block row, which comes back unchanged."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,M", [(4, (16,)), (4, (32, 32)), (4, (4096,)), (16, (16,)), (16, (64,)), (16, (16, 16)),
                                 (16, (16, 32)), (16, (32, 32)), (16, (64, 16)), (16, (1024,)), (16, (4096,)),
                                 (64, (32,)), (64, (64,)), (64, (16, 16))])
def test_transforms(D, M):
    import torch
    from paper_2106_02682_gb300 import synth, ve
    N = int(np.prod(M))
    X = synth.circulant_first_row(M, D, seed=N) * 0.1
    X[0] += 10.0 * np.eye(D)   # every wavevector block positive definite
    for precision, tol in ((ve.VE_PREC_FP64, 4e-13), (ve.VE_PREC_MIXED, 2e-4)):
        x = torch.from_numpy(X).cuda()
        y = torch.empty_like(x)
        ws = torch.empty(ve.ve_circulant_workspace_size(M, D), dtype=torch.uint8, device="cuda")
        ve.ve_circulant_project(x.data_ptr(), y.data_ptr(), M, D, ws.data_ptr(), ws.numel(), precision)
        torch.cuda.synchronize()
        # a few u log2(N) ||x|| of the transforms, a few n u of blocks of norm 10 to 14
        assert np.max(np.abs(y.cpu().numpy() - X)) <= tol
