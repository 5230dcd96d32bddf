"""Device memory of a handle: 3-spin clusters keep no float64 eigenvectors (their projections in float64
and double-float are by the matrix sign)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_three_spin_clusters_hold_no_float64_eigenvectors():
    import torch
    from paper_2106_02682_gb300 import ve
    N, D = 1024, 64
    warm = ve.ve_create((6,), (3,), ve.ve_ham_tfim(1, 1.0, 1.0))  # the library's own first use
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    h = ve.ve_create((3 * N,), (3,), ve.ve_ham_tfim(1, 1.0, 1.0))
    held = before - torch.cuda.mem_get_info()[0]
    state = ve.ve_state_size(h)
    ve.ve_destroy(h)
    ve.ve_destroy(warm)
    # the state, two spectra, the float32 eigenvectors, small arrays; with two float64 stores 196 MB more
    need = state + 2 * 16 * N * D * D // 2 + 4 * 3 * N * D * D
    assert need <= held <= 1.15 * need + 2 ** 24
