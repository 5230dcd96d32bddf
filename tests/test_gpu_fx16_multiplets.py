"""The float32 Jacobi inside the 16 x 16 fixed-point projections (csrc/ve_fx16.cuh) on models whose
blocks have multiplets: eigenvalues equal to float32, coupled by entries at rounding level.  Rotating
such a pair turns it by 45 degrees every time and stalls the sweeps."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("delta", [0.0, 0.3, 0.9, 1.0])
def test_sweeps_of_symmetric_models(delta):
    """A warm projection takes two or three float32 sweeps, whatever the model (3.2 a wavevector block on
    the Ising chain); a stalled one takes the limit of ten, cycle after cycle (18 on average)."""
    from paper_2106_02682_gb300 import ve
    h = ve.ve_create((48,), (2,), ve.ve_ham_xxz(1, 1.0, delta), ve.ve_default_options())
    try:
        ve.ve_iterate(h, 40)
        ve.ve_profile(h, 1)
        ve.ve_iterate(h, 20)
        pair, wavevector = ve.ve_profile_sweeps(h)
    finally:
        ve.ve_destroy(h)
    assert pair <= 5.0 and wavevector <= 5.0
