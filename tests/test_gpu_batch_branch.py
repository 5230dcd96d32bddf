"""Batches on either side of the rule that gives every instance's status a branch of its own in the
batch's graph (csrc/ve_api.cu, kBranchBatch): the iterates are those of single handles."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [8, 9])
def test_batches_reproduce_single_handles(count):
    from paper_2106_02682_gb300 import ve
    inst = [((2 * (4 + i),), (2,), ve.ve_ham_tfim(1, 1.0, 0.4 + 0.1 * i)) for i in range(count)]
    opt = ve.ve_default_options(precision=ve.VE_PREC_MIXED)
    b = ve.ve_create_batch(inst, opt)
    try:
        ve.ve_batch_iterate(b, 25)
        for i, (lattice, cluster, ham) in enumerate(inst):
            h = ve.ve_create(lattice, cluster, ham, opt)
            try:
                _, st = ve.ve_iterate(h, 25)
                assert np.array_equal(ve.ve_get_state(ve.ve_batch_handle(b, i)), ve.ve_get_state(h))
                assert ve.ve_get_status(ve.ve_batch_handle(b, i)).energy_per_spin == st.energy_per_spin
            finally:
                ve.ve_destroy(h)
    finally:
        ve.ve_batch_destroy(b)
