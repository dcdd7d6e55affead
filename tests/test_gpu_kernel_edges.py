"""Edges of the step and adjoint kernels' ranges: the sizes at which a lane,
tile or ring of samples is partly filled, against identities, independent
forward differences and the general paths."""
import pytest

from tests import test_gpu_adjoint as adj

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Nth", [129, 200, 256, 257, 300])
def test_adjoint_step_fp64_wide_rows(Nth):
    """The FP64 adjoint's row segments of 8 (128 < Ntheta <= 256, partly
    filled and full) and 32, and rows longer than the thread block
    (Ntheta > 256), where the source derivatives read columns that other
    threads then overwrite: spin term against differences of the step, taped
    against recomputed."""
    adj.test_one_step_spin_term_against_step_differences(False, 2, Nth)
    adj.test_tape_step_and_adjoint_equal_recompute(False, 2, Nth, "fp64")
