"""The plane pipeline where its warps, accesses and schedules part from the
ordinary: FP64 warps that hold units with and without twiddles.
"""

import pytest

from tests import test_gpu_plane as base

pytestmark = pytest.mark.gpu


# rows of the spectrum plane that are no multiple of a warp: with and without a
# last round that not all threads take
@pytest.mark.parametrize("bc,n", [("sinc", 18), ("sinc", 20), ("sinc", 24), ("sinc", 36), ("sinc", 40), ("sinc", 56),
                                  ("slab", 48)])
def test_fp64_warps_over_two_units(bc, n):
    base.test_plane_pipeline_against_oracle(bc, n, "fp64")
