"""The plane pipeline where its warps, accesses and schedules part from the
ordinary: FP64 warps that hold units with and without twiddles; lanes that are
not the default.
"""

import numpy as np
import pytest

from paper_1712_07973_gb300 import synth
from tests import test_gpu_plane as base

pytestmark = pytest.mark.gpu


# rows of the spectrum plane that are no multiple of a warp: with and without a
# last round that not all threads take
@pytest.mark.parametrize("bc,n", [("sinc", 18), ("sinc", 20), ("sinc", 24), ("sinc", 36), ("sinc", 40), ("sinc", 56),
                                  ("slab", 48)])
def test_fp64_warps_over_two_units(bc, n):
    base.test_plane_pipeline_against_oracle(bc, n, "fp64")


def test_second_lane_where_one_is_the_default():
    # FP32 128^3 runs one lane but takes two; their results are the same
    import torch
    from paper_1712_07973_gb300 import exx
    n, N = 128, 9
    r = synth.OrbitalRecipe(n=n, h=0.4, norb=N, nsites=4, seed=5, gauss_per_orb=3, sigma=(2.0, 4.0), p_type=True)
    psi = torch.from_numpy(synth.make_orbitals(r, dtype=np.float32)).cuda()
    plan = exx.ExxPlan(n, 0.4, 0.25, np.full(N, 2.0), precision="fp32")
    one = plan.info()
    assert one["ntiles"] == 3 and one["lanes"] == 1
    E1, v1 = plan.apply(psi)
    plan.set_lanes(2)
    two = plan.info()
    assert two["lanes"] == 2 and two["workspace_bytes"] > one["workspace_bytes"]
    E2, v2 = plan.apply(psi)
    assert E2 == E1 and torch.equal(v2, v1)
    with pytest.raises(exx.ExxError) as ei:
        plan.set_lanes(3)
    assert ei.value.status == 5
    plan.set_lanes(1)
    E3, v3 = plan.apply(psi)
    assert E3 == E1 and torch.equal(v3, v1)
    assert plan.info() == {**two, "lanes": 1}
    plan.close()
