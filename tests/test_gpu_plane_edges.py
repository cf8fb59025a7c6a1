"""The plane pipeline where its warps, accesses and schedules part from the
ordinary: FP64 warps that hold units with and without twiddles; lanes that are
not the default; buffers off the boundaries that wide accesses need; the
persistent schedule, which solves the same pairs by other transforms.
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


def _psi(n, N, seed, dtype=np.float32):
    import torch
    r = synth.OrbitalRecipe(n=n, h=0.4, norb=N, nsites=3, seed=seed, gauss_per_orb=3,
                            sigma=(0.07 * n * 0.4, 0.12 * n * 0.4), p_type=True)
    return torch.from_numpy(synth.make_orbitals(r, dtype=dtype)).cuda()


def _shifted(t, by):
    """t's values in a buffer that starts `by` elements past an aligned address."""
    import torch
    buf = torch.empty(t.numel() + by, dtype=t.dtype, device=t.device)
    buf[by:] = t.reshape(-1)
    return buf[by:].view(t.shape)


# the same products and sums by narrower accesses: equal to rounding (FP32 1e-6 of
# the largest value, FP64 1e-14).  64^3: enough points for the accumulation by tiles
@pytest.mark.parametrize("n,N,prec", [(16, 9, "fp32"), (24, 3, "fp32"), (64, 10, "fp32"), (24, 9, "fp64")])
@pytest.mark.parametrize("by", [1, 2, 3])
def test_orbitals_and_output_off_their_boundaries(n, N, prec, by):
    from paper_1712_07973_gb300 import exx
    rel = 1e-6 if prec == "fp32" else 1e-14
    psi = _psi(n, N, 60 + n, np.float32 if prec == "fp32" else np.float64)
    plan = exx.ExxPlan(n, 0.4, 0.25, np.linspace(0.5, 2.0, N), precision=prec)
    E0, v0 = plan.gradient(psi)
    for p, q in ((by, by), (by, 0), (0, by)):
        E1, v1 = plan.gradient(_shifted(psi, p), _shifted(psi, q))
        assert abs(E1 - E0) <= 0.1 * rel * abs(E0)
        assert float((v1 - v0).abs().max()) <= rel * float(v0.abs().max())
        assert abs(plan.energy(_shifted(psi, p)) - E0) <= 0.1 * rel * abs(E0)
    plan.close()


@pytest.mark.parametrize("by", [1, 2, 4])  # accumulation widths 1, 2 and 4
@pytest.mark.parametrize("out_by", [0, 1])
def test_batch_buffers_off_their_boundaries(by, out_by):
    import torch
    from paper_1712_07973_gb300 import exx
    spec = [(16, 9), (24, 5), (32, 10)]
    psis = [_psi(n, N, 80 + n) for n, N in spec]
    mols = [{"n": n, "h": 0.4, "alpha": 0.25, "occupations": np.linspace(0.5, 2.0, N)} for n, N in spec]
    b = exx.ExxBatch(mols)
    vx = [torch.empty_like(p) for p in psis]
    b.set_buffers(psis, vx)
    E0 = b.apply().cpu()
    off = [_shifted(p, by) for p in psis]
    out = [_shifted(torch.zeros_like(p), out_by) for p in psis]
    b.set_buffers(off, out)
    E1 = b.apply().cpu()
    assert torch.allclose(E1, E0, rtol=1e-7, atol=0)
    for g, w in zip(out, vx):
        assert float((g - w).abs().max()) <= 1e-6 * float(w.abs().max())
    b.close()


# both schedules hold the FP32 tolerances against the oracle (1e-6 Ha, 2e-6 of the
# action's largest value), so they differ by no more than twice those
def test_persistent_schedule_on_plane_grids():
    import torch
    from paper_1712_07973_gb300 import exx
    spec = [(32, 10), (48, 17), (32, 5), (40, 9), (112, 2)]
    psis = [_psi(n, N, 100 + k) for k, (n, N) in enumerate(spec)]
    mols = [{"n": n, "h": 0.4, "alpha": 0.25, "occupations": np.linspace(0.5, 2.0, N)} for n, N in spec]
    res = []
    for persistent in (False, True):
        b = exx.ExxBatch(mols)
        b.persistent(persistent)
        vx = [torch.empty_like(p) for p in psis]
        b.set_buffers(psis, vx)
        res.append((b.apply().cpu(), vx, b.energy().cpu()))
        b.close()
    (E0, v0, e0), (E1, v1, e1) = res
    assert torch.allclose(E1, E0, rtol=0, atol=2e-6) and torch.allclose(e1, e0, rtol=0, atol=2e-6)
    for g, w in zip(v1, v0):
        assert float((g - w).abs().max()) <= 4e-6 * float(w.abs().max())
