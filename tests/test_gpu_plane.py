"""The plane pipeline (csrc/exx_plane.cuh) against the FP64 oracle at the grids
where its shapes change: the smallest grid, sub-DFT lengths of 2 to 16 with
odd ones among them, groups of 32 and of 16 lines, several CTAs per SM, one
CTA per SM, planes taken in two halves, and the mixed line kinds.
Tolerances are those of the other parity tests: FP64 1e-10 relative; FP32
1e-6 Ha and 2e-6 of the action's largest value.
"""

import numpy as np
import pytest

from oracle import exx_oracle as o
from paper_1712_07973_gb300 import synth

pytestmark = pytest.mark.gpu

CASES = ([("sinc", n, "fp32") for n in (16, 18, 20, 28, 36, 40, 56, 72, 112, 128)]
         + [("sinc", n, "fp64") for n in (16, 28, 48, 72, 80, 112)]
         + [("periodic", n, "fp32") for n in (16, 24, 48, 64, 128)] + [("periodic", 96, "fp64")]
         + [("slab", n, p) for n in (16, 64, 96) for p in ("fp32", "fp64")]
         + [("wire", n, p) for n in (16, 64, 96) for p in ("fp32", "fp64")])


@pytest.mark.parametrize("bc,n,prec", CASES)
def test_plane_pipeline_against_oracle(bc, n, prec):
    import torch
    from paper_1712_07973_gb300 import exx
    dev, h, N = torch.device("cuda:0"), 0.4, 2
    r = synth.OrbitalRecipe(n=n, h=h, norb=N, nsites=2, seed=900 + n, gauss_per_orb=3,
                            sigma=(0.07 * n * h, 0.12 * n * h), p_type=True)
    dt = torch.float64 if prec == "fp64" else torch.float32
    psi = torch.from_numpy(synth.make_orbitals(r)).to(dev, dt)
    occ = np.array([2.0, 1.25])
    G = {"periodic": o.kernel_spectrum_periodic, "slab": o.kernel_spectrum_slab, "wire": o.kernel_spectrum_wire}.get(bc)
    Gh = G(n, h) if G else o.kernel_spectrum(o.kernel_real_space(n, h))
    Eo, vxo, Eijo = o.exx(psi.double().cpu().numpy(), occ, 0.25, h, Gh)
    plan = exx.ExxPlan(n, h, 0.25, occ, precision=prec, kernel=bc)
    Ee = plan.energy(psi)
    E, vx = plan.apply(psi)
    Eij = plan.pair_energies()
    plan.close()
    e_tol = 1e-10 * max(abs(Eo), np.max(np.abs(Eijo))) if prec == "fp64" else 1e-6
    v_tol = (1e-10 if prec == "fp64" else 2e-6) * np.max(np.abs(vxo))
    assert abs(E - Eo) <= e_tol and abs(Ee - Eo) <= e_tol
    assert np.max(np.abs(Eij - [Eijo[0, 0], Eijo[0, 1], Eijo[1, 1]])) <= e_tol
    assert np.max(np.abs(vx.double().cpu().numpy() - vxo)) <= v_tol


@pytest.mark.parametrize("persistent", [False, True])
def test_batch_with_an_odd_number_of_accumulators_before_even_grids(persistent):
    # 3 orbitals on 9^3 hold an odd number of FP64 accumulators; those of the
    # next molecules (vector accesses) must stay aligned
    import torch
    from paper_1712_07973_gb300 import exx
    dev = torch.device("cuda:0")
    mols, psis, ref = [], [], []
    for k, (n, N) in enumerate(((9, 3), (8, 2), (16, 3), (9, 1), (20, 2))):
        r = synth.OrbitalRecipe(n=n, h=0.45, norb=N, nsites=2, seed=40 + k, gauss_per_orb=3,
                                sigma=(0.12 * n * 0.45, 0.2 * n * 0.45), p_type=True)
        psis.append(torch.from_numpy(synth.make_orbitals(r)).to(dev, torch.float32))
        mols.append({"n": n, "h": 0.45, "alpha": 0.25, "occupations": np.full(N, 2.0)})
        Gh = o.kernel_spectrum(o.kernel_real_space(n, 0.45))
        ref.append(o.exx(psis[-1].double().cpu().numpy(), np.full(N, 2.0), 0.25, 0.45, Gh)[:2])
    b = exx.ExxBatch(mols)
    b.persistent(persistent)
    vx = [torch.empty_like(p) for p in psis]
    b.set_buffers(psis, vx)
    E = b.apply().cpu()
    for k, (Eo, vo) in enumerate(ref):
        assert abs(float(E[k]) - Eo) <= 1e-6
        assert np.max(np.abs(vx[k].double().cpu().numpy() - vo)) <= 2e-6 * np.max(np.abs(vo))
    b.close()
