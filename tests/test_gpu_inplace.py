"""FP32 calls whose output shares memory with the orbitals: in place, shifted
by an orbital, and between the molecules of a batch.  The output must not be
written before the last read of the orbitals, so each call must equal the one
with buffers of its own, to FP32 rounding (1e-6 of the largest value: the same
sums, from other instances of the accumulation kernel).
"""

import numpy as np
import pytest

from paper_1712_07973_gb300 import synth

pytestmark = pytest.mark.gpu


def _orbitals(n, N, seed):
    import torch
    r = synth.OrbitalRecipe(n=n, h=0.45, norb=N, nsites=3, seed=seed, gauss_per_orb=3,
                            sigma=(0.12 * n * 0.45, 0.2 * n * 0.45), p_type=True)
    return torch.from_numpy(synth.make_orbitals(r, dtype=np.float32)).cuda()


def _same(got, want):
    return float((got - want).abs().max()) <= 1e-6 * float(want.abs().max())


# one tile and several, ragged ones; the accumulation with one orbital per CTA row (up to 56^3) and
# without; scalar accesses (9^3); slab and plane pipelines
@pytest.mark.parametrize("n,N,bc", [(9, 10, "sinc"), (12, 9, "sinc"), (24, 5, "sinc"), (24, 19, "sinc"),
                                    (56, 10, "sinc"), (64, 10, "sinc"), (64, 10, "periodic")])
@pytest.mark.parametrize("call", ["apply", "gradient"])
@pytest.mark.parametrize("shift", [0, 1, -1])
def test_plan_output_over_the_orbitals(n, N, bc, call, shift):
    import torch
    from paper_1712_07973_gb300 import exx
    psi = _orbitals(n, N, 70 + n)
    plan = exx.ExxPlan(n, 0.45, 0.25, np.linspace(0.5, 2.0, N), precision="fp32", kernel=bc)
    E0, want = getattr(plan, call)(psi)
    buf = torch.zeros((N + 2, n, n, n), device="cuda")
    src, out = buf[1:N + 1], buf[1 + shift:N + 1 + shift]
    src.copy_(psi)
    E1, got = getattr(plan, call)(src, out)
    plan.close()
    assert E1 == E0
    assert _same(got, want)


@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("graph", [False, True])
def test_batch_outputs_over_orbitals(persistent, graph):
    # in place, then with the outputs of two molecules of one size swapped; then with
    # buffers of their own again (the schedule goes back, graphs included)
    import torch
    from paper_1712_07973_gb300 import exx
    spec = [(24, 9), (24, 9), (16, 5), (32, 17)]
    psis = [_orbitals(n, N, 90 + k) for k, (n, N) in enumerate(spec)]
    mols = [{"n": n, "h": 0.45, "alpha": 0.25, "occupations": np.linspace(0.5, 2.0, N)} for n, N in spec]
    b = exx.ExxBatch(mols)
    b.persistent(persistent)
    s = torch.cuda.Stream()
    b.graph(graph)
    E = torch.zeros(len(mols), dtype=torch.float64, device="cuda")

    def call(ins, outs):
        b.set_buffers(ins, outs, stream=s)
        s.wait_stream(torch.cuda.current_stream())
        b.gradient(E, stream=s)
        s.synchronize()
        return E.clone(), [o.clone() for o in outs]

    E0, want = call(psis, [torch.empty_like(p) for p in psis])
    a = [p.clone() for p in psis]
    E1, got = call(a, a)
    assert torch.equal(E1, E0) and all(map(_same, got, want))
    a = [p.clone() for p in psis]
    E2, got = call(a, [a[1], a[0], a[2], a[3]])
    assert torch.equal(E2, E0) and all(map(_same, got, want))
    E3, got = call(psis, [torch.empty_like(p) for p in psis])
    assert torch.equal(E3, E0) and all(map(_same, got, want))
    b.close()
