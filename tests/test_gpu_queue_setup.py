"""The first enable of the persistent schedule when one of its allocations
fails: the status, the batch as it was before (schedule, results, workspace),
and a later enable that works.  The failure is simulated on the host
(EXX_TEST_FAIL_ALLOC); nothing is exhausted on the device.
"""

import numpy as np
import pytest

from paper_1712_07973_gb300 import synth

pytestmark = pytest.mark.gpu

# two groups of the plane pipeline (tables of their own for the queue), one of the slab pipeline
SPEC = [(24, 9), (16, 3), (12, 5), (24, 3)]


@pytest.mark.parametrize("lanes,allocations", [("1", 4 + 2 + 2 + 2), ("2", 4 + 2 + 2)])
def test_failed_enable_leaves_the_batch_as_it_was(monkeypatch, lanes, allocations):
    import torch
    from paper_1712_07973_gb300 import exx
    monkeypatch.setenv("EXX_LANES", lanes)
    psis, mols = [], []
    for k, (n, N) in enumerate(SPEC):
        r = synth.OrbitalRecipe(n=n, h=0.45, norb=N, nsites=3, seed=20 + k, gauss_per_orb=3,
                                sigma=(0.12 * n * 0.45, 0.2 * n * 0.45), p_type=True)
        psis.append(torch.from_numpy(synth.make_orbitals(r, dtype=np.float32)).cuda())
        mols.append({"n": n, "h": 0.45, "alpha": 0.25, "occupations": np.full(N, 2.0)})
    vx = [torch.empty_like(p) for p in psis]

    def results(b):
        for v in vx:
            v.fill_(7.0)
        return b.apply().cpu(), [v.clone() for v in vx]

    straight = exx.ExxBatch(mols)
    before = straight.info()
    straight.persistent(True)
    after = straight.info()
    straight.set_buffers(psis, vx)
    Ep, vp = results(straight)
    straight.close()
    for k in range(1, allocations + 2):
        b = exx.ExxBatch(mols)
        b.set_buffers(psis, vx)
        E0, v0 = results(b)
        monkeypatch.setenv("EXX_TEST_FAIL_ALLOC", str(k))
        if k <= allocations:
            with pytest.raises(exx.ExxError) as ei:
                b.persistent(True)
            assert ei.value.status == 3
            assert b.info() == before
            E1, v1 = results(b)
            assert torch.equal(E1, E0) and all(map(torch.equal, v1, v0))
            monkeypatch.delenv("EXX_TEST_FAIL_ALLOC")
        b.persistent(True)
        monkeypatch.delenv("EXX_TEST_FAIL_ALLOC", raising=False)
        assert b.info() == after
        E2, v2 = results(b)
        assert torch.equal(E2, Ep) and all(map(torch.equal, v2, vp))
        b.persistent(False)
        E3, v3 = results(b)
        assert torch.equal(E3, E0) and all(map(torch.equal, v3, v0))
        b.close()
