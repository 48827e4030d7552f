"""The bounded waits of the FP32 tensor-core GEMM, without a fault: one that runs out.

As for the BF16 GEMM: with FF_TEST_STALL_ONCE set when a context is created, its first GEMM launch
withholds the completion signal of each CTA's first accumulators, the epilogue's wait ends after
a short limit, every role (splitting warps, weight loads, MMA issuer, both epilogue groups) leaves
through the abort path, and the evaluation reports FF_ERR_TIMEOUT.  The context must then evaluate
like a fresh one, bit for bit.  The two systems give a CTA one tile (2 edges) and several.
"""
import os

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _bind(ff, hp, s):
    m = ff.FFModel(hp, seed=42, precision=0)
    pos = torch.tensor(s.pos, dtype=torch.float64, device="cuda")
    m.bind(pos, torch.tensor(s.Z, dtype=torch.int32, device="cuda"), s.box, s.pbc)
    return m, pos


@pytest.mark.parametrize("key", ["dimer", "csh512"])
def test_a_wait_that_runs_out_is_reported_and_the_context_recovers(key):
    import paper_2502_06073_gb300 as ff
    s = synth.systems.dimer_system(1.4) if key == "dimer" else synth.csh_system(sub=True)
    hp = synth.preset("fm_water")
    os.environ["FF_TEST_STALL_ONCE"] = "1"
    try:
        m, pos = _bind(ff, hp, s)
    finally:
        del os.environ["FF_TEST_STALL_ONCE"]
    with pytest.raises(ff.FFError, match="FF_ERR_TIMEOUT"):
        m.energy_forces(pos)
    _, Ea, F = m.energy_forces(pos)
    ref, pos_r = _bind(ff, hp, s)
    _, Ea_r, F_r = ref.energy_forces(pos_r)
    assert torch.equal(Ea, Ea_r) and torch.equal(F, F_r)
    assert np.isfinite(F.cpu().numpy()).all()
