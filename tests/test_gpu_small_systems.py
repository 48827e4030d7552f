"""The tensor-product variant for few atoms (one block per atom) against the general one.

A cluster is evaluated alone, which takes the variant for few atoms, and as each member of a
batch of copies that is too large for it.  Copies do not interact and every kernel works edge by
edge or atom by atom in the same order in both, so per-atom energies and forces agree bit for
bit.  The clusters include an isolated atom and a pair (fewer edges than a block's teams).
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(hp, precision, pos, Z, box, ptr):
    import paper_2502_06073_gb300 as ff
    m = ff.FFModel(hp, seed=42, precision=precision)
    p = torch.tensor(pos, dtype=torch.float64, device="cuda")
    m.bind(p, torch.tensor(Z, dtype=torch.int32, device="cuda"), box, [False] * 3, ptr)
    _, Ea, F = m.energy_forces(p)
    return Ea.cpu().numpy(), F.cpu().numpy()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("model", ["small", "fm64", "fm_water", "fm256"])
def test_few_atoms_variant_equals_the_general_one(model, precision):
    hp = synth.preset(model)
    c = synth.systems.cluster_system(n=13)
    d = synth.systems.dimer_system(1.3)
    pos = np.concatenate([c.pos, d.pos, np.zeros((1, 3))])
    Z = np.concatenate([c.Z, d.Z, [8]]).astype(np.int32)
    ptr = np.array([0, c.n, c.n + 2, c.n + 3], np.int32)
    n, copies = len(Z), 60                      # 16 atoms alone, 960 in the batch
    box = [60.0] * 3
    Ea, F = _run(hp, precision, pos, Z, box, ptr)
    big = np.concatenate([[0]] + [ptr[1:] + k * n for k in range(copies)]).astype(np.int32)
    Eb, Fb = _run(hp, precision, np.tile(pos, (copies, 1)), np.tile(Z, copies), box, big)
    assert np.abs(F).max() > 0 and np.isfinite(F).all()
    for k in (0, copies // 2, copies - 1):
        np.testing.assert_array_equal(Eb[k * n:(k + 1) * n], Ea)
        np.testing.assert_array_equal(Fb[k * n:(k + 1) * n], F)
