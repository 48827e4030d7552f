"""Binding one context to one system after another.

Every comparison is bit for bit with a fresh context bound to the same system: the same kernels
run on the same list in the same order.
"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ff():
    import paper_2502_06073_gb300 as ff
    ff._build.build()
    ff.load_library()
    assert torch.cuda.is_available()
    return ff


def _dev(a, dt=torch.float64):
    return torch.tensor(np.asarray(a), dtype=dt, device="cuda")


def test_batches_divided_differently(ff):
    """The same 1,024 molecules as systems of one, two and five molecules each: the system of an
    atom decides its neighbours and the weight of its energy in the adjoint."""
    s = synth.molecules_system(1024, seed=1003)
    pos, Z = _dev(s.pos), _dev(s.Z, torch.int32)
    hp = synth.preset("small")
    m = ff.FFModel(hp, seed=42)

    def forces(model, step):
        ptr = np.unique(np.append(s.sys_ptr[::step], s.sys_ptr[-1])).astype(np.int32)
        model.bind(pos, Z, s.box, s.pbc, ptr)
        Es, _, _ = model.energy_forces(pos, forces=False)
        g = torch.linspace(0.5, 2.0, ptr.shape[0] - 1, dtype=torch.float64, device="cuda")
        return Es, model.forces_adjoint(g)

    for step in (1, 2, 5, 1):
        Es, F = forces(m, step)
        Es_ref, F_ref = forces(ff.FFModel(hp, seed=42), step)
        assert torch.equal(Es, Es_ref) and torch.equal(F, F_ref)
