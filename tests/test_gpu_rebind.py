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


def _small(ff, s):
    m = ff.FFModel(synth.preset("small", skin=0.7), seed=42)
    m.bind(_dev(s.pos), _dev(s.Z, torch.int32), s.box, s.pbc)
    return m


def test_a_rejected_species_leaves_nothing_bound(ff):
    """The list of the rejected system is not built, and neither that system nor the one before
    it can be evaluated: an atomic number outside the table selects no row of it."""
    s = synth.config1_system()
    pos, Z = _dev(s.pos), _dev(s.Z, torch.int32)
    m = _small(ff, s)
    m.energy_forces(pos)
    bad = Z.clone()
    bad[3] = 95
    with pytest.raises(ff.FFError, match="FF_ERR_SPECIES"):
        m.bind(pos, bad, s.box, s.pbc)
    v, mass = torch.zeros_like(pos), _dev(s.masses)
    for call in (lambda: m.energy_forces(pos), lambda: m.energy_forces_graph(pos),
                 lambda: m.forces_adjoint(), lambda: m.virial(), lambda: m.edges(),
                 lambda: m.md(pos.clone(), v, mass, 1, 0.5), lambda: m.autotune(pos)):
        with pytest.raises(ff.FFError, match="FF_ERR_STATE"):
            call()
    m.bind(pos, Z, s.box, s.pbc)
    ref = _small(ff, s)
    for a, b in zip(m.energy_forces(pos), ref.energy_forces(pos)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("call", ["energy_forces", "energy_forces_graph"])
def test_positions_rejected_at_the_bind_can_be_replaced(ff, call):
    """A bind to a larger system at a non-finite position fails; its other data are in place, and
    an evaluation at good positions is that of a context bound there."""
    s0 = synth.config1_system()
    s = synth.water_system(400, L=22.88, seed=7)
    m = _small(ff, s0)
    bad = s.pos.copy()
    bad[17, 2] = np.inf
    with pytest.raises(ff.FFError, match="FF_ERR_NONFINITE"):
        m.bind(_dev(bad), _dev(s.Z, torch.int32), s.box, s.pbc)
    with pytest.raises(ff.FFError, match="FF_ERR_STATE"):
        m.edges()
    ref = _small(ff, s)
    out = []
    for model in (m, ref):
        pos = _dev(s.pos)
        if call == "energy_forces":
            out.append(model.energy_forces(pos))
        else:
            Ea = torch.empty(s.n, dtype=torch.float32, device="cuda")
            F = torch.empty(s.n, 3, dtype=torch.float32, device="cuda")
            out.append(model.energy_forces_graph(pos, None, Ea, F))
    for a, b in zip(*out):
        assert torch.equal(a, b)


def test_a_bind_on_another_stream_waits_for_the_replays_of_the_first(ff):
    """The second system has the first one's size, so that its lists go into the same buffers,
    while replays on the first system are still in flight on their own stream."""
    a = synth.water_system(1365, L=34.44, seed=1001)
    b = synth.water_system(1365, L=34.44, seed=1002)
    hp = synth.preset("fm_water")
    pos_a, Z_a, pos_b, Z_b = (_dev(a.pos), _dev(a.Z, torch.int32), _dev(b.pos),
                              _dev(b.Z, torch.int32))
    Ea = [torch.empty(a.n, dtype=torch.float32, device="cuda") for _ in range(2)]
    F = [torch.empty(a.n, 3, dtype=torch.float32, device="cuda") for _ in range(2)]
    ref = ff.FFModel(hp, seed=42, precision=1)
    ref.bind(pos_a, Z_a, a.box, a.pbc)
    ref.energy_forces_graph(pos_a, None, Ea[0], F[0])
    ref_b = ff.FFModel(hp, seed=42, precision=1)
    ref_b.bind(pos_b, Z_b, b.box, b.pbc)
    out_ref = ref_b.energy_forces(pos_b)
    m = ff.FFModel(hp, seed=42, precision=1)
    Es = torch.empty(1, dtype=torch.float64, device="cuda")
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s1):
        m.bind(pos_a, Z_a, a.box, a.pbc)
        for _ in range(20):
            m.energy_forces_graph(pos_a, Es, Ea[1], F[1])
    with torch.cuda.stream(s2):
        m.bind(pos_b, Z_b, b.box, b.pbc)
        out = m.energy_forces(pos_b)
    torch.cuda.synchronize()
    assert torch.equal(Ea[0], Ea[1]) and torch.equal(F[0], F[1])
    for x, y in zip(out, out_ref):
        assert torch.equal(x, y)
