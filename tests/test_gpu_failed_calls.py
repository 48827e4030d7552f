"""A call that reports an error leaves the context as usable, and as right, as it was before.

Every comparison is bit for bit with a context that never saw the failing call: the same kernels
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


def _water():
    return synth.water_system(400, L=22.88, seed=7)   # 1,200 atoms


def _bind(ff, s, precision=0):
    m = ff.FFModel(synth.preset("small", skin=0.7), seed=42, precision=precision)
    pos = _dev(s.pos)
    m.bind(pos, _dev(s.Z, torch.int32), s.box, s.pbc)
    return m, pos


def _rejected(s, kind):
    """Positions whose list update fails, at a stage of its own, and the status it reports."""
    bad = s.pos.copy()
    if kind == "nonfinite":        # the other atoms closer together: more edges than before
        bad *= 0.9
        bad[5, 1] = np.nan
        return bad, "FF_ERR_NONFINITE"
    if kind == "box":              # an image shift beyond 100 box lengths
        bad[0, 0] += 150.0 * s.box[0]
        return bad, "FF_ERR_BOX"
    bad *= 0.02                    # every atom has 1,199 neighbours, above FF_MAX_NEIGHBORS
    return bad, "FF_ERR_CAPACITY"


KINDS = ["nonfinite", "box", "crowded"]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kind", KINDS)
def test_adjoint_virial_and_edges_after_a_failed_update(ff, kind, precision):
    s = _water()
    ref, pos_r = _bind(ff, s, precision)
    ref.energy_forces(pos_r, forces=False)
    F_ref = ref.forces_adjoint()
    W_ref = ref.virial()
    m, pos = _bind(ff, s, precision)
    m.energy_forces(pos, forces=False)
    bad, status = _rejected(s, kind)
    bad = _dev(bad)
    with pytest.raises(ff.FFError, match=status):
        m.energy_forces(bad)
    assert torch.equal(m.forces_adjoint(), F_ref)
    assert torch.equal(m.virial(), W_ref)
    for a, b in zip(m.edges(), ref.edges()):
        np.testing.assert_array_equal(a, b)
    # and an accepted update afterwards is that of a fresh context
    _, Ea, F = m.energy_forces(pos)
    _, Ea_ref, F2_ref = ref.energy_forces(pos_r)
    assert torch.equal(Ea, Ea_ref) and torch.equal(F, F2_ref)


@pytest.mark.parametrize("kind", KINDS)
def test_graph_replay_after_a_failed_update(ff, kind):
    s = _water()
    m, pos = _bind(ff, s)
    Es = torch.empty(1, dtype=torch.float64, device="cuda")
    Ea = torch.empty(s.n, dtype=torch.float32, device="cuda")
    F = torch.empty(s.n, 3, dtype=torch.float32, device="cuda")
    m.energy_forces_graph(pos, Es, Ea, F)
    m.energy_forces_graph(pos, Es, Ea, F)
    ref = [t.clone() for t in (Es, Ea, F)]
    bad, status = _rejected(s, kind)
    bad = _dev(bad)
    with pytest.raises(ff.FFError, match=status):
        m.energy_forces(bad)
    for t in (Es, Ea, F):
        t.zero_()
    m.energy_forces_graph(pos, Es, Ea, F)
    for t, r in zip((Es, Ea, F), ref):
        assert torch.equal(t, r)


def test_a_list_update_of_non_finite_positions_costs_no_more_than_a_good_one(ff):
    """An MD run that has blown up: every coordinate is NaN.  The atoms fall into no cell (in one
    cell together they would be tested pair by pair, 7e10 of them here); the call reports them
    within three times the time of a good bind."""
    g = np.arange(64) * 2.2
    pos = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    box, pbc = np.full(3, 64 * 2.2), np.array([True] * 3)
    pos, Z = _dev(pos), torch.ones(64 ** 3, dtype=torch.int32, device="cuda")
    bad = torch.full_like(pos, float("nan"))
    m = ff.FFModel(synth.preset("small"), seed=42)

    def timed(call):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        call()
        b.record()
        b.synchronize()
        return a.elapsed_time(b)

    def rejected():
        with pytest.raises(ff.FFError, match="FF_ERR_NONFINITE"):
            m.bind(bad, Z, box, pbc)

    m.bind(pos, Z, box, pbc)
    good = min(timed(lambda: m.bind(pos, Z, box, pbc)) for _ in range(3))
    t = min(timed(rejected) for _ in range(3))
    assert t <= 3 * good, (t, good)
