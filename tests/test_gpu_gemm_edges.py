"""MLP widths at the edges of the GEMM tiles, through whole evaluations against the FP64 oracle.

The widths are chosen so that the dense layers meet a K that ends inside a 32- or 64-element
chunk, column counts just above and below a 128-column slice, a last slice of 16 columns, and
the smallest and largest widths; the 96-atom cell has about 5,400 edges, not a multiple of the
128-row tile, and a dimer pair of atoms has two.  Bars as for every other FP32 evaluation:
per-atom energies 5e-6 of the largest, forces 1e-4 eV/A; and, since the random-weight forces are of the
order of 0.05 eV/A, 2e-5 of the largest force as well (FP32 rounding of about ten chained
products of length <= 600: u sqrt(600) sqrt(10) = 5e-6, with a factor of four).
"""
import numpy as np
import pytest

import synth
from oracle import Allegro64

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _evaluate(hp, s, precision=0):
    import paper_2502_06073_gb300 as ff
    m = ff.FFModel(hp, seed=42, precision=precision)
    pos = torch.tensor(s.pos, dtype=torch.float64, device="cuda")
    m.bind(pos, torch.tensor(s.Z, dtype=torch.int32, device="cuda"), s.box, s.pbc)
    _, Ea, F = m.energy_forces(pos)
    return Ea.double().cpu().numpy(), F.double().cpu().numpy()


WIDTHS = [([16, 16], [16]), ([48, 144], [144]), ([80, 112, 272], [176, 272]),
          ([64, 240], [16, 240]), ([512], [512]), ([32, 400], [400])]


@pytest.mark.parametrize("two_body,latent", WIDTHS)
def test_fp32_widths_at_tile_edges(two_body, latent):
    s = synth.config1_system()
    hp = synth.preset("small", two_body=two_body, latent=latent, lmax=2)
    E_ref, Ea_ref, F_ref = Allegro64(hp, 42).evaluate(s.pos, s.Z, s.box, s.pbc)
    Ea, F = _evaluate(hp, s)
    assert np.abs(Ea - Ea_ref).max() <= 5e-6 * np.abs(Ea_ref).max()
    assert np.abs(F - F_ref).max() <= min(1e-4, 2e-5 * np.abs(F_ref).max())


def test_fp32_two_edges():
    s = synth.systems.dimer_system(1.4)
    hp = synth.preset("fm_water")
    E_ref, Ea_ref, F_ref = Allegro64(hp, 42).evaluate(s.pos, s.Z, s.box, s.pbc)
    Ea, F = _evaluate(hp, s)
    assert np.abs(Ea - Ea_ref).max() <= 5e-6 * np.abs(Ea_ref).max()
    assert np.abs(F - F_ref).max() <= min(1e-4, 2e-5 * np.abs(F_ref).max())
