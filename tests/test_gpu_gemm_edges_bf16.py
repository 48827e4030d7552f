"""MLP widths at the edges of the BF16 GEMM's tiles: the row-per-lane epilogue of the persistent
kernel, half chunks (N % 32 = 16), last slices of 16 columns, N = 16, and two edges in all.

The same widths as the FP32 test.  The persistent kernel is held to the one-tile kernels, which
transpose through shared memory and clip by themselves: no element-wise arithmetic differs, only
the order of row sums over up to 512 columns (u sqrt(512) = 1.4e-6, for forces that are differences
of sums some ten times larger, with a factor of three: 5e-5 of the largest).  A column too many or
too few in a row of 272 would be 4e-3.  And both are held to the FP32 path within the rounding of
their operands: 2^-8 in each of about eight chained products, twice that many for the forces, with
a factor of three, 5e-2.
"""
import pytest

import synth
from test_gpu_gemm_edges import WIDTHS

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _evaluate(hp, s, precision, tiles=None):
    import paper_2502_06073_gb300 as ff
    m = ff.FFModel(hp, seed=42, precision=precision)
    pos = torch.tensor(s.pos, dtype=torch.float64, device="cuda")
    m.bind(pos, torch.tensor(s.Z, dtype=torch.int32, device="cuda"), s.box, s.pbc)
    if tiles:
        m.set_tiles(*tiles)
    _, Ea, F = m.energy_forces(pos)
    return Ea.double(), F.double()


def _compare(hp, s):
    off = lambda x, y: float((x - y).abs().max() / y.abs().max())  # noqa: E731
    row = _evaluate(hp, s, 1, (128, 0))
    for tiles in ((128, 2), (256, 0)):
        for a, b in zip(row, _evaluate(hp, s, 1, tiles)):
            assert off(a, b) <= 5e-5, tiles
    for a, b in zip(row, _evaluate(hp, s, 0)):
        assert off(a, b) <= 5e-2


@pytest.mark.parametrize("two_body,latent", WIDTHS)
def test_bf16_widths_at_tile_edges(two_body, latent):
    _compare(synth.preset("small", two_body=two_body, latent=latent, lmax=2),
             synth.config1_system())


def test_bf16_two_edges():
    _compare(synth.preset("fm_water"), synth.systems.dimer_system(1.4))
