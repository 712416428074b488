"""The FP64 gather of a weak field in a tile that also holds a strong one.

Staged fields carry 60 bits of the tile's largest value, here 1.5: a unit is 2^-59.  A
uniform weak field of a whole number of units, 4 k + 2, must come back to 1.5 units rms
over random offsets.  It is exact as staged; the gather drops 16 products for each of four
nodes and 4 more, each twice 1/12 of a unit rms and without sign, and rounds five
shifts: below 0.7 units rms.  (Staged at 58 bits, all of these are four times as large,
and the staged value is off by two units.)
The momentum of a particle at rest, without a magnetic field, is -dt E to one rounding
of the weak value, far below a unit.
"""
import numpy as np
import pytest

from paper_1204_0838_gb300 import pic, workloads as W

pytestmark = pytest.mark.gpu

LAM = W.LAMBDA0
SHAPE = (24, 16, 16)
UNIT = 2.0 ** -59


@pytest.mark.parametrize("tile", ["8,8,8", "10,8,8"])
def test_weak_uniform_field_beside_a_strong_value(tile, monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    monkeypatch.setenv("PIC_TILE", tile)
    g = pic.Sim(*SHAPE, LAM / 8, LAM / 3, LAM / 2, LAM, periodic_x=True, precision="fp64", track_ids=True)
    weak = np.array([4 * 0x1f3579bdb2a6 + 2, -(4 * 0x35b7d9ace5c3 + 2), 4 * 0x9e3779b97f5 + 2]) * UNIT
    F = np.zeros((9,) + SHAPE)
    F[:3] = weak[:, None, None, None]
    F[:3, 7, 7, 7] = 1.5  # in the tile, out of reach of cells 0 .. 3
    n = 4000
    rng = np.random.default_rng(4)
    xi = rng.uniform(0, 4, (3, n))
    g.set_fields(F)
    g.set_particles(xi, np.zeros((3, n)), np.full(n, 1e-30), np.arange(n, dtype=np.uint32))
    dt = g.info()["dt"]
    g.step(1)
    p = g.particles()
    for a in range(3):
        err = (p["u"][a] / dt + weak[a]) / UNIT
        assert np.sqrt(np.mean(err ** 2)) <= 1.5, (a, err.std(), err.mean())
    g.close()
