"""FP32: a particle beside a non-finite field value, but outside its reach, moves as if
that value were zero; one that it reaches is absorbed and reported, and leaves the
other particle of its cell alone.  Half-staggered axes read c-2 .. c+1 below half a cell
and c-1 .. c+2 from half a cell on.  The two gathers add the same products in the same
order: momenta to 4 units of the last place.
"""
import numpy as np
import pytest

from paper_1204_0838_gb300 import pic, workloads as W

pytestmark = pytest.mark.gpu

LAM = W.LAMBDA0
SHAPE = (24, 16, 16)
CELL = np.array([10, 9, 7])
HALF = {0: (0,), 1: (1,), 2: (2,), 3: (1, 2), 4: (0, 2), 5: (0, 1)}  # half-staggered axes of Ex .. Bz


def _sim(offsets, F):
    g = pic.Sim(*SHAPE, LAM / 8, LAM / 3, LAM / 2, LAM, periodic_x=True, precision="fp32", track_ids=True)
    n = len(offsets)
    xi = (CELL + np.array(offsets)).T
    g.set_fields(F)
    g.set_particles(xi, np.full((3, n), 0.25), np.full(n, 1e-3), np.arange(n, dtype=np.uint32))
    return g


@pytest.fixture(autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")


def _fields():
    F = 0.1 * np.random.default_rng(2).standard_normal((9,) + SHAPE)
    F[6:] = 0.0
    return F


@pytest.mark.parametrize("tile", ["8,8,8", "12,8,8"])
@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("comp,axis", [(c, a) for c in range(6) for a in HALF[c]])
@pytest.mark.parametrize("offset", [0.25, 0.75])
def test_value_outside_the_reach_does_not_matter(offset, comp, axis, value, tile, monkeypatch):
    monkeypatch.setenv("PIC_TILE", tile)
    node = CELL.copy()
    node[axis] += 2 if offset < 0.5 else -2  # one beyond the particle's own window
    F = _fields()
    F[(comp,) + tuple(node)] = 0.0
    ref = _sim([[offset] * 3, [offset] * 3], F)
    ref.step(1)
    F[(comp,) + tuple(node)] = value
    g = _sim([[offset] * 3, [offset] * 3], F)
    g.step(1)
    a, b = g.particles(), ref.particles()
    assert a["id"].size == 2
    assert np.abs(a["u"] - b["u"]).max() <= 4 * 2.0 ** -24 * np.abs(b["u"]).max()
    ref.close()
    g.close()


def test_only_the_particle_that_is_reached_is_absorbed():
    F = _fields()
    F[0, CELL[0] + 2, CELL[1], CELL[2]] = np.nan
    g = _sim([[0.25] * 3, [0.75] * 3], F)
    with pytest.raises(pic.PicError):
        g.step(1)
    p = g.particles()
    assert list(p["id"]) == [0] and np.isfinite(p["u"]).all()
    g.close()
