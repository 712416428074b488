"""One step against the FP64 oracle at the sizes where the push can go wrong: tiles that do not divide the grid, strides known to the compiler and
not, one particle, an odd number in a cell (half a pair), more particles in a
tile than one pass takes (2304), more in a cell than are ranked (32), and
momenta with which most particles leave their cell (the separate deposit).

Tolerances: FP64 the 1e-10 parity bar, relative to the largest value and in
cells.  FP32 (eps = 2^-24): momenta 32 eps of the largest |u| (a few dozen
roundings of the Boris push and the gather), positions 32 eps of a cell, and
for a current value 16 eps sum |q w jc| over the particles whose window can
reach the node: a contribution q w jc run A has |run| <= 3/4, A <= 0.45, the
running sum carries the roundings of at most eight shape factors and of the
move (below 24 eps), A four, and they may all add up.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1204_0838_gb300 import pic, workloads as W

from .pairs import by_id

pytestmark = pytest.mark.gpu

LAM = W.LAMBDA0
EPS = 2.0 ** -24


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    pic.lib()


def _positions(kind, shape, n, rng):
    """n positions whose offsets are float32 numbers."""
    cell = np.stack([rng.integers(0, s, n) for s in shape])
    if kind == "cell":      # all in one cell
        cell[:] = np.array([5, 6, 3])[:, None]
    elif kind == "tile":    # all in one 8x8x8 tile
        cell = np.stack([rng.integers(8, 16, n), rng.integers(0, 8, n), rng.integers(8, 16, n)])
    elif kind == "corner":  # across the periodic faces
        cell = np.stack([rng.integers(-1, 1, n) % s for s in shape])
    return cell + rng.random((3, n)).astype(np.float32).astype(np.float64).clip(0, 0.9999)


@pytest.mark.parametrize("shape,tile,kind,n,umax", [
    ((32, 16, 16), None, "any", 20000, 3.0), ((32, 16, 16), None, "any", 9000, 0.05),
    ((17, 13, 11), "5,3,3", "any", 7001, 1.0), ((32, 16, 16), "16,4,8", "any", 9001, 1.0),
    ((24, 16, 16), "3,8,2", "any", 9000, 1.0), ((17, 9, 10), None, "any", 5000, 1.0),
    ((16, 16, 16), None, "cell", 1, 1.0), ((16, 16, 16), None, "cell", 3, 0.01),
    ((16, 16, 16), None, "cell", 65, 0.01), ((16, 16, 16), None, "cell", 4001, 0.5),
    ((16, 16, 16), None, "tile", 2304, 0.5), ((16, 16, 16), None, "tile", 2305, 0.5),
    ((16, 16, 16), None, "tile", 9999, 2.0), ((16, 16, 16), None, "corner", 500, 2.0)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_step_against_oracle(precision, shape, tile, kind, n, umax, monkeypatch):
    if tile:
        monkeypatch.setenv("PIC_TILE", tile)
    args = (*shape, LAM / 8, LAM / 3, LAM / 2, LAM)
    g = pic.Sim(*args, periodic_x=True, precision=precision, track_ids=True)
    o = O.Sim(*args, periodic_x=True)
    inf = o.info()
    rng = np.random.default_rng(n)
    xi = _positions(kind, shape, n, rng)
    u = rng.uniform(-umax, umax, (3, n)).astype(np.float32).astype(np.float64)
    w = (rng.uniform(0.5, 1.5, n) * 0.01).astype(np.float32).astype(np.float64)
    F = (0.1 * rng.standard_normal((9,) + shape)).astype(np.float32).astype(np.float64)
    F[6:] = 0.0
    for s in (g, o):
        s.set_fields(F)
        s.set_particles(xi, u, w, np.arange(n, dtype=np.uint32))
    cells = np.floor(xi).astype(int)
    g.step(1)
    o.step(1)
    pg, po = by_id(g.particles()), by_id(o.particles())
    assert np.array_equal(pg["id"], po["id"])
    fp32 = precision == "fp32"
    assert np.abs(pg["u"] - po["u"]).max() <= (32 * EPS if fp32 else 1e-10) * max(1.0, np.abs(po["u"]).max())
    dx = np.abs(pg["xi"] - po["xi"])
    dx = np.minimum(dx, np.array(shape)[:, None] - dx)
    assert dx.max() <= (32 * EPS if fp32 else 1e-10)
    assert np.array_equal(pg["w"], po["w"])
    # sum of |w| over the cells within 3 of a node
    near = np.zeros(shape)
    np.add.at(near, tuple(cells), w)
    for axis in range(3):
        near = sum(np.roll(near, k, axis) for k in range(-3, 4))
    jc = [1 / (inf["dt"] * inf["d" + "xyz"[b]] * inf["d" + "xyz"[c]]) for b, c in ((1, 2), (0, 2), (0, 1))]
    for a in range(3):
        ref = o.field(6 + a)
        bar = 16 * EPS * jc[a] * near if fp32 else 1e-10 * np.abs(ref).max()
        assert np.all(np.abs(g.field(6 + a) - ref) <= bar), "J%s" % "xyz"[a]
    g.close()
