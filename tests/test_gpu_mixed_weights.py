"""FP32 current of light particles in a tile that also holds a heavy one, against
the FP64 oracle.

Tolerance (eps = 2^-24), per node: 16 eps sum |q w jc| over the particles whose
window can reach it, as for equal weights (test_gpu_push.py), and for each of them
the rounding of its integer contribution: the tile's unit is at most 2^-41 of
B = 1.001 |q jc| sum |w| over the tile, a contribution is rounded by half a unit
and its factor P by at most another half times A <= 0.45.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1204_0838_gb300 import pic, workloads as W

pytestmark = pytest.mark.gpu

LAM = W.LAMBDA0
EPS = 2.0 ** -24
SHAPE = (16, 16, 16)


@pytest.mark.parametrize("tile", ["8,8,8", "8,8,16"])
@pytest.mark.parametrize("per_cell,umax", [(1, 0.02), (2, 0.3), (3, 2.0), (40, 0.3)])
@pytest.mark.parametrize("ratio", [1.0, 30.0, 1e4, 1e6, 1e8])
def test_light_particles_beside_a_heavy_one(ratio, per_cell, umax, tile, monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    monkeypatch.setenv("PIC_TILE", tile)
    args = (*SHAPE, LAM / 8, LAM / 3, LAM / 2, LAM)
    g = pic.Sim(*args, periodic_x=True, precision="fp32")
    o = O.Sim(*args, periodic_x=True)
    inf = o.info()
    rng = np.random.default_rng(per_cell)
    cells = np.stack(np.meshgrid(*3 * [[8, 9, 10]], indexing="ij")).reshape(3, -1)  # reach 6 .. 13
    cells = np.concatenate([np.repeat(cells, per_cell, axis=1), [[15], [15], [15]]], axis=1)  # the heavy one: 13 .. 18
    n = cells.shape[1]
    xi = cells + rng.random((3, n)).astype(np.float32).astype(np.float64).clip(0, 0.9999)
    u = rng.uniform(0.2 * umax, umax, (3, n)).astype(np.float32).astype(np.float64)
    w = np.full(n, 1e-3)
    w[-1] *= ratio
    w = w.astype(np.float32).astype(np.float64)
    for s in (g, o):
        s.set_particles(xi, u, w)
        s.step(1)
    near, count = np.zeros(SHAPE), np.zeros(SHAPE)
    np.add.at(near, tuple(cells), w)
    np.add.at(count, tuple(cells), 1.0)
    for axis in range(3):
        near = sum(np.roll(near, k, axis) for k in range(-3, 4))
        count = sum(np.roll(count, k, axis) for k in range(-3, 4))
    unit = 2.0 ** -41 * 1.001 * w.sum()
    for a, (b, c) in enumerate(((1, 2), (0, 2), (0, 1))):
        jc = 1 / (inf["dt"] * inf["d" + "xyz"[b]] * inf["d" + "xyz"[c]])
        err = np.abs(g.field(6 + a) - o.field(6 + a))
        assert np.all(err <= jc * (16 * EPS * near + 0.75 * unit * count)), "J%s" % "xyz"[a]
    g.close()
