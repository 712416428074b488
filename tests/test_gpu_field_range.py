"""The FP64 field update on blocks whose values span many decades, against the FP64
oracle, cell by cell: weak cells keep their relative precision beside strong ones.

The amplitude falls along one axis by a constant factor per cell to the middle of the
grid and rises again.  Tolerance per cell: 2^-48 of the largest field value within five
cells (E takes H = B - dt/2 curl' E within one cell and B takes that E: four cells; the
cells that vouch for the precision of one in fixed point lie at most two further along
z, and reach one less): either side forms about ten sums and products, each rounded by
2^-53 of it or, in fixed point, by less than 3 x 2^-51.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1204_0838_gb300 import pic, workloads as W

pytestmark = pytest.mark.gpu

LAM = W.LAMBDA0


@pytest.mark.parametrize("solver", ["perfect", "yee"])
@pytest.mark.parametrize("shape,axis,factor,pml", [
    ((17, 33, 30), 1, 1e-3, 0), ((16, 9, 70), 2, 0.1, 0), ((16, 8, 160), 2, 0.4, 0), ((40, 9, 33), 0, 1e-4, 0),
    ((18, 40, 34), 1, 1e-3, 6), ((16, 18, 70), 2, 0.1, 6)])
def test_weak_cells_beside_strong_ones(shape, axis, factor, pml, solver):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    args = (*shape, LAM / 8, LAM / 3, LAM / 2, LAM)
    g = pic.Sim(*args, periodic_x=True, precision="fp64", pml=pml, solver=solver)
    o = O.Sim(*args, periodic_x=True, pml=pml, solver=solver)
    rng = np.random.default_rng(6)
    n = shape[axis]
    amp = factor ** np.minimum(np.arange(n), n - np.arange(n)).astype(float)
    F = rng.standard_normal((9,) + shape) * amp.reshape([-1 if a == axis else 1 for a in range(3)])
    F[:3] *= np.array([1.0, 1e-5, 1e-2]).reshape(3, 1, 1, 1)  # components of unequal size
    F[6:] = 0.0
    for s in (g, o):
        s.set_fields(F)
        s.step(1)
    loc = np.abs(F[:6]).max(axis=0)
    for a in range(3):
        loc = np.max([np.roll(loc, k, a) for k in range(-5, 6)], axis=0)
    for c in range(6):
        err = np.abs(g.field(c) - np.asarray(o.field(c)))
        assert np.all(err <= 2.0 ** -48 * loc), (pic.COMPONENTS[c], (err / loc).max() * 2.0 ** 48)
    g.close()
