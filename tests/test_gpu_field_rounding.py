"""Rounding of the FP64 field update's fixed-point increments.

Where the two terms of a curl component have different scales, the finer one is
rounded to the coarser one's unit.  With E = 0 and a strong uniform Bz = 1 (no
derivative, unit of the products 2^-58 or less) beside weak random Bx, By, the increments of Ex
and Ey are that rounding: uniform on half a unit either way, its mean over 8192 cells
0 +- 0.29 / sqrt(8192) = 0.003 units.  The bar is 0.03.
"""
import numpy as np
import pytest

from paper_1204_0838_gb300 import pic, workloads as W

pytestmark = pytest.mark.gpu

LAM = W.LAMBDA0
SHAPE = (16, 16, 32)


def test_increments_of_unequal_scales_round_without_bias():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    g = pic.Sim(*SHAPE, LAM / 8, LAM / 3, LAM / 2, LAM, periodic_x=True, precision="fp64")
    rng = np.random.default_rng(8)
    F = np.zeros((9,) + SHAPE)
    F[3:5] = 2.0 ** -20 * rng.uniform(-1, 1, (2,) + SHAPE)
    F[5] = 1.0
    g.set_fields(F)
    inf = g.info()
    g.step(1)
    cz = inf["dt"] / inf["dz"]
    want = [-cz * (F[4] - np.roll(F[4], 1, 2)), cz * (F[3] - np.roll(F[3], 1, 2))]
    for c in range(2):
        err = (g.field(c) - want[c]) * 2.0 ** 58
        assert np.abs(err).max() <= 1.0
        assert abs(err.mean()) <= 0.03, (c, err.mean())
    g.close()
