"""The FP64 field update runs blocks of finite values in fixed point and blocks
that hold a NaN or an infinity in FP64: non-finite values must spread over the
same cells as in the FP64 oracle, and the finite rest must agree with it.  Sizes
at the edges of the 4x8x32 blocks.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1204_0838_gb300 import pic, workloads as W

pytestmark = pytest.mark.gpu

LAM = W.LAMBDA0


@pytest.mark.parametrize("shape,comp,value", [((17, 9, 33), 1, np.inf), ((16, 8, 32), 0, np.nan),
                                              ((20, 17, 64), 5, -np.inf), ((18, 4, 31), 3, np.nan)])
def test_non_finite_values_spread_as_in_fp64(shape, comp, value):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    args = (*shape, LAM / 8, LAM / 3, LAM / 2, LAM)
    g = pic.Sim(*args, periodic_x=True, precision="fp64")
    o = O.Sim(*args, periodic_x=True)
    F = 0.1 * np.random.default_rng(3).standard_normal((9,) + shape)
    F[6:] = 0.0
    F[comp, 5, 3, 7] = value
    for s in (g, o):
        s.set_fields(F)
        s.step(1)
    for c in range(6):
        a, b = g.field(c), np.asarray(o.field(c))
        fine = np.isfinite(b)
        assert np.array_equal(fine, np.isfinite(a)), c
        assert np.abs(a[fine] - b[fine]).max() <= 1e-12 * np.abs(b[fine]).max()
    g.close()
