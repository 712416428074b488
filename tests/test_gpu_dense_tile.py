"""A tile of many passes adds its current to the grid once: each add rounds to FP32.

200,000 particles of one cell that all move towards larger x, y, z, no others, against
the sum in FP64 of the currents of the same particles in 100 steps of 2,000, one pass
each.  The particles' contributions are the same numbers on both sides, so that what
differs is, relative to a value (rms over the nodes where J is at least 0.005 B, B =
|q jc| sum |w|):
- one rounding of the dense tile's value, 2^-24 / sqrt 3, and of the 100 parts', a tenth
  of that;
- the rounding of 200,000 contributions to integers of unit 2^-41 B or less, 0.3
  units each and without sign: 447 x 0.3 x 2^-41 / 0.005 = 2^-26.4.
Together 0.7 x 2^-24; the bar is 2^-24.  (One add per pass, 87 of them, rounds partial
sums that grow to the value: sqrt(87 / 3) / sqrt 12 = 1.5 units of the last place, 2^-24
to 2^-23 of the value each.)
"""
import numpy as np
import pytest

from paper_1204_0838_gb300 import pic, workloads as W

pytestmark = pytest.mark.gpu

LAM = W.LAMBDA0
SHAPE = (16, 16, 16)


def test_current_of_a_dense_tile_is_rounded_once(monkeypatch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    monkeypatch.setenv("PIC_TILE", "8,8,8")
    rng = np.random.default_rng(12)
    n, part = 200000, 2000
    xi = np.array([[10], [4], [12]]) + rng.random((3, n)).astype(np.float32).astype(np.float64).clip(0, 0.9999)
    u = rng.uniform(0.2, 0.6, (3, n)).astype(np.float32).astype(np.float64)
    w = np.full(n, float(np.float32(1e-6)))
    g = pic.Sim(*SHAPE, LAM / 8, LAM / 3, LAM / 2, LAM, periodic_x=True, precision="fp32", max_particles=n)

    def current(sel):
        g.set_fields(np.zeros((9,) + SHAPE))
        g.set_particles(xi[:, sel], u[:, sel], w[sel])
        g.step(1)
        return np.stack([g.field(c) for c in (6, 7, 8)])

    inf = g.info()
    dense = current(slice(0, n))
    ref = sum(current(slice(a, a + part)) for a in range(0, n, part))
    rel = []
    for a, (b, c) in enumerate(((1, 2), (0, 2), (0, 1))):
        big = np.abs(ref[a]) >= 0.005 * w.sum() / (inf["dt"] * inf["d" + "xyz"[b]] * inf["d" + "xyz"[c]])
        rel.append(dense[a][big] / ref[a][big] - 1.0)
    assert all(r.size for r in rel)
    assert np.sqrt(np.mean(np.concatenate(rel) ** 2)) <= 2.0 ** -24
    g.close()
