"""The particle diagnostics read four particles per thread and round, and the
emittance passes over particles below gamma_min without the exact test: particle
counts around the batches, thresholds below 1, at a particle's own gamma, one
rounding below it and above all of them, against the FP64 oracle.

Tolerance: the sums are FP64 sums of at most 1e5 terms in any order, 1e5 x 2^-53
= 1e-11 relative, 1e-10 allowed; the emittance's square is a difference of products
of such sums, none above the square of the largest momentum times the largest
distance from the axis.  FP32 handles hold the spacings in FP32: the oracle's
emittance is scaled by that rounding.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1204_0838_gb300 import pic, workloads as W

pytestmark = pytest.mark.gpu

LAM = W.LAMBDA0
MC2 = 0.51099895069
BINS, E_MAX = 37, 9.0


@pytest.mark.parametrize("n", [1, 255, 1025, 100003])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_particle_diagnostics_against_the_oracle(precision, n):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    shape = (16, 12, 20)
    args = (*shape, LAM / 8, LAM / 3, LAM / 2, LAM)
    g = pic.Sim(*args, periodic_x=True, precision=precision)
    o = O.Sim(*args, periodic_x=True)
    rng = np.random.default_rng(n)
    # |u| from the middles of the spectrum's bins, no particle near an edge
    gam = 1.0 + (rng.integers(0, BINS + 5, n) + 0.5) * (E_MAX / BINS) / MC2
    v = rng.standard_normal((3, n))
    u = v / np.sqrt((v ** 2).sum(0)) * np.sqrt(gam ** 2 - 1.0)
    u[:, 0] = (0.0, 0.75, 0.0)  # gamma 1.25 exactly
    u = u.astype(np.float32).astype(np.float64)
    xi = (rng.random((3, n)).astype(np.float32) * 0.999 + rng.integers(0, 12, (3, n))).astype(np.float64)
    xi = np.floor(xi) + (xi - np.floor(xi)).astype(np.float32)
    w = rng.uniform(0.5, 1.5, n).astype(np.float32).astype(np.float64)
    for s in (g, o):
        s.set_particles(xi, u, w, np.arange(n, dtype=np.uint32))
    near = float(np.sqrt(1.0 + (u[:, -1] ** 2).sum()))  # another particle's gamma
    scale = np.abs(u).max() * 0.5 * max(shape[1] * LAM / 3, shape[2] * LAM / 2)
    spacing = 2 * np.pi * np.array([1 / 3, 1 / 2])  # times omega0 / c
    held = spacing.astype(np.float32) / spacing if precision == "fp32" else 1.0
    for gmin in (0.0, 0.5, 1.25, np.nextafter(1.25, 0.0), near * (1 - 1e-7), 30.0, 1e30):
        a, b = g.diag("emittance", 2, gmin), o.diag("emittance", 2, gmin) * held
        assert np.all(np.abs(a ** 2 - b ** 2) <= 1e-10 * scale ** 2), gmin
    for gmin in (0.0, 1.2, 4.1, 1e30):
        a, b = g.diag("charge", 1, gmin), o.diag("charge", 1, gmin)
        assert np.all(np.abs(a - b) <= 1e-10 * np.abs(b)), gmin
    a, b = g.diag("spectrum", BINS, 0.0, E_MAX), o.diag("spectrum", BINS, 0.0, E_MAX)
    assert np.all(np.abs(a - b) <= 1e-10 * np.abs(b).max())
    g.close()


@pytest.mark.parametrize("nb,lo,hi", [(1, -2.0, 2.0), (40, -2.0, 2.0), (64, -0.7, 1.9), (100000, -2.0, 2.0)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_phase_space_bins_are_those_of_the_fp64_quotient(precision, nb, lo, hi):
    """Momenta on the bins' edges, one rounding off them, anywhere, and outside; weights
    are small whole numbers, so that the sums are exact."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    shape = (16, 8, 8)
    args = (*shape, LAM / 8, LAM / 3, LAM / 2, LAM)
    g = pic.Sim(*args, periodic_x=True, precision=precision)
    rng = np.random.default_rng(nb)
    n = 6000
    real = np.float32 if precision == "fp32" else np.float64
    edge = (lo + rng.integers(0, nb + 1, n) * ((hi - lo) / nb)).astype(real)
    ux = np.concatenate([edge, np.nextafter(edge, real(9)), np.nextafter(edge, real(-9)),
                         rng.uniform(lo - 0.1, hi + 0.1, n).astype(real)]).astype(np.float64)
    xi = rng.random((3, ux.size)) * np.array(shape)[:, None] * 0.99
    w = rng.integers(1, 8, ux.size).astype(np.float64)
    u = np.zeros((3, ux.size))
    u[0] = ux
    g.set_particles(xi, u, w, np.arange(ux.size, dtype=np.uint32))
    got = g.diag("phase_x_px", shape[0] * nb, lo, hi).reshape(shape[0], nb)
    ref = np.zeros((shape[0], nb))
    inside = (ux >= lo) & (ux < hi)
    b = np.minimum(np.floor((ux[inside] - lo) / (hi - lo) * nb).astype(int), nb - 1)
    np.add.at(ref, (np.floor(xi[0][inside]).astype(int), b), w[inside])
    unit = got.sum() / ref.sum()
    assert np.all(np.abs(got - ref * unit) <= 1e-9 * unit)
    g.close()


@pytest.mark.parametrize("shape", [(16, 4, 4), (17, 9, 33), (70, 96, 100)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_field_energy_against_the_oracle(precision, shape):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    args = (*shape, LAM / 8, LAM / 3, LAM / 2, LAM)
    g = pic.Sim(*args, periodic_x=True, precision=precision)
    o = O.Sim(*args, periodic_x=True)
    F = np.random.default_rng(5).standard_normal((9,) + shape).astype(np.float32).astype(np.float64)
    F[6:] = 0.0
    for s in (g, o):
        s.set_fields(F)
    a, b = g.diag("field_energy"), o.diag("field_energy")
    assert np.all(np.abs(a - b) <= 1e-9 * np.abs(b))  # 4e6 terms x 2^-53
    g.close()
