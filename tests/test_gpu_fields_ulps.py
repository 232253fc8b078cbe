"""Velocities in units in the last place: where the fixed-point sums are exact (FP64
populations of [2^-6, 1): whole multiples of 2^-58; FP32 deviations of 2^-36 and more: of
2^-60) the quotient is rounded once, on a reciprocal good to 2^-56: half a unit, and up to
an eighth.  Velocities from 2^-50 to 0.2, densities over the range of that form."""
import numpy as np
import pytest

import paper_1303_0625_gb300 as G

pytestmark = pytest.mark.gpu

CX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])[:, None, None]
CY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])[:, None, None]
WT = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_velocity_within_five_eighths_of_a_unit(precision):
    nx, ny = 512, 400
    rng = np.random.default_rng(8)
    f = WT * rng.uniform(0.6, 1.9, (1, ny, nx)) * (1 + 0.01 * rng.uniform(-1, 1, (9, ny, nx)))
    small = rng.uniform(size=(ny, nx)) < 0.7  # opposite populations closer, down to a few units
    for i, k in ((1, 3), (2, 4), (5, 7), (6, 8)):
        near = f[i] + np.exp2(-rng.integers(4, 51, (ny, nx))) * rng.uniform(-1, 1, (ny, nx))
        f[k] = np.where(small & (near >= 2.0 ** -6), near, f[k])
    if precision == "fp32":
        d = (f - WT).astype(np.float32)
        d[np.abs(d) < 2.0 ** -35] = 0.0
        f = d.astype(np.float64) + WT
        exact = (f - WT).astype(np.float32).astype(np.longdouble)  # as stored
        rho = 1 + exact.sum(axis=0)
    else:
        exact = f.astype(np.longdouble)
        rho = exact.sum(axis=0)
    g = G.Lattice(nx, ny, 0.8, precision=precision)
    g.set_f(f)
    _, ux, uy = g.fields()
    inside = (rho >= 0.5) & (rho < 2)
    for u, c in ((ux, CX), (uy, CY)):
        want = (c * exact).sum(axis=0) / rho
        unit = np.spacing(np.abs(want).astype(np.float64))
        assert (np.abs(u - want) <= 0.63 * unit)[inside].all(), (np.abs(u - want) / unit)[inside].max()
