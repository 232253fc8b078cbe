"""Density and velocity of arbitrary populations against extended precision: densities
inside the range of the fixed-point form, at its ends and outside, velocities down to a
single unit of the stored form, with and without a body force.

Bounds: the fixed-point sums are exact to 9 units of 2^-61 (FP64: 2^-59) and the results
rounded once; the FP64 form rounds each of at most 9 additions (2^-53 of sum |f|) and a
division.  Both are within 2e-15 (1 + sum |f|) / rho."""
import numpy as np
import pytest

import paper_1303_0625_gb300 as G
from paper_1303_0625_gb300 import lbm as L

pytestmark = pytest.mark.gpu

CX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])
CY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])
WT = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("body", [(0.0, 0.0), (3e-5, -0.01), (0.7, 0.0)])
def test_fields_of_any_populations(precision, body):
    nx, ny = 65, 40
    rng = np.random.default_rng(5)
    scale = np.exp(rng.uniform(np.log(1e-9), np.log(0.3), (1, ny, nx)))
    f = WT[:, None, None] * rng.choice([1.0, 0.4999999, 0.5, 1.9999999, 2.0, 0.1, 4.0], (1, ny, nx), p=[.6, .1, .1, .05, .05, .05, .05])
    f = f + WT[:, None, None] * scale * rng.uniform(-1, 1, f.shape)
    f[:, 3, 5] = WT          # at rest
    f[1, 4, 6] += 2.0 ** -30
    g = G.Lattice(nx, ny, 0.8, body_force=body, precision=precision)
    g.set_f(f)
    v = g.get_f().astype(np.longdouble)  # as stored
    rho, ux, uy = g.fields()
    r = v.sum(axis=0)
    tol = 2e-15 * (1 + np.abs(v).sum(axis=0)) / r
    assert (np.abs(rho - r) <= tol * r).all()
    for u, c, b in ((ux, CX, body[0]), (uy, CY, body[1])):
        want = ((c[:, None, None] * v).sum(axis=0) - np.longdouble(b) / 2) / r
        assert (np.abs(u - want) <= tol).all(), np.abs(u - want).max()
