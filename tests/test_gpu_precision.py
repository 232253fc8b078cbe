"""What the arithmetic of the kernels loses to rounding.

Mass and momentum: advection and collision conserve both; what the constants' rounding
lets drift is systematic.  Bound: what weights rounded to nearest would give, 9 fl(1/9) - 1
= 2^-27 of the deviation (3 w_i over e_i e_i: of the momentum), times omega, a step.  Omega
times weight rounded one by one lets them drift by up to ten times as much.  FP64: mass
drifts by the weights' rounding, -2^-54 (of all of it, not of the deviation), within 10%:
rounding at random leaves 1% over 6144 nodes and 100 steps, (1 - omega) f + omega (...) 20%.

Force records, relative 2-norm over 100 steps of eight seeded boxes with two disks against
the FP64 oracle.  Bound: the geometric mean of the errors that nine separate FP32 equilibria
relaxed as g - omega (g - eq) gave next to the disks, measured on the same boxes, plus 10%.

Batches: first force records of 24 channels (nothing but the links' terms and their sums),
in units of rho0 r.  Bound: rms errors that FP64 sums over the lanes gave, measured on the
same channels, plus 10% (FP32 sums: 1.3 to 2.2 times as much).
"""
import math

import numpy as np
import pytest

import paper_1303_0625_gb300 as G
import workloads as W
from _pairs import PREC, make_gpu, make_oracle, seeded_f

pytestmark = pytest.mark.gpu

CX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])[:, None, None]
CY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])[:, None, None]
WT = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]


def _box(tau, nx=96, ny=64, **kw):
    w = dict(nx=nx, ny=ny, tau=tau, rho0=1.0, bc_x=W.PERIODIC, bc_y=W.PERIODIC, u0=(0.0, 0.0),
             wall_ux=(0.0, 0.0), body_force=(0.0, 0.0), rho_w_mode=W.RHOW_CONST, refill=1, solids=[])
    w.update(kw)
    return w


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("tau", [0.55, 0.8, 0.85])
def test_fp32_mass_and_momentum_do_not_drift(tau, variant):
    w = _box(tau, u0=(0.1, -0.1))
    g = make_gpu(w, "fp32")
    g.set_kernel_variant(variant)
    g.set_f(1.1 * seeded_f(w, 2))

    def sums():
        d = g.get_f() - WT
        return np.array([math.fsum((c * d).ravel()) for c in (1.0, CX, CY)])

    before = sums()
    g.step(200)
    assert (np.abs(sums() - before) <= 200 / tau * 2.0 ** -27 * np.abs(before)).all()


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("tau", [0.6, 1.2])
def test_fp64_mass_drifts_by_the_weights_rounding(tau, variant):
    w = _box(tau)
    g = make_gpu(w, "fp64")
    g.set_kernel_variant(variant)
    g.set_f(seeded_f(w, 2))
    before = math.fsum(g.get_f().ravel())
    g.step(100)
    want = -100 / tau * 2.0 ** -54
    assert abs((math.fsum(g.get_f().ravel()) - before) / before - want) <= 0.1 * abs(want)


def _flow(w, seed):
    """Equilibrium of a smooth velocity field, a few waves each way."""
    rng = np.random.default_rng(seed)
    x, y = (np.arange(n) / n * 2 * np.pi for n in (w["nx"], w["ny"]))
    ux, uy, rho = np.zeros((w["ny"], w["nx"])), np.zeros((w["ny"], w["nx"])), np.ones((w["ny"], w["nx"]))
    for _ in range(3):
        k, m = rng.integers(1, 4, 2)
        a, b, c = rng.uniform(0, 2 * np.pi, 3)
        ux += 0.006 * np.sin(m * y + a)[:, None] * np.cos(k * x + b)[None]
        uy += 0.006 * np.sin(k * x + c)[None] * np.cos(m * y + a)[:, None]
        rho += 0.001 * np.cos(m * y + c)[:, None] * np.sin(k * x + a)[None]
    e = CX * ux + CY * uy
    return rho * WT * (1 + 3 * e + 4.5 * e * e - 1.5 * (ux * ux + uy * uy))


@pytest.mark.parametrize("boundary,motion,bound", [
    (0, "rest", 6.868e-6), (0, "spin", 7.795e-7), (0, "move", 1.439e-6),
    (1, "rest", 8.847e-6), (1, "spin", 8.448e-7), (1, "move", 1.502e-6)])
def test_fp32_force_records(boundary, motion, bound):
    errors = []
    for seed in range(8):
        rng = np.random.default_rng([seed, 7])
        vx, vy, om = dict(rest=(0.0, 0.0, 0.0), spin=(0.0, 0.0, 0.002), move=(0.03, 0.02, 0.001))[motion]
        disks = [dict(cx=24 + 48 * k + rng.uniform(-2, 2), cy=40 + rng.uniform(-10, 10), r=rng.uniform(7, 14),
                      vx=vx, vy=vy, omega=om, rho_s=1.5, motion=0) for k in range(2)]
        w = _box(rng.uniform(0.7, 0.95), ny=80, boundary=boundary, solids=disks)
        o, g, f = make_oracle(w), make_gpu(w, "fp32", ring=100), _flow(w, seed)
        o.set_f(f)
        g.set_f(f)
        ref = o.step(100)
        errors.append(np.linalg.norm(g.step_record(100) - ref) / np.linalg.norm(ref))
    assert np.exp(np.mean(np.log(errors))) <= 1.1 * bound, errors


@pytest.mark.parametrize("seed,nx,ny,bound", [
    (47, (40, 150), (24, 64), 1.953e-8), (47, (200, 400), (100, 200), 1.250e-8),
    (48, (40, 150), (24, 64), 1.903e-8), (49, (200, 400), (100, 200), 8.852e-9)])
def test_fp32_batch_sums_of_links(seed, nx, ny, bound):
    ws = W.cylinder_sweep(24, seed_offset=seed, nx_range=nx, ny_range=ny)
    b = G.Batch.from_workloads(ws, precision=PREC["fp32"], force_ring=8)
    b.run(1)
    off = [(b.case(k).forces(0, 1) - make_oracle(w).step(1))[0, 0, 1, :2] / w["solids"][0]["r"]
           for k, w in enumerate(ws)]
    assert np.sqrt(np.mean(np.square(off))) <= 1.1 * bound
