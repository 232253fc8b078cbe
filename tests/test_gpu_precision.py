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


def _records(w, precision, overlap, steps, save=None, load=None):
    g = make_gpu(w, precision, ring=40)
    g.set_force_overlap(overlap)
    if load is None:
        g.set_f(seeded_f(w, 3))
    else:
        g.load(load)
    rec = g.step_record(steps)
    return rec, g.get_f(), g.solids(), g.save() if save else None


@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("r", [15.0, 30.0, 51.0, 70.0, 151.0])  # FP64 parts: 5, 10, 16 chunks; two turns of rows; none
def test_forces_do_not_depend_on_where_they_are_summed(r, precision, boundary):
    """The link sums of a disk come out bit for bit whether one block takes them or several,
    with the per-solid work beside the advection-collision kernel and before it, and a free
    disk's path with them; a state saved one way goes on the other."""
    n = int(4 * r + 30)
    disks = [dict(cx=n / 4, cy=n / 4 + 3.3, r=r / 2, vx=0.02, vy=0.01, omega=0.001, rho_s=1.5, motion=0),
             dict(cx=5 * n / 8, cy=5 * n / 8, r=r, vx=0.01, vy=-0.02, omega=0.0, rho_s=1.2, motion=1)]
    w = _box(0.8, n, n, gravity=(0.0, -1e-5), boundary=boundary, solids=disks)
    beside, before = (_records(w, precision, on, 30, save=True) for on in (True, False))
    for a, b in zip(beside[:3], before[:3]):
        assert np.array_equal(a, b)
    again = [_records(w, precision, on, 10, load=beside[3]) for on in (True, False)]
    for a, b in zip(*again):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("precision,few", [("fp64", 32), ("fp64", 255), ("fp32", 255)])
def test_forces_do_not_depend_on_the_number_of_solids(precision, few):
    """Another disk, far from the first, changes the number of blocks that share a disk's links."""
    one = dict(cx=40.2, cy=41.7, r=22.0, vx=0.02, vy=0.01, omega=0.002, rho_s=1.5, motion=0)
    small = [dict(cx=100.0 + 16 * (k % 32), cy=20.0 + 16 * (k // 32), r=4.0, vx=0.0, vy=0.0, omega=0.0, rho_s=1.0, motion=0)
             for k in range(few)]
    first = []
    for k in (few - 1, few):
        w = _box(0.8, 640, 180, solids=[one] + small[:k])
        g = make_gpu(w, precision, ring=4)
        g.set_f(seeded_f(w, 4))
        first.append(g.step_record(1)[:, 0])
    assert np.array_equal(*first)


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
def test_a_state_may_hold_larger_disks_than_its_context(precision):
    def box(r):
        return _box(0.8, 420, 410, solids=[dict(cx=210.3, cy=205.1, r=r, vx=0.01, vy=0.02, omega=0.0, rho_s=1.5, motion=0)])

    g = make_gpu(box(190.0), precision, ring=40)
    g.set_f(seeded_f(box(190.0), 5))
    g.step(5)
    state = g.save()
    h = make_gpu(box(3.0), precision, ring=40)
    h.load(state)
    assert np.array_equal(g.step_record(10), h.step_record(10))
    assert np.array_equal(g.get_f(), h.get_f())
