"""Edges of the row kernel of the FP64 and FP32 modes and of the link kernels.

The row kernel puts walls, periodic wraps and open columns in place in the lanes that
hold them: domain widths around multiples of 32 lanes times 1, 2 and 4 nodes (the last
column in the first lane of a warp, inside a lane's nodes, at a warp's end), every edge
kind, every width per thread.  The link kernels walk a disk's rows 128 at a time and its
links in chunks: a disk of more than 128 rows, tiny disks, disks in reach of each other
and across the periodic edge.  Bounds: those of the parity tests (FP64 1e-12, FP32
forces 1e-5).
"""
import numpy as np
import pytest

import workloads as W
from _pairs import force_rel, make_gpu, make_oracle, run_pair, seeded_f

pytestmark = pytest.mark.gpu

EDGES = {"periodic": (W.PERIODIC, W.PERIODIC), "channel": (W.PERIODIC, W.WALL),
         "box": (W.WALL, W.WALL), "open": (W.OPEN, W.WALL)}


def _disk(cx, cy, r, vx=0.0, vy=0.0, om=0.0, motion=0):
    return dict(cx=cx, cy=cy, r=r, vx=vx, vy=vy, omega=om, rho_s=1.5, motion=motion)


def _check(w, steps, precision, **kw):
    o, g, ref, got = run_pair(w, steps, precision=precision, perturb=1, **kw)
    radii = [s["r"] for s in w["solids"]]
    assert np.array_equal(o.owner(), g.owner())
    assert force_rel(got, ref, radii) <= (1e-12 if precision == "fp64" else 1e-5)
    fl = o.owner() < 0
    tol = 1e-12 if precision == "fp64" else 2e-6
    assert np.abs(g.get_f()[:, fl] - o.get_f()[:, fl]).max() <= tol


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nx", [32, 33, 64, 65, 66, 127, 129])
@pytest.mark.parametrize("edges", sorted(EDGES))
def test_row_edges_match_oracle(edges, nx, precision):
    bx, by = EDGES[edges]
    w = dict(nx=nx, ny=26, tau=0.7, rho0=1.0, bc_x=bx, bc_y=by, u0=(0.0, 0.0),
             wall_ux=(0.01, 0.03) if by == W.WALL and bx != W.OPEN else (0.0, 0.0),
             body_force=(0.0, 0.0), inflow_umax=0.04 if bx == W.OPEN else 0.0,
             rho_w_mode=W.RHOW_LOCAL if nx % 2 else W.RHOW_CONST, refill=1,
             solids=[_disk(nx / 2 + 0.3, 13.2, 4.3, 0.0 if bx == W.OPEN else 0.05, 0.01, 0.004)])
    for v in range(3):
        _check(w, 12, precision, variant=v)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("solids", ["tall", "tiny", "close", "edge", "many"])
def test_links_of_a_disk_match_oracle(solids, boundary, precision):
    nx, ny = (170, 165) if solids == "tall" else (96, 70)
    disks = {
        "tall": [_disk(84.3, 82.1, 70.4, 0.04, -0.03, 0.0003)],
        "tiny": [_disk(20.2, 20.7, 0.6, 0.05, 0.02), _disk(50.0, 40.0, 1.0, 0.03, 0.04)],
        "close": [_disk(30.0, 30.0, 9.0, 0.04, 0.0), _disk(50.2, 31.0, 9.0, -0.04, 0.01, 0.01),
                  _disk(40.0, 50.0, 8.0, 0.0, -0.05)],
        "edge": [_disk(1.2, 35.0, 7.3, 0.06, 0.0, 0.01), _disk(60.0, 68.9, 6.0, 0.02, 0.05)],
        "many": [_disk(8.0 + 16.0 * (k % 6), 9.0 + 17.0 * (k // 6), 5.0 + 0.1 * k, 0.03, -0.02, 0.001 * k)
                 for k in range(24)],
    }[solids]
    w = dict(nx=nx, ny=ny, tau=0.7, rho0=1.0, bc_x=W.PERIODIC, bc_y=W.PERIODIC, u0=(0.0, 0.0),
             wall_ux=(0.0, 0.0), body_force=(0.0, 0.0), rho_w_mode=W.RHOW_LOCAL if boundary else
             W.RHOW_CONST, refill=1, boundary=boundary, solids=disks)
    _check(w, 30, precision)


@pytest.mark.parametrize("overlap", [0, 1])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nmoving", [1, 2, 16, 17])
def test_few_moving_solids_match_oracle(nmoving, precision, overlap):
    """Up to 16 moving solids are re-rasterised by one cluster of blocks, with the ring
    in the same launch where nothing runs beside it; 17 by a cooperative grid."""
    disks = [_disk(10.3 + 18.0 * (k % 6), 10.1 + 17.0 * (k // 6), 5.2 + 0.13 * k, 0.05 - 0.005 * k, 0.03, 0.002 * k)
             for k in range(nmoving)] + [_disk(100.0, 61.0, 4.4)]
    w = dict(nx=111, ny=71, tau=0.8, rho0=1.0, bc_x=W.PERIODIC, bc_y=W.PERIODIC, u0=(0.0, 0.0),
             wall_ux=(0.0, 0.0), body_force=(0.0, 0.0), rho_w_mode=W.RHOW_CONST, refill=1, solids=disks)
    o, g = make_oracle(w), make_gpu(w, precision, ring=40)
    g.set_force_overlap(bool(overlap))
    f0 = seeded_f(w, 1)
    o.set_f(f0)
    g.set_f(f0)
    ref, got = o.step(40), g.step_record(40)
    assert np.array_equal(o.owner(), g.owner())
    assert force_rel(got, ref, [s["r"] for s in disks]) <= (1e-12 if precision == "fp64" else 1e-5)
    fl = o.owner() < 0
    assert np.abs(g.get_f()[:, fl] - o.get_f()[:, fl]).max() <= (1e-12 if precision == "fp64" else 2e-6)
