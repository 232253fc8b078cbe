"""The autotuner chooses between launch shapes, not between names of the same one."""
import pytest

import workloads as W
from _pairs import make_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,collision,boundary,shapes,overlaps", [
    ("fp32", 0, 0, {0, 1, 2}, {1}), ("fp32", 1, 0, {0}, {1}), ("fp32", 0, 1, {0, 1, 2}, {0, 1}),
    ("fp64", 0, 0, {0, 1, 2}, {0, 1}), ("fp64", 1, 0, {0}, {0, 1}),
    ("fp16", 0, 1, {0, 1, 2}, {0, 1}), ("fp16", 1, 0, {0}, {0, 1}), ("fp16", 0, 0, set(range(6)), {0, 1})])
def test_autotune_reports_the_first_of_equal_shapes(precision, collision, boundary, shapes, overlaps):
    disk = dict(cx=60.0, cy=40.0, r=9.0, vx=0.02, vy=0.01, omega=0.0, rho_s=1.5, motion=0)
    w = dict(nx=128, ny=80, tau=0.8, rho0=1.0, bc_x=W.PERIODIC, bc_y=W.PERIODIC, u0=(0.0, 0.0),
             wall_ux=(0.0, 0.0), body_force=(0.0, 0.0), rho_w_mode=W.RHOW_CONST, refill=1,
             collision=collision, boundary=boundary, solids=[disk])
    g = make_gpu(w, precision, ring=8)
    for _ in range(6):
        t = g.t
        assert g.autotune(1) in shapes and int(g.force_overlap()) in overlaps
        assert g.t == t + 24
