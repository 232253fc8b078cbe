"""The work that users of this framework have it do, as cases to be timed.

Three kinds of case, each through the public entry points:

  domain    one lattice-Boltzmann domain with disks (Lattice): a number of steps, then what
            a simulation program reads: both force records on the host, the fields and the
            owner map on the device, the solids' state
  channels  a batch of independent open channels (Batch): a block of steps between two
            readings of the drag, then every case's fields
  net       the warm-start network (UNet): a forward pass, or training steps

Results come back in the type that the run stores its populations in (the C API widens all
of them to FP64): FP64 runs as FP64, FP32 runs as FP32, FP16 runs as FP16, density as its
deviation from rho0.  The network's own results are FP32.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1303_0625_gb300 as G
from paper_1303_0625_gb300 import lbm as L

KEPT = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16}
BYTES = {"fp64": 8, "fp32": 4, "fp16": 2}
TUNE_STEPS = 12 * (1 + 4)  # steps that Lattice.autotune(4) advances the domain by


def listed():
    return [
        # The Galilean-pair channel of the accuracy studies: one disk moving through fluid at
        # rest, FP64, local wall density, 100-step graphs: the smallest domain in use.
        _domain("galilean_pair_fp64", 256, 128, "channel", 1, 12, 12, precision="fp64",
                rho_w="local", tau=0.8, steps=100, graph=100, speed=0.05),
        # A small ragged periodic box, direct launches, the forces read every 20 steps: a
        # program under development, or one that couples the disks to something else.
        _domain("ragged_box_fp32", 321, 197, "periodic", 6, 6, 14, steps=20, spin=0.001),
        # The paper's sedimentation channel at its own size (120 x 1200, d = 30, interpolated
        # boundary, density ratio 1.03), FP64, as the Galilean experiment runs it.
        _domain("paper_channel_fp64", 1200, 120, "channel", 1, 15, 15, precision="fp64",
                boundary="interpolated", motion="free", density=1.03, gravity=4.03e-4,
                tau=0.6, steps=100, graph=100),
        # FP64 on a mid-size suspension: the reference mode of the precision studies.
        _domain("suspension_2048_fp64", 2048, 1024, "periodic", 125, 8, 20, precision="fp64", steps=10),
        # The headline workload: 8192 x 4096, 2000 moving disks, FP32, autotuned (viscosity and
        # speed such that the flow between close disks stays stable at any horizon).
        _domain("suspension_8192_fp32", 8192, 4096, "periodic", 2000, 8, 20, tau=0.8, speed=0.03,
                steps=20, tune=True),
        # The same in FP16 storage, which is used where memory or bandwidth counts most.
        _domain("suspension_8192_fp16", 8192, 4096, "periodic", 2000, 8, 20, precision="fp16",
                tau=0.8, speed=0.03, steps=20, tune=True),
        # Sedimentation of 200 free disks in a walled box, with lubrication, at the kernel variant
        # that tuning found for it (few steps: the instant at which a free disk takes a node
        # depends on the last bits of its path).
        _domain("sedimentation_fp32", 2048, 8192, "box", 200, 10, 10, motion="free", density=1.5,
                gravity=1e-5, tau=0.7, steps=20, variant=1),
        # The collision and boundary that the paper's own simulations name: MRT with the
        # interpolated boundary, on a suspension.
        _domain("mrt_interpolated_fp32", 4096, 2048, "periodic", 500, 8, 20, collision="mrt",
                boundary="interpolated", steps=20, tune=True),
        # The cylinder sweep: 512 channels of all sizes, tuned, one 100-step block.
        dict(name="cylinder_sweep_512", kind="channels", cases=512, nx=0, ny=0, steps=100,
             precision="fp32", tune=True),
        # The channels of the warm-start measurement (time to drag), one block between tests.
        dict(name="warm_start_channels_96", kind="channels", cases=96, nx=256, ny=128, steps=100,
             precision="fp32", tune=False),
        # Inference of the shipped network on a batch of channels.
        dict(name="network_forward", kind="net", mode="forward", batch=16, height=128, width=256,
             levels=4, base=32, steps=1),
        # Training of it: mini-batches, then the parameters as they are kept.
        dict(name="network_training", kind="net", mode="train", batch=16, height=128, width=256,
             levels=4, base=32, steps=4),
    ]


def _domain(name, nx, ny, bc, disks, rmin, rmax, *, motion="prescribed", precision="fp32",
            collision="bgk", boundary="halfway", rho_w="const", tau=0.65, steps=20, tune=False,
            variant=0, graph=0, speed=0.05, spin=0.0, density=1.0, gravity=0.0):
    c = dict(kind="domain", nx=nx, ny=ny, bc=bc, disks=disks, rmin=float(rmin), rmax=float(rmax),
             motion=motion, precision=precision, collision=collision, boundary=boundary,
             rho_w=rho_w, tau=tau, steps=steps, tune=tune, variant=variant, graph=graph, speed=speed, spin=spin,
             density=density, gravity=gravity)
    if name:
        c["name"] = name
    return c


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def draw(rng: random.Random):
    """One more case: sizes over the whole range of the listed ones, odd ones among them."""
    kind = rng.choice(["domain"] * 7 + ["channels"] * 3 + ["net"] * 2)
    if kind == "domain":
        precision = rng.choice(["fp64", "fp32", "fp32", "fp32", "fp16"])
        most = 2048 * 1024 if precision == "fp64" else 8192 * 4096
        nodes = _log(rng, 64 * 64, most)
        shape = _log(rng, 0.3, 3.0)
        nx = max(64, min(8192, int(math.sqrt(nodes * shape))))
        ny = max(64, min(8192, int(nodes / nx)))
        bc = rng.choice(["periodic", "periodic", "channel", "box"])
        motion = "free" if bc == "box" else rng.choice(["prescribed", "prescribed", "rest"])
        rmax = min(20.0, min(nx, ny) / 2 - 10)
        rmin = rng.uniform(0.4, 1.0) * rmax
        rmin = max(5.0, rmin)
        cells = len(_cells(nx, ny, bc, rmax))
        disks = max(1, min(cells, int(nx * ny / 16777 * rng.uniform(0.5, 1.5))))
        collision = rng.choice(["bgk", "bgk", "bgk", "mrt"])
        steps = max(10, min(20 if motion == "free" else 100, int(2e8 / (nx * ny))))
        return _domain(None, nx, ny, bc, disks, rmin, rmax, motion=motion, precision=precision,
                       collision=collision, boundary=rng.choice(["halfway", "halfway", "interpolated"]),
                       rho_w=rng.choice(["const", "const", "local"]),
                       tau=round(rng.uniform(0.75, 0.95), 4),
                       steps=steps, tune=nx * ny >= 1 << 20 and motion != "free",
                       variant=1 if motion == "free" else 0, graph=rng.choice([0, steps]),
                       speed=0.03, spin=rng.choice([0.0, 0.001]), density=1.5, gravity=1e-5)
    if kind == "channels":
        if rng.random() < 0.5:
            return dict(kind="channels", cases=int(_log(rng, 4, 256)), nx=0, ny=0, steps=rng.choice([50, 100]),
                        precision=rng.choice(["fp32", "fp32", "fp64"]) if rng.random() < 0.2 else "fp32",
                        tune=rng.random() < 0.5)
        return dict(kind="channels", cases=int(_log(rng, 4, 256)), nx=rng.randrange(150, 400),
                    ny=2 * rng.randrange(48, 100), steps=100, precision="fp32", tune=rng.random() < 0.3)
    levels = rng.choice([2, 3, 4, 4])
    unit = 1 << (levels - 1)
    return dict(kind="net", mode=rng.choice(["forward", "train"]), batch=rng.randrange(1, 17),
                height=unit * rng.randrange(64 // unit, 160 // unit + 1),
                width=unit * rng.randrange(96 // unit, 320 // unit + 1), levels=levels,
                base=rng.choice([16, 32, 32]), steps=rng.choice([1, 2]))


# ------------------------------------------------------------------ inputs


def _cells(nx, ny, bc, rmax):
    """Corners of square cells that hold one disk each, three nodes apart from the next."""
    side = 2.0 * rmax + 4.0
    mx = 4.0 if bc == "box" else 0.0
    my = 0.0 if bc == "periodic" else 4.0
    kx, ky = max(1, int((nx - 2 * mx) // side)), max(1, int((ny - 2 * my) // side))
    return [(mx + side * i, my + side * j, side) for j in range(ky) for i in range(kx)]


def _disks(case, seed):
    """Rows (cx, cy, r, vx, vy, omega, rho_s): disks that do not overlap, all of them with one
    velocity, so that they keep their distances at any horizon."""
    rng = np.random.default_rng([seed, 11])
    nx, ny, bc = case["nx"], case["ny"], case["bc"]
    cells = _cells(nx, ny, bc, case["rmax"])
    if case["disks"] == 1:  # one disk in the middle of the channel, wherever that is
        at = [(nx * rng.uniform(0.4, 0.6), ny * rng.uniform(0.47, 0.53))]
        rs = [case["rmax"]]
    else:
        at, rs = [], []
        for c in rng.permutation(len(cells))[: case["disks"]]:
            x0, y0, side = cells[c]
            r = rng.uniform(case["rmin"], case["rmax"])
            free = side - 3.0 - 2.0 * r
            at.append((x0 + 1.5 + r + free * rng.uniform(), y0 + 1.5 + r + free * rng.uniform()))
            rs.append(r)
    vx = vy = 0.0
    if case["motion"] == "prescribed":
        vx = case["speed"] * rng.uniform(0.5, 1.0)
        vy = 0.0 if bc != "periodic" else case["speed"] * rng.uniform(-1.0, 1.0)
    return [(x, y, r, vx, vy, case["spin"] if case["motion"] != "free" else 0.0, case["density"])
            for (x, y), r in zip(at, rs)]


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
OP = (0, 3, 4, 1, 2, 7, 8, 5, 6)


def _equilibrium(rho, ux, uy):
    uu = ux * ux + uy * uy
    out = torch.empty((9,) + tuple(rho.shape), dtype=torch.float64, device=rho.device)
    for i in range(9):
        eu = EX[i] * ux + EY[i] * uy
        out[i] = rho * WT[i] * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu)
    return out


def _initial(case, seed):
    """A flow under way: the equilibrium of a smooth velocity field, a few waves each way."""
    rng = np.random.default_rng([seed, 12])
    dev = _device()
    x = torch.arange(case["nx"], dtype=torch.float64, device=dev) / case["nx"] * (2 * math.pi)
    y = torch.arange(case["ny"], dtype=torch.float64, device=dev) / case["ny"] * (2 * math.pi)
    ux = torch.zeros(case["ny"], case["nx"], dtype=torch.float64, device=dev)
    uy, rho = torch.zeros_like(ux), torch.ones_like(ux)
    for _ in range(3):
        k, m = rng.integers(1, 4, 2)
        a, b, c = rng.uniform(0, 2 * math.pi, 3)
        ux += 0.006 * torch.sin(m * y + a)[:, None] * torch.cos(k * x + b)[None, :]
        uy += 0.006 * torch.sin(k * x + c)[None, :] * torch.cos(m * y + a)[:, None]
        rho += 0.001 * torch.cos(m * y + c)[:, None] * torch.sin(k * x + a)[None, :]
    return _equilibrium(rho, ux, uy)


BC = {"periodic": (L.LBM_PERIODIC, L.LBM_PERIODIC), "channel": (L.LBM_PERIODIC, L.LBM_WALL),
      "box": (L.LBM_WALL, L.LBM_WALL), "open": (L.LBM_OPEN, L.LBM_WALL)}


def _prepare_domain(case, seed):
    dev = _device()
    stream = torch.cuda.Stream()
    bcx, bcy = BC[case["bc"]]
    free = case["motion"] == "free"
    lat = G.Lattice(case["nx"], case["ny"], case["tau"], bc_x=bcx, bc_y=bcy,
                    precision=L.PRECISION_NAMES[case["precision"]],
                    rho_w_mode=L.LBM_RHOW_LOCAL if case["rho_w"] == "local" else L.LBM_RHOW_CONST,
                    collision=L.LBM_MRT if case["collision"] == "mrt" else L.LBM_BGK,
                    boundary=L.LBM_INTERPOLATED if case["boundary"] == "interpolated" else L.LBM_HALFWAY,
                    gravity=_gravity(case), lub_range=2.0 if free else 0.0,
                    force_ring=max(64, case["steps"]), stream=stream.cuda_stream)
    for x, y, r, vx, vy, om, rho_s in _disks(case, seed):
        lat.add_disk(x, y, r, vx, vy, om, rho_s, L.LBM_FREE if free else L.LBM_PRESCRIBED)
    f = _initial(case, seed)
    torch.cuda.synchronize()
    L.lbm_set_populations(lat.handle, f, on_device=True)
    lat.sync()
    lat.set_kernel_variant(case["variant"])
    if case["graph"]:
        lat.set_graph(case["graph"])
    if case["tune"]:
        lat.autotune(4)
    shape = (case["ny"], case["nx"])
    return dict(case=case, lat=lat, stream=stream,
                fields=[torch.empty(shape, dtype=torch.float64, device=dev) for _ in range(3)],
                owner=torch.empty(shape, dtype=torch.int32, device=dev))


def _gravity(case):
    if case["motion"] != "free":
        return (0.0, 0.0)
    return (0.0, -case["gravity"]) if case["bc"] == "box" else (case["gravity"], 0.0)


def _channels(case, seed):
    """The open channels of a batch, as plain values: the cylinder sweep (nx = 0), or channels
    of one size with 1 to 4 disks each as the warm start has them."""
    rng = np.random.default_rng([seed, 13])
    size = np.random.default_rng(case["cases"])  # the same sizes whatever the seed
    out = []
    while len(out) < case["cases"]:
        if not case["nx"]:
            nx, ny = int(size.integers(128, 1025)), 2 * int(size.integers(32, 257))
            if nx / 4.0 - ny / 10.0 < 4.0:
                continue
            tau, r = 0.6, ny / 10.0
            most = min(100.0, 0.1 / 1.5 / ((tau - 0.5) / 3.0 / (2.0 * r)))  # inlet peak at most 0.1
            umax = 1.5 * rng.uniform(1.0, most) * (tau - 0.5) / 3.0 / (2.0 * r)
            disks = [(nx / 4.0, ny / 2.0 + rng.uniform(-2.0, 2.0), r)]
        else:
            nx, ny, disks = case["nx"], case["ny"], []
            for _ in range(40):
                r = rng.uniform(6.0, 16.0)
                x, y = rng.uniform(4 * r, nx - 4 * r), rng.uniform(3 * r, max(3 * r + 1e-3, ny - 3 * r))
                if all((x - a) ** 2 + (y - b) ** 2 > (r + c + 4) ** 2 for a, b, c in disks):
                    disks.append((x, y, r))
                if len(disks) == 1 + len(out) % 4:
                    break
            re, d, umean = rng.uniform(1.0, 100.0), 2.0 * max(q[2] for q in disks), 0.05 / 1.5
            tau = max(0.53, 0.5 + 3.0 * umean * d / re)
            umax = 1.5 * re * (tau - 0.5) / (3.0 * d)
            if umax > 0.12:
                continue
        out.append((nx, ny, tau, umax, disks))
    return out


def _prepare_channels(case, seed):
    stream = torch.cuda.Stream()
    chans = _channels(case, seed)
    b = G.Batch([L.make_config(nx, ny, tau, bc_x=L.LBM_OPEN, bc_y=L.LBM_WALL, inflow_umax=umax,
                               precision=L.PRECISION_NAMES[case["precision"]], force_ring=4,
                               stream=stream.cuda_stream) for nx, ny, tau, umax, _ in chans])
    for k, (_, _, _, _, disks) in enumerate(chans):
        for x, y, r in disks:
            b.add_disk(k, x, y, r)
    # no case retires: the sweep's own tolerance is not met for tens of thousands of steps,
    # and the time-to-drag measurement retires cases by its own criterion
    b.set_convergence(every=case["steps"], tol=0.0, max_steps=2_000_000_000)
    if case["tune"]:
        b.autotune(4)
    sizes = [nx * ny for nx, ny, _, _, _ in chans]
    at = np.concatenate([[0], np.cumsum(sizes)])
    fields = torch.empty(3, int(at[-1]), dtype=torch.float64, device=_device())
    views = [[fields[q, at[k]:at[k + 1]] for q in range(3)] for k in range(len(chans))]
    torch.cuda.synchronize()
    return dict(case=case, batch=b, stream=stream, fields=fields, views=views)


def _network_data(case, seed, steps):
    """Inputs as the warm start builds them (solid mask, Re, distance to the nearest disk,
    axial distance, parabola, coordinates), and smooth targets."""
    rng = np.random.default_rng([seed, 14])
    B, H, W = case["batch"], case["height"], case["width"]
    dev = _device()
    n = B * steps
    yy, xx = torch.meshgrid(torch.arange(H, device=dev, dtype=torch.float32),
                            torch.arange(W, device=dev, dtype=torch.float32), indexing="ij")
    x = torch.zeros(n, 8, H, W, device=dev)
    t = torch.zeros(n, 3, H, W, device=dev)
    for k in range(n):
        re = float(rng.uniform(1.0, 100.0))
        near = torch.full((H, W), 1e30, device=dev)
        axial = torch.zeros(H, W, device=dev)
        for _ in range(1 + k % 4):
            r = float(rng.uniform(0.03, 0.1)) * H
            cx, cy = float(rng.uniform(2 * r, W - 2 * r)), float(rng.uniform(2 * r, H - 2 * r))
            d = torch.sqrt((xx - cx) ** 2 + (yy - cy) ** 2) - r
            axial = torch.where(d < near, (xx - cx) / (8 * r), axial)
            near = torch.minimum(near, d)
        para = 4.0 * (yy + 0.5) * (H - yy - 0.5) / (H * H)
        x[k, 0] = (near <= 0).float()
        x[k, 1], x[k, 2] = re / 100.0, math.log10(re) / 2.0
        x[k, 3] = (near / 16.0).clamp(-1.0, 4.0)
        x[k, 4] = axial.clamp(-1.0, 4.0)
        x[k, 5], x[k, 6], x[k, 7] = para, xx / W, (yy + 0.5) / H - 0.5
        for q in range(3):
            t[k, q] = torch.exp(-near.clamp(0.0, 1e3) / 20.0) * math.cos(q + re / 30.0)
    fluid = 1.0 - x[:, 0]
    t = t * fluid[:, None]
    cut = [slice(B * s, B * (s + 1)) for s in range(steps)]
    return [(x[c].contiguous(), t[c].contiguous(), fluid[c].contiguous()) for c in cut]


def _shapes(case):
    ch = [case["base"] << l for l in range(case["levels"])]
    out, cin = [], 8
    for c in ch:
        out += [(c, cin, 3), (c, c, 3)]
        cin = c
    for l in range(case["levels"] - 2, -1, -1):
        out += [(ch[l], ch[l + 1] + ch[l], 3), (ch[l], ch[l], 3)]
    return out + [(3, ch[0], 1)]


def _weights(case, seed):
    rng = np.random.default_rng([seed, 15])
    parts = []
    for co, ci, k in _shapes(case):
        parts.append(rng.normal(0.0, math.sqrt(2.0 / (ci * k * k)), co * ci * k * k))
        parts.append(rng.uniform(-0.05, 0.05, co))
    return np.concatenate(parts).astype(np.float32)


RATE = 1e-5  # the learning rate that training ends with


def _prepare_net(case, seed):
    stream = torch.cuda.Stream()
    net = G.UNet(case["height"], case["width"], levels=case["levels"], base=case["base"],
                 max_batch=case["batch"], seed=1, stream=stream.cuda_stream)
    net.set_params(_weights(case, seed))
    data = _network_data(case, seed, case["steps"])
    shape = (case["batch"], 3, case["height"], case["width"])
    out = torch.empty(shape, device=_device())
    params = torch.empty(net.nparam, device=_device())
    torch.cuda.synchronize()
    return dict(case=case, net=net, data=data, out=out, params=params, stream=stream)


def prepare(case, seed):
    make = {"domain": _prepare_domain, "channels": _prepare_channels, "net": _prepare_net}
    return make[case["kind"]](case, seed)


# --------------------------------------------------------------------- run


def _run_domain(s):
    case, lat = s["case"], s["lat"]
    kept = KEPT[case["precision"]]
    t0 = lat.t
    lat.step(case["steps"])
    rho, ux, uy = s["fields"]
    with torch.cuda.stream(s["stream"]):
        L.lbm_fields(lat.handle, rho, ux, uy, on_device=True)
        L.lbm_get_owner(lat.handle, s["owner"], on_device=True)
        out = dict(rho=(rho - 1.0).to(kept), ux=ux.to(kept), uy=uy.to(kept), owner=s["owner"])
    rec = lat.forces(t0, case["steps"])
    out["forces"] = rec.astype({"fp64": np.float64, "fp32": np.float32, "fp16": np.float16}[case["precision"]])
    out["solids"] = lat.solids()
    return out


def _run_channels(s):
    case, b = s["case"], s["batch"]
    kept = KEPT[case["precision"]]
    b.run(case["steps"])
    st, steps, drag = b.state()
    for k, (rho, ux, uy) in enumerate(s["views"]):
        L.lbm_fields(b.case(k).handle, rho, ux, uy, on_device=True)
    with torch.cuda.stream(s["stream"]):
        rho, ux, uy = s["fields"]
        out = dict(rho=(rho - 1.0).to(kept), ux=ux.to(kept), uy=uy.to(kept))
    out.update(state=st, steps=steps, drag=drag.astype(np.float64 if case["precision"] == "fp64" else np.float32))
    return out


def _run_net(s):
    case, net = s["case"], s["net"]
    if case["mode"] == "forward":
        for x, _, _ in s["data"]:
            L.lbm_unet_forward(net.handle, x, s["out"], case["batch"], on_device=True)
        return s["out"]
    losses = [net.train_step(x, t, f, RATE, on_device=True) for x, t, f in s["data"]]
    L.lbm_unet_get_params(net.handle, s["params"], on_device=True)
    return dict(losses=losses, params=s["params"])


def run(state):
    return {"domain": _run_domain, "channels": _run_channels, "net": _run_net}[state["case"]["kind"]](state)


# -------------------------------------------------------------------- work


def work(case):
    """Populations in and out of every step (a step's force records need those of its own
    time), and the results; about 100 operations a node and step."""
    if case["kind"] == "domain":
        n, b = case["nx"] * case["ny"], BYTES[case["precision"]]
        return dict(bytes=n * (18.0 * b * case["steps"] + 3 * b + 4), flops=100.0 * n * case["steps"])
    if case["kind"] == "channels":
        n = sum(c[0] * c[1] for c in _channels(case, 0))
        b = BYTES[case["precision"]]
        return dict(bytes=n * (18.0 * b * case["steps"] + 3 * b), flops=100.0 * n * case["steps"])
    pixels = case["batch"] * case["height"] * case["width"]
    flops, weights, l, scale = 0.0, 0, 0, []
    levels = case["levels"]
    scale = [l for l in range(levels) for _ in (0, 1)] + [l for l in range(levels - 2, -1, -1) for _ in (0, 1)] + [0]
    for (co, ci, k), l in zip(_shapes(case), scale):
        flops += 2.0 * pixels / 4 ** l * co * ci * k * k
        weights += co * ci * k * k + co
    train = case["mode"] == "train"
    per = dict(bytes=pixels * (8 + 3 + (1 if train else 0)) * 4.0 + weights * (24.0 if train else 2.0),
               flops=flops * (3 if train else 1))
    return {q: v * case["steps"] for q, v in per.items()}


# ------------------------------------------------------------------- exact


class _Exact:
    """The method in plain torch FP64, whole-domain operations, B domains of one size."""

    def __init__(self, B, nx, ny, tau, bc, umax, disks, case):
        self.B, self.nx, self.ny, self.bc = B, nx, ny, bc
        dev = self.dev = _device()
        col = lambda v: torch.as_tensor(v, dtype=torch.float64, device=dev).reshape(-1, 1, 1)  # noqa: E731
        self.tau, self.umax = col(tau), col(umax)
        self.px, self.py = bc == "periodic" or bc == "channel", bc == "periodic"
        self.local = case.get("rho_w") == "local"
        self.mrt, self.cut = case.get("collision") == "mrt", case.get("boundary") == "interpolated"
        self.free = case.get("motion") == "free"
        self.grav = _gravity(case) if "motion" in case else (0.0, 0.0)
        d = torch.as_tensor(np.array(disks, dtype=np.float64), device=dev)
        self.case_of = d[:, 0].long()
        self.x, self.y, self.r = d[:, 1].clone(), d[:, 2].clone(), d[:, 3].clone()
        self.vx, self.vy, self.om, self.rho_s = (d[:, k].clone() for k in (4, 5, 6, 7))
        self.xa, self.ya, self.t = self.x.clone(), self.y.clone(), 0
        self.moves = self.free or bool((self.vx != 0).any()) or bool((self.vy != 0).any())
        self.owner = self.raster()
        self.pending = torch.zeros(len(disks), 3, dtype=torch.float64, device=dev)
        if self.mrt:
            e = np.array([EX, EY], dtype=np.float64)
            q = (e ** 2).sum(0)
            M = np.stack([np.ones(9), 3 * q - 4, 4.5 * q * q - 10.5 * q + 4, e[0], (3 * q - 5) * e[0], e[1],
                          (3 * q - 5) * e[1], e[0] ** 2 - e[1] ** 2, e[0] * e[1]])
            s = np.array([0.0, 1.64, 1.54, 0.0, 1.9, 0.0, 1.9] + [1.0 / float(np.reshape(tau, -1)[0])] * 2)
            self.A = np.linalg.inv(M) @ (s[:, None] * M)

    def start(self, f):
        self.f = [f[i].reshape(self.B, self.ny, self.nx).clone() for i in range(9)]

    def inlet(self):
        yy = torch.arange(self.ny, dtype=torch.float64, device=self.dev)[None, :, None] + 0.5
        return 4.0 * self.umax * yy * (self.ny - yy) / (self.ny * self.ny)

    def raster(self):
        R = int(math.ceil(float(self.r.max()))) + 1
        o = torch.arange(-R, R + 2, device=self.dev)
        owner = torch.full((self.B * self.ny * self.nx,), len(self.x), dtype=torch.int32, device=self.dev)
        for a in range(0, len(self.x), 512):
            q = slice(a, a + 512)
            i = torch.floor(self.x[q]).long()[:, None, None] + o[None, None, :]
            j = torch.floor(self.y[q]).long()[:, None, None] + o[None, :, None]
            dx, dy = i - self.x[q][:, None, None], j - self.y[q][:, None, None]
            rr = (self.r[q] * self.r[q])[:, None, None]
            hit = dx * dx + dy * dy <= rr
            i, j, hit = torch.broadcast_tensors(i, j, hit)
            k, ok = self.place(i, j)
            k = k + (self.case_of[q] * (self.ny * self.nx))[:, None, None]
            s = torch.arange(a, a + len(self.x[q]), dtype=torch.int32, device=self.dev)[:, None, None].expand_as(k)
            ok = ok & hit
            owner.scatter_reduce_(0, k[ok], s[ok], "amin")
        owner[owner == len(self.x)] = -1
        return owner

    def place(self, i, j):
        """Cell of the node (i, j) within its domain, and whether there is one."""
        ok = torch.ones_like(i, dtype=torch.bool)
        if self.px:
            i = i % self.nx
        else:
            ok = ok & (i >= 0) & (i < self.nx)
        if self.py:
            j = j % self.ny
        else:
            ok = ok & (j >= 0) & (j < self.ny)
        return j.clamp(0, self.ny - 1) * self.nx + i.clamp(0, self.nx - 1), ok

    def near(self, d, n, periodic):
        return d - n * torch.floor(d / n + 0.5) if periodic else d

    def velocity(self, s, px, py):
        dx = self.near(px - self.x[s], self.nx, self.px)
        dy = self.near(py - self.y[s], self.ny, self.py)
        return self.vx[s] - self.om[s] * dy, self.vy[s] + self.om[s] * dx, dx, dy

    def step(self):
        B, ny, nx = self.B, self.ny, self.nx
        f = [a.reshape(-1) for a in self.f]
        own = self.owner.reshape(B, ny, nx)
        rho = sum(f) if self.local else None
        rec = torch.zeros(len(self.x), 6, dtype=torch.float64, device=self.dev)
        g = [torch.roll(self.f[i], (EY[i], EX[i]), (1, 2)) for i in range(9)]
        # walls (and the resting edges beyond open columns)
        for i in range(1, 9):
            if EX[i] and not self.px:
                edge = 0 if EX[i] > 0 else nx - 1
                g[i][:, :, edge] = self.f[OP[i]][:, :, edge]
            if EY[i] and not self.py:
                edge = 0 if EY[i] > 0 else ny - 1
                g[i][:, edge, :] = self.f[OP[i]][:, edge, :]
        # links to the solids: the returned populations, and the force records
        for i in range(1, 9):
            nb = torch.roll(own, (-EY[i], -EX[i]), (1, 2))
            if EX[i] and not self.px:
                nb[:, :, nx - 1 if EX[i] > 0 else 0] = -1
            if EY[i] and not self.py:
                nb[:, ny - 1 if EY[i] > 0 else 0, :] = -1
            k = ((own < 0) & (nb >= 0)).reshape(-1).nonzero()[:, 0]
            s = nb.reshape(-1)[k].long()
            x, y = (k % nx), (k // nx) % ny
            base = k - (y * nx + x)
            fi = f[i][k]
            rw = rho[k] if self.local else 1.0
            if self.cut:
                px = self.near(x - self.x[s], nx, self.px)
                py = self.near(y - self.y[s], ny, self.py)
                a, h = EX[i] ** 2 + EY[i] ** 2, px * EX[i] + py * EY[i]
                c = px * px + py * py - self.r[s] ** 2
                disc = h * h - a * c
                q = torch.where(disc > 0, (-h - torch.sqrt(disc.clamp(min=0))) / a, torch.full_like(h, 0.5))
                q = q.clamp(0.0, 1.0)
                ux, uy, dx, dy = self.velocity(s, x + q * EX[i], y + q * EY[i])
                m = -6.0 * WT[i] * rw * (EX[i] * ux + EY[i] * uy)
                kn, ok = self.place(x - EX[i], y - EY[i])
                kn = kn + base
                ok = ok & (self.owner[kn] < 0)
                close = torch.where(ok, 2 * q * fi + (1 - 2 * q) * f[i][kn] + m, fi + m)
                q1 = q.clamp(min=0.25)
                far = (fi + m) / (2 * q1) + (2 * q1 - 1) / (2 * q1) * f[OP[i]][k]
                fbb = torch.where(q >= 0.5, far, close)
            else:
                ux, uy, dx, dy = self.velocity(s, x + 0.5 * EX[i], y + 0.5 * EY[i])
                fbb = fi - 6.0 * WT[i] * rw * (EX[i] * ux + EY[i] * uy)
            cx, cy = EX[i] * (fi + fbb), EY[i] * (fi + fbb)
            gx, gy = cx - ux * (fi - fbb), cy - uy * (fi - fbb)
            rec.index_add_(0, s, torch.stack([cx, cy, dx * cy - dy * cx, gx, gy, dx * gy - dy * gx], 1))
            g[OP[i]].reshape(-1)[k] = fbb
        rec[:, :3] += self.pending
        rec[:, 3:] += self.pending
        self.pending.zero_()
        # collision
        fluid = own < 0
        r = sum(g)
        r = torch.where(fluid, r, torch.ones_like(r))
        ux = (g[1] + g[5] + g[8] - g[3] - g[6] - g[7]) / r
        uy = (g[2] + g[5] + g[6] - g[4] - g[7] - g[8]) / r
        eq = _equilibrium(r, ux, uy)
        new = []
        if self.mrt:
            d = [g[i] - eq[i] for i in range(9)]
        for i in range(9):
            if self.mrt:
                o = g[i] - sum(float(self.A[i, k]) * d[k] for k in range(9) if abs(self.A[i, k]) > 1e-15)
            else:
                o = g[i] - (g[i] - eq[i]) / self.tau
            new.append(torch.where(fluid, o, torch.zeros_like(o)))
        if self.bc == "open":
            self.columns(new, r, ux, uy, fluid)
        self.f = new
        self.move(rec)
        if self.moves:
            self.remask()
        self.t += 1
        return rec

    def columns(self, new, r, ux, uy, fluid):
        """Open columns: non-equilibrium extrapolation from the inner neighbour."""
        nx, uin = self.nx, self.inlet()
        for b, n in ((0, 1), (nx - 1, nx - 2)):
            rn, un, vn = r[:, :, n:n + 1], ux[:, :, n:n + 1], uy[:, :, n:n + 1]
            en = _equilibrium(rn, un, vn)
            eb = _equilibrium(rn, uin, torch.zeros_like(uin)) if b == 0 else _equilibrium(torch.ones_like(rn), un, vn)
            at, inner = fluid[:, :, b:b + 1], fluid[:, :, n:n + 1]
            plain = _equilibrium(torch.ones_like(rn), uin.expand_as(rn), torch.zeros_like(rn)) if b == 0 else None
            for i in range(9):
                old = new[i][:, :, b:b + 1]
                v = torch.where(inner, eb[i] + (new[i][:, :, n:n + 1] - en[i]), plain[i] if b == 0 else old)
                new[i][:, :, b:b + 1] = torch.where(at, v, old)

    def move(self, rec):
        if not self.free:
            self.x, self.y = self.xa + self.vx * (self.t + 1), self.ya + self.vy * (self.t + 1)
            return
        M = self.rho_s * math.pi * self.r ** 2
        buoy = 1.0 - 1.0 / self.rho_s
        ka = buoy.abs() * M * math.hypot(*self.grav)
        zeta = 2.0
        mag = lambda k, gap: torch.where(gap >= zeta, torch.zeros_like(gap), k * ((zeta - gap) / zeta) ** 2)  # noqa: E731
        dx = self.near(self.x[:, None] - self.x[None, :], self.nx, self.px)
        dy = self.near(self.y[:, None] - self.y[None, :], self.ny, self.py)
        d = torch.sqrt(dx * dx + dy * dy)
        m = mag(torch.maximum(ka[:, None], ka[None, :]), d - self.r[:, None] - self.r[None, :])
        m = torch.where(d > 0, m / torch.where(d > 0, d, torch.ones_like(d)), torch.zeros_like(d))
        fx, fy = (m * dx).sum(1), (m * dy).sum(1)
        if not self.py:
            fy = fy + mag(ka, self.y - self.r + 0.5) - mag(ka, self.ny - 0.5 - self.y - self.r)
        if not self.px:
            fx = fx + mag(ka, self.x - self.r + 0.5) - mag(ka, self.nx - 0.5 - self.x - self.r)
        fx, fy = rec[:, 3] + buoy * M * self.grav[0] + fx, rec[:, 4] + buoy * M * self.grav[1] + fy
        vx, vy = self.vx + fx / M, self.vy + fy / M
        self.x, self.y = self.x + 0.5 * (self.vx + vx), self.y + 0.5 * (self.vy + vy)
        self.vx, self.vy, self.om = vx, vy, self.om + rec[:, 5] / (0.5 * M * self.r ** 2)

    def book(self, k, s, sign):
        x, y = k % self.nx, (k // self.nx) % self.ny
        v = [a.reshape(-1)[k] for a in self.f]
        jx, jy = sum(EX[i] * v[i] for i in range(9)), sum(EY[i] * v[i] for i in range(9))
        _, _, dx, dy = self.velocity(s, x.double(), y.double())
        self.pending.index_add_(0, s, sign * torch.stack([jx, jy, dx * jy - dy * jx], 1))

    def remask(self):
        was, now = self.owner, self.raster()
        self.owner = now
        covered = ((was < 0) & (now >= 0)).nonzero()[:, 0]
        fresh = ((was >= 0) & (now < 0)).nonzero()[:, 0]
        self.book(covered, now[covered].long(), 1.0)
        if not len(fresh):
            return
        usable = (now < 0) & (was < 0)
        x, y = fresh % self.nx, (fresh // self.nx) % self.ny
        base = fresh - (y * self.nx + x)
        n = len(fresh)
        val = torch.zeros(3, 8, 9, n, dtype=torch.float64, device=self.dev)
        ok = torch.zeros(3, 8, n, dtype=torch.bool, device=self.dev)
        for d in range(3):
            for i in range(1, 9):
                k, inside = self.place(x + (d + 1) * EX[i], y + (d + 1) * EY[i])
                k = k + base
                ok[d, i - 1] = inside & usable[k]
                for j in range(9):
                    val[d, i - 1, j] = self.f[j].reshape(-1)[k]
        ok[1] &= ok[0]
        ok[2] &= ok[1]
        out, done = torch.zeros(9, n, dtype=torch.float64, device=self.dev), torch.zeros(n, dtype=torch.bool, device=self.dev)
        for level, w in ((2, (3.0, -3.0, 1.0)), (1, (2.0, -1.0, 0.0)), (0, (1.0, 0.0, 0.0))):
            use = ok[level].double()
            count = use.sum(0)
            v = sum(w[d] * val[d] for d in range(3))
            v = (v * use[:, None]).sum(0) / count.clamp(min=1.0)
            take = (count > 0) & ~done
            out = torch.where(take, v, out)
            done |= take
        s = was[fresh].long()
        vx, vy, _, _ = self.velocity(s, x.double(), y.double())
        out = torch.where(done, out, _equilibrium(torch.ones_like(vx), vx, vy))
        for j in range(9):
            self.f[j].reshape(-1)[fresh] = out[j]
        self.book(fresh, s, -1.0)

    def fields(self):
        fluid = self.owner.reshape(self.B, self.ny, self.nx) < 0
        r = sum(self.f)
        nan = torch.full_like(r, math.nan)
        d = sum(self.f[i] - WT[i] for i in range(9))
        ux = (self.f[1] + self.f[5] + self.f[8] - self.f[3] - self.f[6] - self.f[7]) / r
        uy = (self.f[2] + self.f[5] + self.f[6] - self.f[4] - self.f[7] - self.f[8]) / r
        return [torch.where(fluid, a, nan) for a in (d, ux, uy)]


def _exact_domain(case, seed):
    disks = [(0,) + d for d in _disks(case, seed)]
    e = _Exact(1, case["nx"], case["ny"], case["tau"], case["bc"], 0.0, disks, case)
    e.start(_initial(case, seed))
    for _ in range(TUNE_STEPS if case["tune"] else 0):
        e.step()
    rec = torch.stack([e.step() for _ in range(case["steps"])])
    rho, ux, uy = (a[0] for a in e.fields())
    return dict(rho=rho, ux=ux, uy=uy, owner=e.owner.reshape(case["ny"], case["nx"]),
                forces=rec.reshape(case["steps"], len(disks), 2, 3),
                solids=torch.stack([e.x, e.y, e.vx, e.vy, e.om], 1))


def _exact_channels(case, seed):
    chans = _channels(case, seed)
    if sum(c[0] * c[1] for c in chans) > 12e6 or (not case["nx"] and case["cases"] > 24):
        return None  # minutes, one channel after the other
    groups = [list(range(len(chans)))] if case["nx"] else [[k] for k in range(len(chans))]
    parts, drag = [None] * len(chans), np.zeros(len(chans))
    for ks in groups:
        nx, ny = chans[ks[0]][:2]
        disks = [(q, x, y, r, 0.0, 0.0, 0.0, 1.0) for q, k in enumerate(ks) for x, y, r in chans[k][4]]
        e = _Exact(len(ks), nx, ny, [chans[k][2] for k in ks], "open", [chans[k][3] for k in ks], disks, {})
        u = e.inlet().expand(len(ks), ny, nx)
        e.start(_equilibrium(torch.ones_like(u), u, torch.zeros_like(u)))
        extra = 10 * (1 + 4) if case["tune"] else 0  # steps that Batch.autotune(4) advances it by
        for _ in range(extra + case["steps"]):
            rec = e.step()
        total = torch.zeros(len(ks), dtype=torch.float64, device=e.dev).index_add_(0, e.case_of, rec[:, 3])
        fields = e.fields()
        for q, k in enumerate(ks):
            drag[k] = float(total[q])
            parts[k] = [a[q].reshape(-1) for a in fields]
    rho, ux, uy = (torch.cat([p[q] for p in parts]) for q in range(3))
    return dict(rho=rho, ux=ux, uy=uy, state=None, steps=None, drag=drag)


def _forward(w, x, levels):
    F = torch.nn.functional
    conv = lambda v, k: F.conv2d(v, w[k][0], w[k][1], padding=w[k][0].shape[-1] // 2)  # noqa: E731
    e, k = [], 0
    for l in range(levels):
        v = x if l == 0 else F.avg_pool2d(e[-1], 2)
        e.append(F.relu(conv(F.relu(conv(v, k)), k + 1)))
        k += 2
    d = e[-1]
    for l in range(levels - 2, -1, -1):
        d = torch.cat([d.repeat_interleave(2, 2).repeat_interleave(2, 3), e[l]], 1)
        d = F.relu(conv(F.relu(conv(d, k)), k + 1))
        k += 2
    return conv(d, k)


def _exact_net(case, seed):
    pixels = case["batch"] * case["height"] * case["width"]
    if case["mode"] == "train" and pixels * case["steps"] * (case["base"] / 32.0) ** 2 > 3e5:
        return None  # FP64 convolutions, there and back: too long
    dev, at, w = _device(), 0, []
    flat = torch.as_tensor(_weights(case, seed), dtype=torch.float64, device=dev)
    for co, ci, k in _shapes(case):
        a = flat[at:at + co * ci * k * k].reshape(co, ci, k, k).clone()
        at += co * ci * k * k
        w.append([a, flat[at:at + co].clone()])
        at += co
    data = [[v.double() for v in d] for d in _network_data(case, seed, case["steps"])]
    if case["mode"] == "forward":
        x = data[-1][0]
        return torch.cat([_forward(w, x[k:k + 1], case["levels"]) for k in range(case["batch"])])
    every = [p.requires_grad_() for q in w for p in q]
    m, v, losses = [torch.zeros_like(p) for p in every], [torch.zeros_like(p) for p in every], []
    for n, (x, t, fluid) in enumerate(data, 1):
        count = 3.0 * float(fluid.sum())
        total, grads = 0.0, [torch.zeros_like(p) for p in every]
        for k in range(case["batch"]):
            d = (_forward(w, x[k:k + 1], case["levels"]) - t[k:k + 1]) * fluid[k:k + 1, None]
            loss = (d * d).sum() / count
            for a, b in zip(grads, torch.autograd.grad(loss, every)):
                a += b
            total += float(loss.detach())
        losses.append(total)
        with torch.no_grad():
            for p, a, m_, v_ in zip(every, grads, m, v):
                m_.mul_(0.9).add_(0.1 * a)
                v_.mul_(0.999).add_(0.001 * a * a)
                p -= RATE * (m_ / (1 - 0.9 ** n)) / (torch.sqrt(v_ / (1 - 0.999 ** n)) + 1e-8)
    return dict(losses=np.array(losses), params=torch.cat([p.detach().reshape(-1) for p in every]))


def exact(case, seed):
    """What run() returns for these inputs, in 64 bits."""
    return {"domain": _exact_domain, "channels": _exact_channels, "net": _exact_net}[case["kind"]](case, seed)
