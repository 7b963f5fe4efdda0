"""The work a user of this framework has it do, as cases that can be timed and compared.

Two kinds of work: runs of the coupled lattice Boltzmann step through the C ABI's Python binding
(``_lbm``), and the learned warm start's layers and network (``_nn``, ``warmstart``).  A lattice pass is
what a sample of a study is: the initial phase field goes in, the method steps, the diagnostics the study
reads and the fields come out (into pinned host memory, as the library returns fields to the host).

``exact`` restates the paper's step (arXiv 2311.05091, Sec. 2-3, Appendix A) and the warm start's layers
plainly in 64 bits with torch, batched over instances.
"""
from __future__ import annotations

import ctypes
import math
import random

import numpy as np
import torch
import torch.nn.functional as F

from paper_2311_05091_gb300 import _lbm as L
from paper_2311_05091_gb300 import _nn
from paper_2311_05091_gb300.warmstart import COUT_PAD, WarmStartNet, forward_flops, layer_shapes, train_flops

DEV = "cuda"
W_IFACE = 4.0                     # interface width of every workload of this repository
UNEVEN_SIDES = (64, 128, 256, 512)
Q = {"D2Q9": 9, "D3Q15": 15, "D3Q19": 19}
LATTICE = {"D2Q9": L.LBM_D2Q9, "D3Q15": L.LBM_D3Q15, "D3Q19": L.LBM_D3Q19}


# ---------------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------------
def _lattice(kind, lattice, nx, ny, nz=1, batch=1, f16=False, steps=64, angle=False, **more):
    return dict(kind=kind, lattice=lattice, nx=nx, ny=ny, nz=nz, batch=batch, f16=f16, steps=steps, angle=angle, **more)


def listed():
    return [
        # The smallest lattice of the studies (half-disk drop on a flat wall, y walls): the steps between two
        # samples of its contact angle.  Launches and the latency of one step are all there is.
        dict(_lattice("wall", "D2Q9", 128, 64, steps=32, angle=True), name="wall_128x64"),
        # An open channel with obstacles, velocity inlet and pressure outlet: no axis periodic and rows of odd
        # length, so neither aligned copies nor the periodic form of the kernels apply.
        dict(_lattice("channel", "D2Q9", 483, 127, steps=100), name="channel_483x127"),
        # The contact-angle sweep at the size of the relaxation studies, NS populations stored as FP16: the steps
        # between two samples of its angles.
        dict(_lattice("disk", "D2Q9", 256, 256, batch=5, f16=True, steps=64, angle=True), name="disk_256x5_f16"),
        # The headline workload: five contact angles on 1024^2, density and viscosity ratio 10.
        dict(_lattice("disk", "D2Q9", 1024, 1024, batch=5, steps=48), name="disk_1024x5"),
        # 64 lattices of uneven size advanced by one persistent launch per step: the label generation of the
        # warm start and every parameter study over geometries.
        dict(_lattice("uneven", "D2Q9", 0, 0, batch=64, steps=64, sizes=0), name="uneven_64"),
        # The 3D porous run (sphere pack, periodic, body force) with its phase-flux diagnostic: the largest state.
        dict(_lattice("porous", "D3Q19", 256, 256, 256, steps=20), name="porous_256"),
        # A drop on a wall in 3D with density ratio 10 on the paper's lattice and rows of odd length: walls, mass
        # flux and the general form of the 3D kernels.
        dict(_lattice("drop3d", "D3Q15", 117, 97, 75, steps=24), name="drop3d_117x97x75"),
        # A wide layer of the warm start's decoder at full resolution (forward, bias and ReLU): memory-bound.
        dict(kind="conv", n=16, h=256, w=256, cin=64, cout=32, relu=True, name="conv_256_64to32"),
        # A layer of its coarsest level, in the direction of the data gradient (no bias, no ReLU): the tensor cores
        # have the most to do per byte.
        dict(kind="conv", n=16, h=32, w=32, cin=256, cout=256, relu=False, name="conv_32_256to256"),
        # Weight and bias gradient of a middle decoder layer.
        dict(kind="wgrad", n=16, h=128, w=128, cin=128, cout=64, name="wgrad_128_128to64"),
        # One training iteration of the network at its standard widths and batch.
        dict(kind="train", n=16, h=256, w=256, widths="32-64-128-256", name="train_256x16"),
        # The warm start of one geometry: inference and projection for a single image.
        dict(kind="predict", n=1, h=256, w=256, widths="32-64-128-256", name="predict_256x1"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["wall", "channel", "disk", "disk", "uneven", "porous", "drop3d", "conv", "conv", "wgrad",
                       "train", "predict"])
    if kind == "wall":
        nx = _log(rng, 64, 1024)
        return _lattice(kind, "D2Q9", nx, max(48, nx // 2 + rng.randrange(8)), steps=rng.choice([16, 32]),
                        angle=rng.random() < 0.5)
    if kind == "channel":
        nx = _log(rng, 120, 1500)
        return _lattice(kind, "D2Q9", nx, max(48, _log(rng, 48, 500)), steps=rng.choice([50, 100]))
    if kind == "disk":
        f16 = rng.random() < 0.4
        n = _log(rng, 96, 1000)
        ny = n + rng.randrange(-15, 16)
        return _lattice(kind, "D2Q9", 8 * (n // 8) if f16 else n, ny, batch=rng.randrange(1, 6), f16=f16,
                        steps=rng.choice([24, 48]), angle=rng.random() < 0.3)
    if kind == "uneven":
        return _lattice(kind, "D2Q9", 0, 0, batch=_log(rng, 4, 64), steps=rng.choice([32, 64]),
                        sizes=rng.randrange(1, 10000))
    if kind == "porous":
        nx = _log(rng, 48, 230)
        return _lattice(kind, "D3Q19", nx, nx + rng.randrange(-6, 7), nx + rng.randrange(-6, 7),
                        f16=nx % 8 == 0 and rng.random() < 0.5, steps=20)
    if kind == "drop3d":
        nx = _log(rng, 40, 180)
        return _lattice(kind, rng.choice(["D3Q15", "D3Q19"]), nx, nx + rng.randrange(-8, 9), max(36, nx // 2),
                        steps=rng.choice([12, 24]))
    if kind in ("conv", "wgrad"):
        lv = rng.randrange(4)
        c = [16, 32, 64, 128, 256]
        side = 256 >> lv
        h, w = max(8, _log(rng, side // 4, side)), max(8, _log(rng, side // 4, side))
        case = dict(kind=kind, n=_log(rng, 1, 16), h=h, w=w, cin=rng.choice(c[max(0, lv - 1):lv + 3]),
                    cout=rng.choice(c[1:][lv:lv + 2]))
        return dict(case, relu=rng.random() < 0.5) if kind == "conv" else case
    side = rng.choice([64, 128, 192, 256])
    return dict(kind=kind, n=_log(rng, 1, 16), h=side, w=rng.choice([side, 64, 128, 200]),
                widths=rng.choice(["32-64-128-256", "32-64-128", "32-64"]))


def _sizes(case):
    """(nx, ny) of every instance of a lattice case."""
    if case["kind"] != "uneven":
        return [(case["nx"], case["ny"])] * case["batch"]
    r = random.Random(case["sizes"] * 7919 + 1)
    sides = [r.choice(UNEVEN_SIDES) for _ in range(case["batch"])]
    return [(s, s) for s in sides]


def work(case):
    """Bytes and operations one pass cannot do without.

    Lattice, per node and step: both population sets and the history (phi1, u, S) read and written, phi0 and the
    phi1 stencil read; the operations are the stencils, forces and two moment-space collisions.  The fields go out
    once.  Layers: tensors and weights once, two operations per multiply-add."""
    if "lattice" in case:
        q = Q[case["lattice"]]
        d = 2 if q == 9 else 3
        nodes = sum(a * b for a, b in _sizes(case)) * case["nz"]
        per_step = 2 * q * (4 + (2 if case["f16"] else 4)) + 4 + 4 + 2 * 4 * (1 + 2 * d)
        return {"bytes": nodes * (case["steps"] * per_step + 4 * (3 + d)),
                "flops": nodes * case["steps"] * (500 if d == 2 else 60 * q)}
    P = case["n"] * case["h"] * case["w"]
    if case["kind"] in ("conv", "wgrad"):
        ci, co = case["cin"], case["cout"]
        wbytes = (2 if case["kind"] == "conv" else 4) * 9 * ci * co + 4 * co
        return {"bytes": 4 * P * (ci + co) + wbytes, "flops": 18.0 * P * ci * co}
    widths = _widths(case)
    nw = sum(9 * ci * co + co for ci, co in layer_shapes(widths))
    if case["kind"] == "train":
        return {"bytes": P * 4 * (3 + COUT_PAD) + 4 * nw * 9, "flops": float(case["n"] * train_flops(widths, case["h"], case["w"]))}
    return {"bytes": P * 4 * 3 + 2 * nw, "flops": float(case["n"] * forward_flops(widths, case["h"], case["w"]))}


# ---------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------
def _diffuse(dist):
    return 0.5 + 0.5 * torch.tanh(2.0 * dist / W_IFACE)


def _axes(*n):
    """Node coordinates of axes of the given lengths, broadcast against each other (the first length is x)."""
    d = len(n)
    return [torch.arange(m, dtype=torch.float64, device=DEV).reshape([-1 if d - 1 - k == a else 1 for k in range(d)])
            for a, m in enumerate(n)]


def _near(x, c, n):
    """Periodic distance along one axis of length n."""
    t = (x - c).abs()
    return torch.minimum(t, n - t)


def _disks(r, nx, ny, count, rmin, rmax, x_range=(0.0, 1.0), gap=2.0 * W_IFACE):
    """Up to `count` disks that keep `gap` from each other (periodic distance)."""
    out, tries = [], 0
    while len(out) < count and tries < 2000:
        tries += 1
        rad = min(r.uniform(rmin, rmax), 0.2 * min(nx, ny))
        cx, cy = nx * r.uniform(*x_range), ny * r.random()
        if all(math.hypot(min(abs(cx - a), nx - abs(cx - a)), min(abs(cy - b), ny - abs(cy - b))) >= rad + c + gap
               for a, b, c in out):
            out.append((cx, cy, rad))
    return out


def _setup(case, seed):
    """Initial fields (one float32 pair per instance), parameters, periodicity and the diagnostics' arguments."""
    r = random.Random(seed * 1000003 + 17)
    kind, nx, ny, nz = case["kind"], case["nx"], case["ny"], case["nz"]
    if kind == "wall":
        x, y = _axes(nx, ny)
        rows = max(6, ny // 8)
        yw, R = rows - 0.5, 0.39 * ny * r.uniform(0.9, 1.05)
        xc = nx // 2 + r.randrange(-nx // 8, nx // 8 + 1)
        phi0 = _diffuse(yw - y).expand(ny, nx)
        phi1 = (1.0 - phi0) * _diffuse(R - torch.hypot(x - xc, y - yw))
        prm = dict(theta_deg=r.uniform(30.0, 150.0), kappa=0.0, sigma=0.01, d0=0.5)
        return [(phi0, phi1)], [prm], (True, False, False), dict(mode=0, column=xc)
    if kind == "channel":
        x, y = _axes(nx, ny)
        phi0 = torch.zeros(ny, nx, dtype=torch.float64, device=DEV)
        for cx, cy, rad in _disks(r, nx, ny, 3, 6.0, ny / 8.0, x_range=(0.4, 0.85)):
            phi0 = torch.maximum(phi0, _diffuse(rad - torch.hypot(x - cx, y - cy)))
        R = ny * r.uniform(0.15, 0.25)
        phi1 = (1.0 - phi0) * _diffuse(R - torch.hypot(x - 0.2 * nx, y - ny * r.uniform(0.4, 0.6)))
        prm = dict(theta_deg=r.uniform(60.0, 120.0), kappa=0.1, sigma=0.005, rho=(2.0, 2.0, 1.0),
                   mu=(0.1, 0.1, 0.05), d0=0.5)
        yy = (np.arange(ny) + 0.5 - ny / 2) / (ny / 2)
        prof = 1.5 * r.uniform(0.008, 0.015) * (1.0 - yy ** 2)
        inlet = np.stack([prof, 0 * prof]).astype(np.float32)
        return [(phi0, phi1)], [prm], (False, False, False), dict(inlet=inlet, phi_in=0.0, p_out=0.0)
    if kind == "disk":
        x, y = _axes(nx, ny)
        m = min(nx, ny)
        Rs, R0 = 0.156 * m * r.uniform(0.9, 1.1), 0.117 * m * r.uniform(0.9, 1.1)
        xc, yc = nx // 2 + r.randrange(-m // 16, m // 16 + 1), ny // 2 + r.randrange(-m // 16, m // 16 + 1)
        phi0 = _diffuse(Rs - torch.hypot(x - xc, y - yc))
        phi1 = (1.0 - phi0) * _diffuse(R0 - torch.hypot(x - xc, y - (yc + Rs)))
        thetas = [30.0 + 120.0 * (k + r.random()) / case["batch"] for k in range(case["batch"])]
        prm = [dict(theta_deg=t, kappa=R0 / Rs, sigma=0.01, rho=(10.0, 10.0, 1.0), mu=(0.1, 0.1, 0.01), d0=0.5)
               for t in thetas]
        return [(phi0, phi1)] * case["batch"], prm, (True, True, False), dict(mode=1, column=xc, y_c=yc, disk_radius=Rs)
    if kind == "uneven":
        fields, prm = [], []
        for nx, ny in _sizes(case):
            x, y = _axes(nx, ny)
            disks = _disks(r, nx, ny, r.randrange(1, 7), 8.0, 40.0)
            phi0 = torch.zeros(ny, nx, dtype=torch.float64, device=DEV)
            for cx, cy, rad in disks:
                phi0 = torch.maximum(phi0, _diffuse(rad - torch.hypot(_near(x, cx, nx), _near(y, cy, ny))))
            big = max(disks, key=lambda t: t[2])
            R0 = min(r.uniform(10.0, 60.0), 0.2 * nx)
            drop = _diffuse(R0 - torch.hypot(_near(x, big[0], nx), _near(y, (big[1] + big[2]) % ny, ny)))
            fields.append((phi0, (1.0 - phi0) * drop))
            prm.append(dict(theta_deg=r.uniform(30.0, 150.0), kappa=R0 / big[2], sigma=0.01, d0=0.5))
        return fields, prm, (True, True, False), {}
    if kind == "porous":
        # spheres of the pack's radii on a jittered grid, about 40 % solid, fluid 1 in the slab next to the inlet
        x, y, z = _axes(nx, ny, nz)
        phi0 = torch.zeros(nz, ny, nx, dtype=torch.float32, device=DEV)
        m = max(1, round(nx / 29.0))
        pitch = [nx / m, ny / m, nz / m]
        for k in range(m ** 3):
            cell = (k % m, (k // m) % m, k // (m * m))
            c = [(a + 0.5 + r.uniform(-0.1, 0.1)) * p for a, p in zip(cell, pitch)]
            rad = r.uniform(0.36, 0.47) * min(pitch)
            lo = [max(0, int(t - rad - 8)) for t in c]
            hi = [int(t + rad + 9) for t in c]
            sub = phi0[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]]
            dist = torch.sqrt((x[..., lo[0]:hi[0]] - c[0]) ** 2 + (y[:, lo[1]:hi[1]] - c[1]) ** 2 +
                              (z[lo[2]:hi[2]] - c[2]) ** 2)
            sub.copy_(torch.maximum(sub, _diffuse(rad - dist).float()))
        phi0 = phi0.double()
        phi1 = (1.0 - phi0) * _diffuse(nx / 8.0 - x)
        prm = dict(theta_deg=120.0, kappa=0.0, sigma=0.01, d0=1.0 / 3.0, body_force=(1e-6, 0.0, 0.0))
        return [(phi0, phi1)], [prm], (True, True, True), dict(flux=True)
    # drop3d: a spherical drop on a flat solid layer, walls in z, density and viscosity ratio 10
    x, y, z = _axes(nx, ny, nz)
    zw = max(6, nz // 8) - 0.5
    R = 0.3 * min(nx, ny, nz) * r.uniform(0.9, 1.1)
    xc, yc = nx / 2 + r.uniform(-3, 3), ny / 2 + r.uniform(-3, 3)
    phi0 = _diffuse(zw - z).expand(nz, ny, nx)
    phi1 = (1.0 - phi0) * _diffuse(R - torch.sqrt((x - xc) ** 2 + (y - yc) ** 2 + (z - zw) ** 2))
    prm = dict(theta_deg=r.uniform(45.0, 135.0), kappa=0.0, sigma=0.005, rho=(10.0, 10.0, 1.0), mu=(0.1, 0.1, 0.01),
               d0=0.25, eta_hat=0.05 if case["lattice"] == "D3Q15" else 0.1)
    return [(phi0, phi1)], [prm], (True, True, False), {}


class _Run:
    """What a program keeps between passes: the context or network, its inputs on the device, its output buffers."""


def _pinned(*shape):
    return torch.empty(shape, dtype=torch.float32, pin_memory=True).numpy()


def _prepare_lattice(case, seed):
    fields, prm, periodic, diag = _setup(case, seed)
    s = _Run()
    s.case, s.diag, s.batch = case, diag, case["batch"]
    s.phi0 = torch.cat([a.reshape(-1) for a, _ in fields]).float()
    s.phi1 = torch.cat([b.reshape(-1) for _, b in fields]).float()
    params = [L.lbm_default_params(W=W_IFACE, M_deg=0.1, **p) for p in prm]
    if case["kind"] == "uneven":
        s.ctx = L.MultiContext(_sizes(case), periodic=periodic[:2], batch=params)
        d = 2
    else:
        s.ctx = L.Context(LATTICE[case["lattice"]], case["nx"], case["ny"], case["nz"], periodic=periodic,
                          batch=params, flags=L.LBM_STORE_G_F16 if case["f16"] else 0)
        d = s.ctx.d
    total = s.phi0.numel()
    s.out = _pinned(total), _pinned(d * total), _pinned(total)
    torch.cuda.synchronize()          # the context works on its own stream
    L.lbm_set_solid_device(s.ctx.ctx, s.phi0.data_ptr())
    if "inlet" in diag:
        s.ctx.set_inout(3, diag["inlet"], diag["phi_in"], diag["p_out"])
    s.ctx.sync()
    return s


def _run_lattice(s):
    h, n = s.ctx.ctx, s.case["steps"]
    L.lbm_set_phase_device(h, s.phi1.data_ptr())
    s.ctx.step(n)
    r = {}
    if s.case["angle"]:               # the angle a relaxation study samples
        a = s.diag
        r["angle"] = [list(s.ctx.contact_angle(k, a["mode"], a["column"], a.get("y_c", 0.0), a.get("disk_radius", 0.0)))
                      for k in range(s.batch)]
    if "flux" in s.diag:              # the sums of the relative permeability
        f = s.ctx.phase_flux(0, 0)
        r["flux"] = [f[k] for k in ("q1", "q2", "q", "s1", "s2")]
    phi1, u, p = s.out
    fp = ctypes.POINTER(ctypes.c_float)
    st = L.library().lbm_get_fields(h, *(a.ctypes.data_as(fp) for a in (phi1, u, p)))
    if st:
        raise L.LbmError(st, "lbm_get_fields")
    r.update(phi1=phi1, u=u, p=p)
    return r


def _widths(case):
    return tuple(int(t) for t in case["widths"].split("-"))


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _layer_inputs(case, seed):
    """x: activations behind a ReLU; dy: a gradient through one; weights He-initialised."""
    g = _gen(seed)
    n, h, w, ci, co = (case[k] for k in ("n", "h", "w", "cin", "cout"))
    rnd = lambda *s: torch.randn(s, generator=g, device=DEV)
    x = rnd(n, h, w, ci).relu_()
    wt = (rnd(9, co, ci) * math.sqrt(2.0 / (9 * ci))).bfloat16()
    bias = 0.1 * rnd(co)
    dy = 1e-4 * rnd(n, h, w, co) * (torch.rand(n, h, w, co, generator=g, device=DEV) < 0.5)
    return x, wt, bias, dy


def _images(case, seed):
    """A disk and a droplet per image, the field the network has to reach (a shifted droplet) and cos theta."""
    r = random.Random(seed * 31 + 7)
    n, h, w = case["n"], case["h"], case["w"]
    x, y = _axes(w, h)
    phi0, phi1, target, cth = [], [], [], []
    for _ in range(n):
        m = min(h, w)
        Rs, R0 = m * r.uniform(0.06, 0.15), m * r.uniform(0.06, 0.2)
        cx, cy = w / 2 + r.uniform(-4, 4), h / 2 + r.uniform(-4, 4)
        a = _diffuse(Rs - torch.hypot(x - cx, y - (cy - Rs)))
        phi0.append(a)
        phi1.append((1 - a) * _diffuse(R0 - torch.hypot(x - cx, y - cy)))
        target.append((1 - a) * _diffuse(0.9 * R0 - torch.hypot(x - cx, y - (cy + 0.2 * R0))))
        cth.append(math.cos(math.radians(r.uniform(30.0, 150.0))))
    f = lambda t: torch.stack(t).float().contiguous()
    return f(phi0), f(phi1), f(target), torch.tensor(cth, dtype=torch.float32, device=DEV)


def _prepare_net(case, seed):
    s = _Run()
    s.case = case
    if case["kind"] in ("conv", "wgrad"):
        n, h, w, ci, co = (case[k] for k in ("n", "h", "w", "cin", "cout"))
        s.x, s.wt, s.bias, s.dy = _layer_inputs(case, seed)
        if case["kind"] == "conv":
            s.y = torch.empty(n, h, w, co, device=DEV)
        else:
            s.dw, s.db = torch.empty(9, co, ci, device=DEV), torch.empty(co, device=DEV)
            s.work = torch.empty(_nn.wgrad_workspace(n, h, w, ci, co), device=DEV)
        return s
    s.phi0, s.phi1, s.target, s.cth = _images(case, seed)
    s.net = WarmStartNet(_widths(case), n=case["n"], h=case["h"], w=case["w"], seed=seed)
    s.field = torch.empty_like(s.phi1)
    return s


def _run_net(s):
    c = s.case
    if c["kind"] == "conv":
        _nn.conv3x3(s.x.data_ptr(), s.wt.data_ptr(), s.bias.data_ptr() if c["relu"] else 0, s.y.data_ptr(), c["n"],
                    c["h"], c["w"], c["cin"], c["cout"], c["relu"])
        return s.y
    if c["kind"] == "wgrad":
        _nn.conv3x3_wgrad(s.x.data_ptr(), s.dy.data_ptr(), s.dw.data_ptr(), s.db.data_ptr(), s.work.data_ptr(),
                          s.work.numel(), c["n"], c["h"], c["w"], c["cin"], c["cout"])
        return {"dw": s.dw, "db": s.db}
    if c["kind"] == "train":
        # the rate at the very start of the schedule's warm-up, zero: the optimiser does all its work, and every pass
        # sees the same weights
        loss = s.net.train_step(s.phi0, s.phi1, s.cth, s.target, 0.0)
        return {"out": s.net.act["out"], "loss": loss, "dW": s.net.dW, "db": s.net.db}
    return {"out": s.net.act["out"], "field": s.net.predict(s.phi0, s.phi1, s.cth, s.field)}


def prepare(case, seed):
    return _prepare_lattice(case, seed) if "lattice" in case else _prepare_net(case, seed)


def run(state):
    return _run_lattice(state) if "lattice" in state.case else _run_net(state)


# ---------------------------------------------------------------------------------------------------
# 64-bit restatement of the step, batched over instances: fields [b, (z,) y, x], populations [q, b, ...]
# ---------------------------------------------------------------------------------------------------
def _velocities(name):
    if name == "D2Q9":
        return [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
    axes = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
    if name == "D3Q15":
        return axes + [(x, y, z) for z in (1, -1) for y in (1, -1) for x in (1, -1)]
    edges = []
    for a, b in ((0, 1), (0, 2), (1, 2)):
        for s, t in ((1, 1), (-1, -1), (1, -1), (-1, 1)):
            v = [0, 0, 0]
            v[a], v[b] = s, t
            edges.append(tuple(v))
    return axes + edges


def _weights(name, d0, c):
    if name == "D2Q9":
        by = [(1 - d0) ** 2, (d0 - d0 ** 2) / 2, d0 ** 2 / 4]
    elif name == "D3Q15":
        by = [1 - 3 * d0 + 2 * d0 ** 2, (d0 - d0 ** 2) / 2, None, d0 ** 2 / 8]
    else:
        by = [1 - 3 * d0 + 3 * d0 ** 2, (d0 - 2 * d0 ** 2) / 2, d0 ** 2 / 4]
    return np.array([by[sum(abs(a) for a in ci)] for ci in c])


def _hermite(name, c, w):
    """Rows orthogonal under w (weighted Gram-Schmidt of monomials) and the rate group of each."""
    d = len(c[0])
    e = lambda *axes: tuple(sum(1 for a in axes if a == k) for k in range(d))
    pairs = [(a, b) for a in range(d) for b in range(a + 1, d)]
    rows = [(e(), "0")] + [(e(a), "1") for a in range(d)] + [(e(a, a), "2a") for a in range(d)]
    rows += [(e(a, b), "2b") for a, b in pairs]
    if name == "D3Q15":
        rows += [(e(a, b, b), "3") for a, b in ((0, 1), (1, 2), (2, 0))] + [(e(0, 1, 2), "3"), (e(0, 0, 1, 1), "4")]
    else:
        rows += [(e(a, b, b), "3") for a in range(d) for b in range(d) if a != b]
        rows += [(e(a, a, b, b), "4") for a, b in pairs]
    v = np.array(c, dtype=float)
    H = []
    for ex, _ in rows:
        h = np.prod([v[:, a] ** ex[a] for a in range(d)], axis=0)
        m = h.copy()
        for k in H:
            h = h - (w * m * k).sum() / (w * k * k).sum() * k
        H.append(h)
    H = np.array(H)
    inv = (w * H).T / (w * H * H).sum(axis=1)
    return H, inv, [g for _, g in rows]


class _Exact:
    def __init__(self, name, prm, periodic):
        """prm: parameter dicts of the instances (d0 and eta_hat shared)."""
        full = dict(theta_deg=90.0, kappa=0.0, sigma=0.01, rho=(1.0, 1.0, 1.0), mu=(0.01, 0.01, 0.01), d0=0.5,
                    eta_hat=0.1, body_force=(0.0, 0.0, 0.0))
        prm = [{**full, **p} for p in prm]
        self.c = _velocities(name)
        self.d = d = len(self.c[0])
        self.per = periodic[:d]
        self.cs2 = self.d0 = d0 = prm[0]["d0"]
        self.w = _weights(name, d0, self.c)
        t = lambda a: torch.as_tensor(np.asarray(a, dtype=float), device=DEV)
        col = lambda a: t(a).reshape([-1] + [1] * d)
        H, inv, self.groups = _hermite(name, self.c, self.w)
        self.H, self.inv = t(H), t(inv)
        self.opp = [self.c.index(tuple(-a for a in ci)) for ci in self.c]
        sc = _velocities("D2Q9" if d == 2 else "D3Q19")
        self.sten = list(zip(sc, _weights("D2Q9" if d == 2 else "D3Q19", 1.0 / 3.0, sc)))
        th = np.radians([p["theta_deg"] for p in prm])
        sgn = np.sign([p["theta_deg"] - 90.0 for p in prm])
        sg, ka = np.array([p["sigma"] for p in prm]), np.array([p["kappa"] for p in prm])
        s01 = 9.0 / (1.0 + ka) * (1.0 + 2.0 * sgn * np.sin(np.pi / 4 * np.cos(th)) ** 2) * sg
        s02 = s01 + sg * np.cos(th)
        gam = [s01 + s02 - sg, s01 + sg - s02, s02 + sg - s01]
        self.gam = [col(g) for g in gam]
        self.gT = 3.0 / (1.0 / self.gam[0] + 1.0 / self.gam[1] + 1.0 / self.gam[2])
        self.M = 0.1
        self.eta = np.array([p["eta_hat"] for p in prm]) / gam[1]
        self.s1 = col(1.0 / (0.5 + self.M / (gam[1] * self.eta * d0)))
        self.eta = col(self.eta)
        self.rho = [col([p["rho"][k] for p in prm]) for k in range(3)]
        self.mu = [col([p["mu"][k] for p in prm]) for k in range(3)]
        self.b = [col([p["body_force"][k] for p in prm]) for k in range(d)]
        self.K = 1.0 - d0 if d == 2 else 1.0 - 2.0 * d0
        self.h = (1 - d0, 2 - 4 * d0, (1 - 3 * d0) / 2) if d == 2 else (1 - d0, 3 - 7 * d0, 1 - 3 * d0)
        self.inlet = None

    def ax(self, a):
        return self.d - a            # array axis of component a (axis 0 is the instance)

    def pad(self, v):
        for a in range(self.d):
            k, n = self.ax(a), v.shape[self.ax(a)]
            lo, hi = v.narrow(k, 0, 1), v.narrow(k, n - 1, 1)
            v = torch.cat([hi, v, lo] if self.per[a] else [lo, v, hi], dim=k)
        return v

    def nb(self, P, ci):
        for a in range(self.d):
            k = self.ax(a)
            P = P.narrow(k, 1 + ci[a], P.shape[k] - 2)
        return P

    def grad_lap(self, v):
        P, g, lap = self.pad(v), [0.0] * self.d, torch.zeros_like(v)
        for ci, wi in self.sten:
            if any(ci):
                n = self.nb(P, ci)
                lap += 6.0 * wi * (n - v)
                for a in range(self.d):
                    if ci[a]:
                        g[a] = g[a] + 3.0 * wi * ci[a] * n
        return g, lap

    def mubar(self, phi0, phi1, lap0, lap1):
        mu = []
        for g, ph, lp in zip(self.gam, (phi0, phi1, 1 - phi0 - phi1), (lap0, lap1, -lap0 - lap1)):
            mu.append(g * (12.0 / W_IFACE * ph * (1 - ph) * (1 - 2 * ph) - 0.75 * W_IFACE * lp))
        return mu, self.gT / 3.0 * ((mu[1] - mu[0]) / self.gam[0] + (mu[1] - mu[2]) / self.gam[2])

    def feq(self, phi, em, u):
        out = []
        for i, ci in enumerate(self.c):
            cu = sum(ci[a] * u[a] for a in range(self.d)) if any(ci) else 0.0
            out.append(phi + (self.w[0] - 1) * em if i == 0 else self.w[i] * (em + phi * cu / self.cs2))
        return torch.stack(out)

    def second(self, ci, diag, off):
        """c c : (symmetric tensor) / its Hermite norms."""
        d, cs2 = self.d, self.cs2
        v = sum((ci[a] ** 2 - cs2) * diag[a] for a in range(d)) / (cs2 - cs2 ** 2)
        return v + sum(ci[a] * ci[b] * off[a, b] for a in range(d) for b in range(a + 1, d) if ci[a] * ci[b]) / cs2 ** 2

    def geq(self, p, rho, u, S):
        d = self.d
        diag = [rho * u[a] * u[a] - S[a] * u[a] for a in range(d)]
        off = {(a, b): rho * u[a] * u[b] - 0.5 * (S[a] * u[b] + u[a] * S[b]) for a in range(d) for b in range(a + 1, d)}
        out = []
        for i, ci in enumerate(self.c):
            cu = sum(ci[a] * u[a] for a in range(d)) if any(ci) else 0.0
            lam = (self.w[0] - 1) * p / self.cs2 if i == 0 else self.w[i] * p / self.cs2
            out.append(lam + self.w[i] * (rho * cu / self.cs2 + self.second(ci, diag, off)))
        return torch.stack(out)

    def moments(self, v):
        return torch.matmul(self.H, v.reshape(v.shape[0], -1)).reshape(v.shape)

    def collide(self, v, veq, src, rates):
        m, r = self.moments(v - veq), self.moments(src)
        for k, g in enumerate(self.groups):
            m[k] = (1 - 0.5 * rates[g]) * r[k] - rates[g] * m[k]
        return v + torch.matmul(self.inv, m.reshape(m.shape[0], -1)).reshape(m.shape)

    def stream(self, v):
        out = torch.empty_like(v)
        for i, ci in enumerate(self.c):
            t = v[i]
            for a in range(self.d):
                if ci[a]:
                    t = torch.roll(t, ci[a], dims=self.ax(a))
            for a in range(self.d):
                if ci[a] and not self.per[a]:
                    t = t.clone()
                    k = self.ax(a)
                    at = 0 if ci[a] > 0 else t.shape[k] - 1
                    t.narrow(k, at, 1).copy_(v[self.opp[i]].narrow(k, at, 1))
            out[i] = t
        return out

    def open_columns(self):
        """Velocity inlet at the first column, pressure outlet at the last (non-equilibrium extrapolation)."""
        nf, ng = self.f.clone(), self.g.clone()
        for xb, xf in ((0, 1), (-1, -2)):
            f, g = self.f[..., xf], self.g[..., xf]
            sub = lambda v: v.squeeze(-1)
            phi = f.sum(0)
            dens = lambda p0, p1: sub(self.rho[0]) * p0 + sub(self.rho[1]) * p1 + sub(self.rho[2]) * (1 - p0 - p1)
            rf = dens(self.phi0[..., xf], phi)
            u = [sum(ci[a] * g[i] for i, ci in enumerate(self.c)) / rf for a in range(self.d)]
            p = self.cs2 / (1 - self.w[0]) * (g[1:].sum(0) - self.w[0] * rf * sum(t * t for t in u) / (1 - self.cs2))
            if xb == 0:
                pb, ub, pr = torch.full_like(phi, self.phi_in), [t.expand_as(phi) for t in self.inlet], p
            else:
                pb, ub, pr = phi, u, torch.full_like(phi, self.p_out)
            zero = torch.zeros_like(phi)
            Z = [zero] * self.d
            nf[..., xb] = f + self.feq(pb, zero, ub) - self.feq(phi, zero, u)
            ng[..., xb] = g + self.geq(pr, dens(self.phi0[..., xb], pb), ub, Z) - self.geq(p, rf, u, Z)
        self.f, self.g = nf, ng

    def start(self, phi0, phi1):
        self.phi0 = phi0
        self.g0, self.lap0 = self.grad_lap(phi0)
        _, lap1 = self.grad_lap(phi1)
        z = torch.zeros_like(phi1)
        self.f = self.feq(phi1, self.eta * self.mubar(phi0, phi1, self.lap0, lap1)[1], [z] * self.d)
        self.g = torch.zeros_like(self.f)
        self.hp, self.hu, self.hS = phi1, [z] * self.d, [z] * self.d

    def step(self):
        d, cs2, phi0 = self.d, self.cs2, self.phi0
        r, mv = self.rho, self.mu
        phi1 = self.f.sum(0)
        phi2 = 1 - phi0 - phi1
        g1, lap1 = self.grad_lap(phi1)
        mu, mub = self.mubar(phi0, phi1, self.lap0, lap1)
        gm, _ = self.grad_lap(mub)
        deg = phi1 * (1 - phi1) * (1 - phi0)
        S = [(r[1] - r[2]) * self.M * deg * gm[a] / self.gam[1] for a in range(d)]
        rho = r[0] * phi0 + r[1] * phi1 + r[2] * phi2
        gr = [(r[0] - r[2]) * self.g0[a] + (r[1] - r[2]) * g1[a] for a in range(d)]
        muv = mv[0] * phi0 + mv[1] * phi1 + mv[2] * phi2
        Fv = [(mu[0] - mu[2]) * self.g0[a] + (mu[1] - mu[2]) * g1[a] + (1 - phi0) * self.b[a] for a in range(d)]
        for a in range(d):
            for b in range(a + 1, d):
                gab, _ = self.grad_lap(self.hS[a] * self.hu[b] - self.hu[a] * self.hS[b])
                Fv[b] = Fv[b] + 0.5 * gab[a]
                Fv[a] = Fv[a] - 0.5 * gab[b]
        us = [(sum(ci[a] * self.g[i] for i, ci in enumerate(self.c) if ci[a]) + 0.5 * Fv[a]) / rho for a in range(d)]
        u = [t - 0.5 * phi0 * t for t in us]
        Ft = [Fv[a] - phi0 * rho * us[a] for a in range(d)]
        nu = muv / (rho * (1 - phi0).clamp_min(2.0 ** -24))
        s2a, s2b = 1 / (0.5 + 2 * nu / (1 - cs2)), 1 / (0.5 + nu / cs2)
        udg = sum(u[a] * gr[a] for a in range(d))
        q = sum((rho * u[a] - S[a]) * u[a] for a in range(d))
        rp = r[0] * phi0 + r[1] * self.hp + r[2] * (1 - phi0 - self.hp)
        qp = sum((rp * self.hu[a] - self.hS[a]) * self.hu[a] for a in range(d))
        H = self.K * ((self.h[0] - self.h[1]) / s2a + self.h[2])
        p = cs2 / (1 - self.w[0]) * (self.g[1:].sum(0) + (0.5 + H) * udg - self.w[0] * q / (1 - cs2) +
                                     0.5 * self.K * (q - qp))
        # CH
        em = self.eta * mub
        src = [phi1 * u[a] - self.hp * self.hu[a] + cs2 * (1 - deg) * self.eta * gm[a] for a in range(d)]
        R = torch.stack([self.w[i] * sum(ci[a] * src[a] for a in range(d)) / cs2 if any(ci) else torch.zeros_like(phi1)
                         for i, ci in enumerate(self.c)])
        ch = {"0": 1.0, "1": self.s1, "2a": 1.0, "2b": 1.0, "3": 1.0, "4": 1.0}
        f = self.collide(self.f, self.feq(phi1, em, u), R, ch)
        # NS
        sym = lambda A, B, a, b: 0.5 * (A[a] * B[b] + B[a] * A[b])
        m2 = {}
        for a in range(d):
            for b in range(a, d):
                v = u[a] * Fv[b] + Fv[a] * u[b] - sym(S, u, a, b) + sym(self.hS, self.hu, a, b)
                v = v + cs2 * (u[a] * gr[b] + gr[a] * u[b])
                m2[a, b] = v + (1 - 3 * cs2) * udg if a == b else v
        G = torch.stack([self.w[i] * (udg + (sum(ci[a] * Ft[a] for a in range(d)) / cs2 if any(ci) else 0.0) +
                                      self.second(ci, [m2[a, a] for a in range(d)], m2)) for i, ci in enumerate(self.c)])
        ns = {"0": s2a, "1": 1.0, "2a": s2a, "2b": s2b, "3": 1.0, "4": s2a}
        g = self.collide(self.g, self.geq(p, rho, u, S), G, ns)
        self.f, self.g = self.stream(f), self.stream(g)
        if self.inlet is not None:
            self.open_columns()
        self.hp, self.hu, self.hS, self.p = phi1, u, S, p


def _exact_lattice(case, seed):
    fields, prm, periodic, diag = _setup(case, seed)
    sizes = _sizes(case)
    out = [None] * len(sizes)
    for size in sorted(set(sizes)):
        at = [k for k, s in enumerate(sizes) if s == size]
        e = _Exact(case["lattice"], [prm[k] for k in at], periodic)
        if "inlet" in diag:
            e.inlet = [torch.as_tensor(v, device=DEV).double()[None] for v in diag["inlet"]]
            e.phi_in, e.p_out = diag["phi_in"], diag["p_out"]
        f32 = lambda j: torch.stack([fields[k][j].float().double() for k in at])
        e.start(f32(0), f32(1))
        for _ in range(case["steps"]):
            e.step()
        for j, k in enumerate(at):
            out[k] = (e.hp[j], torch.stack([v[j] for v in e.hu]), e.p[j])
    r = {}
    if case["angle"]:
        r["angle"] = [[None, None]] * case["batch"]     # read off the fields below by a fixed construction
    if "flux" in diag:
        (p1, u, _), p0 = out[0], fields[0][0].float().double()
        pore = p0 <= 0.5
        p2, ux = 1 - p0 - p1, u[0]
        s = [float((t * pore).sum()) for t in (p1 * ux, p2 * ux, ux, p1, p2)]
        r["flux"] = [s[0], s[1], s[2], s[3] / (s[3] + s[4]), s[4] / (s[3] + s[4])]
    for j, key in enumerate(("phi1", "u", "p")):
        r[key] = torch.cat([o[j].reshape(-1) for o in out])
    return r


# ---------------------------------------------------------------------------------------------------
# 64-bit restatement of the warm start: operands of the convolutions rounded to BF16, as they are documented
# ---------------------------------------------------------------------------------------------------
def _bf(t):
    return t.float().bfloat16().double()


class _Conv(torch.autograd.Function):
    """3x3 convolution, NHWC, zero padding; wt [tap][cout][cin]; BF16 operands in all three products."""

    @staticmethod
    def shifts(x):
        n, h, w, c = x.shape
        P = F.pad(x, (0, 0, 1, 1, 1, 1))
        return [P[:, t // 3:t // 3 + h, t % 3:t % 3 + w].reshape(-1, c) for t in range(9)]

    @staticmethod
    def forward(ctx, x, wt, b):
        ctx.save_for_backward(x, wt)
        xr, wr = _bf(x), _bf(wt)
        y = sum(s @ wr[t].T for t, s in enumerate(_Conv.shifts(xr)))
        return y.reshape(*x.shape[:3], -1) + b

    @staticmethod
    def backward(ctx, dy):
        x, wt = ctx.saved_tensors
        dr, wr = _bf(dy), _bf(wt)
        flat = dr.reshape(-1, dr.shape[-1])
        dw = torch.stack([flat.T @ s for s in _Conv.shifts(_bf(x))])
        dx = sum(s @ wr[8 - t] for t, s in enumerate(_Conv.shifts(dr)))
        return dx.reshape(x.shape), dw, dy.sum((0, 1, 2))


def _net(x, params, levels):
    it = iter(params)
    conv = lambda v: _Conv.apply(v, *next(it))
    pool = lambda v: v.reshape(v.shape[0], v.shape[1] // 2, 2, v.shape[2] // 2, 2, -1).mean((2, 4))
    up = lambda v: v.repeat_interleave(2, 1).repeat_interleave(2, 2)
    skip, h = [], x
    for k in range(levels):
        h = conv(conv(pool(h) if k else h).relu()).relu()
        skip.append(h)
    for k in range(levels - 2, -1, -1):
        h = conv(conv(up(h)).relu() + skip[k]).relu()
    return conv(h)


def _exact_net(case, seed):
    if case["kind"] in ("conv", "wgrad"):
        x, wt, bias, dy = _layer_inputs(case, seed)
        x = x.double()
        if case["kind"] == "conv":
            y = _Conv.apply(x, wt.double(), bias.double() if case["relu"] else 0.0)
            return y.relu() if case["relu"] else y
        d = _bf(dy).reshape(-1, dy.shape[-1])
        return {"dw": torch.stack([d.T @ s for s in _Conv.shifts(_bf(x))]), "db": dy.double().sum((0, 1, 2))}
    phi0, phi1, target, cth = _images(case, seed)
    widths, n = _widths(case), case["n"]
    rng = np.random.default_rng(seed)       # the network's own initialisation: He, a small output layer
    shapes, params = layer_shapes(widths), []
    for k, (ci, co) in enumerate(shapes):
        std = np.sqrt(2.0 / (9 * ci)) * (0.1 if k == len(shapes) - 1 else 1.0)
        wt = torch.tensor(rng.normal(0.0, std, (9, co, ci)), dtype=torch.float32, device=DEV).double()
        params.append((wt.requires_grad_(), torch.zeros(co, dtype=torch.float64, device=DEV).requires_grad_()))
    x = torch.zeros(*phi0.shape, 16, dtype=torch.float64, device=DEV)
    x[..., 0], x[..., 1], x[..., 2] = phi0.double(), phi1.double(), cth.double().reshape(-1, 1, 1)
    with torch.set_grad_enabled(case["kind"] == "train"):
        out = _net(x, params, len(widths))
    if case["kind"] == "train":
        err = phi1.double() + out[..., 0] - target.double()
        (err.square().sum() / err.numel()).backward()
        return {"out": out.detach(), "loss": err.detach().square().sum().reshape(1), "dW": [w.grad for w, _ in params],
                "db": [b.grad for _, b in params]}
    hi = (1.0 - phi0.double()).clamp_min(0.0)
    q = torch.minimum((phi1.double() + out[..., 0]).clamp_min(0.0), hi)
    for _ in range(3):                      # the projection's mass-correction passes
        bump = torch.where(hi > 0, q * (hi - q) / torch.where(hi > 0, hi, 1.0), 0.0)
        lam = ((phi1.double().sum((1, 2)) - q.sum((1, 2))) / bump.sum((1, 2))).clamp(-1.0, 1.0)
        q = q + lam.reshape(n, 1, 1) * bump
    return {"out": out, "field": q}


def exact(case, seed):
    with torch.no_grad() if case["kind"] != "train" else torch.enable_grad():
        return _exact_lattice(case, seed) if "lattice" in case else _exact_net(case, seed)
