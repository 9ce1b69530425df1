"""What a user of the library has it do, as cases that can be timed and compared.

A case is one call of a user's program on inputs of the sizes and
distributions of this repository's configurations, tests and benchmark:

* ``window``   one fluid step: K substeps through ``Simulator.run`` (Verlet
               lists, the fused substep), then the positions;
* ``grad``     the differentiable window: ``GicWindow`` forward and backward
               to the initial velocities, c_drag and mu;
* ``parts``    the same substeps through the separate entry points
               (``gic_sort``, ``gic_contact``, ``gic_g2p_couple``,
               ``gic_integrate``, ``gic_p2g``);
* ``host``     ``gic_window_forward_host``: the window on pinned host buffers;
* ``project``  ``gic_project``: the two pressure projections that consume
               alpha_s.

Inputs are made on the GPU from the seed.  ``exact`` restates the method in
64-bit torch operations with absolute positions.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import torch

from paper_2504_00745_gb300 import gic
from paper_2504_00745_gb300.window import GicWindow, Simulator

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64
FRAC = 1 << 30


# ------------------------------------------------------------------ the cases

def _window(name, packing, n, grid, h, r, K, dt, **more):
    c = dict(name=name, kind="window", packing=packing, n=n, nx=grid[0], ny=grid[1], nz=grid[2], h=h, r=r, nn=2.2,
             fx=1.0, fy=1.0, K=K, dt=dt, k_n=1.0e5, bits=32, fluid="modes", amp=0.5, sigma=0.0)
    c.update(more)
    return c


def listed():
    return [
        # the plain configuration, all FP64: the smallest call, where launches and latency count
        _window("plain_8k_fp64", "cubic", 8000, (32, 32, 32), 1 / 32, 0.004, 10, 1e-5, fx=0.2, fy=0.2, bits=64,
                fluid="noise", amp=0.1),
        # a small overlapping block on the production precision: every granule has contacts, also with the walls
        _window("block_7k", "rough", 7001, (32, 32, 32), 1 / 32, 0.004, 10, 1e-5, nn=1.98, fx=0.2, fy=0.2,
                fluid="noise", amp=0.1),
        # the dam break: a corner column, the ordinary forward simulation (FP32)
        _window("dam_break_1m", "fcc", 1_000_000, (128, 128, 128), 1 / 128, 0.0015, 100, 2e-5, nn=2.208, fx=0.3),
        # the same in all FP64, the accuracy reference on the GPU (a fifth of the substeps)
        _window("dam_break_1m_fp64", "fcc", 1_000_000, (128, 128, 128), 1 / 128, 0.0015, 20, 2e-5, nn=2.208, fx=0.3,
                bits=64),
        # a polydisperse bed under shear: dense, lognormal radii, many granules per contact cell
        _window("bed_8m", "bed", 8_000_000, (256, 256, 256), 1 / 256, 8e-4, 10, 1e-5, k_n=20.0, fluid="shear", amp=0.8),
        # the scale sweep: the largest single-GPU workload
        _window("sweep_16m", "fcc", 16_000_000, (384, 384, 384), 1 / 384, 6e-4, 20, 1e-5, nn=2.145, amp=1.0),
        # wet sand: the capillary pair force between near neighbours, odd sizes, a grid that is not a cube
        _window("wet_300k", "wet", 300_007, (96, 80, 72), 1 / 96, 0.002, 20, 1e-5, nn=2.02, fx=0.7, fy=0.6,
                k_n=400.0, sigma=0.07),
        # the differentiable window: loss on the final positions, gradients through 50 substeps
        _window("grad_100k", "loose", 100_000, (64, 64, 64), 1 / 64, 0.002, 50, 2e-5, kind="grad", fx=0.24,
                fy=0.24, amp=0.1),
        # gradients through contacts that last (a contact-stable packing) at the dam break's size
        _window("grad_dense_1m", "dense", 1_000_000, (128, 128, 128), 1 / 128, 0.0015, 20, 1e-5, kind="grad", nn=1.99,
                fx=0.3, k_n=200.0),
        # the separate entry points, for programs that put their own steps between them
        _window("parts_1m", "dense", 1_000_000, (128, 128, 128), 1 / 128, 0.0015, 5, 1e-5, kind="parts", nn=1.99,
                fx=0.3, k_n=200.0),
        # a program that keeps its data on the host: copies included
        _window("host_1m", "fcc", 1_000_000, (128, 128, 128), 1 / 128, 0.0015, 20, 2e-5, kind="host", nn=2.208,
                fx=0.3),
        # the projections of the dam break's grid, once per fluid step, free surface on top
        dict(name="project_128", kind="project", nx=128, ny=128, nz=128, h=1 / 128, dt=2e-3, tol=1e-11, open=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["window", "window", "window", "window", "grad", "parts", "host", "project"])
    if kind == "project":
        nx, ny, nz = (_log(rng, 20, 150) for _ in range(3))
        return dict(kind="project", nx=nx, ny=ny, nz=nz, h=1 / max(nx, ny, nz), dt=rng.choice([1e-3, 2e-3]),
                    tol=1e-11, open=rng.choice([32, 32, 32, 48, 33, 63]))
    most = {"window": 4_000_000, "grad": 500_000, "parts": 2_000_000, "host": 2_000_000}[kind]
    packing = rng.choice(["cubic", "fcc", "dense", "loose", "bed", "wet"] if kind in ("window", "grad")
                         else ["fcc", "dense", "bed"])
    bits = 64 if kind != "host" and rng.random() < 0.25 else 32
    n = _log(rng, 900, most if bits == 32 else min(most, 600_000))
    # the box: MAC cells 4.3 to 7.8 radii wide, as in the configurations (a bed's radius is its median)
    ratio = rng.uniform(4.3, 7.8)
    r = rng.choice([0.004, 0.002, 0.0015, 8e-4, 6e-4])
    if packing == "bed":
        n = max(n, 20_000)
    per_cell = {"loose": 0.3, "cubic": 0.39, "bed": 0.5}.get(packing, 0.55) * ratio ** 3 / (4 / 3 * math.pi)
    cells = n / per_cell
    fx, fy = rng.choice([(1.0, 1.0), (0.3, 1.0), (0.5, 0.5)])
    flat = rng.uniform(0.15, 0.6)  # height of the packing over the width of its footprint
    side = (cells / flat) ** (1 / 3)
    lim = lambda a: int(min(max(a, 10), 340))
    nx, ny = lim(side / fx * rng.uniform(0.9, 1.1)), lim(side / fy * rng.uniform(0.9, 1.1))
    nz = lim(1.7 * cells / max(nx * fx * ny * fy, 1) + 8)
    w = 2650 * 4 / 3 * math.pi * r ** 3
    K = rng.choice([8, 15, 20]) if kind == "grad" else rng.choice([4, 7, 10] if packing == "bed" else [4, 7, 10, 20])
    dt = 1e-5
    # the contact's period well resolved; where granules touch from the start, contacts outlast the window
    k_n = min(1e5, {"dense": 5e-4, "wet": 5e-4, "bed": 6e-5}.get(packing, 0.05) * w / dt ** 2)
    return dict(kind=kind, packing=packing, n=n, nx=nx, ny=ny, nz=nz, h=ratio * r, r=r,
                nn={"dense": 1.985, "wet": 2.02}.get(packing, 2.17), fx=fx, fy=fy, K=K, dt=dt, k_n=k_n, bits=bits,
                fluid=rng.choice(["modes", "noise"]), amp=rng.choice([0.1, 0.5, 1.0]),
                sigma=0.07 if packing == "wet" else 0.0)


# ------------------------------------------------------------------ inputs

def _gen(seed, stream):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1009 + stream) & 0x7FFFFFFF)


def _uniform(gen, shape, lo, hi, dtype=F64):
    return torch.rand(shape, generator=gen, device=DEV, dtype=dtype) * (hi - lo) + lo


def _bed_tile(gen, med):
    """A tile of 12 x 12 x 15 FCC cells, periodic in x and y: lognormal radii
    (sigma 0.25, clipped to [0.5, 2] medians), overlaps moved apart, what is
    left of them (beyond 0.1% of the smallest radius) taken from the larger
    granule."""
    a = 2.35 * med * math.sqrt(2.0)
    M = torch.tensor([24, 24, 30], device=DEV)
    g = torch.stack(torch.meshgrid(*(torch.arange(int(m), device=DEV) for m in M), indexing="ij"), -1).reshape(-1, 3)
    g = g[g.sum(1) % 2 == 0]
    m = g.shape[0]
    where = torch.full((24, 24, 30), -1, dtype=torch.int64, device=DEV)
    where[g[:, 0], g[:, 1], g[:, 2]] = torch.arange(m, device=DEV)
    offs = [(i, j, k) for i in range(-2, 3) for j in range(-2, 3) for k in range(-2, 3)
            if (i + j + k) % 2 == 0 and 0 < i * i + j * j + k * k <= 8]
    nbr = []
    for o in offs:
        t = g + torch.tensor(o, device=DEV)
        inside = (t[:, 2] >= 0) & (t[:, 2] < 30)
        i = where[t[:, 0] % 24, t[:, 1] % 24, t[:, 2].clamp(0, 29)]
        nbr.append(torch.where(inside, i, torch.full_like(i, -1)))
    nbr = torch.stack(nbr, 1)
    has = nbr >= 0
    nb = nbr.clamp(min=0)
    r = (med * torch.exp(0.25 * torch.randn(m, generator=gen, device=DEV, dtype=F64))).clamp(0.5 * med, 2 * med)
    L = torch.tensor([12 * a, 12 * a, 1e9], device=DEV, dtype=F64)
    x = g.to(F64) * (a / 2) + _uniform(gen, (m, 3), -0.02 * med, 0.02 * med)
    x[:, 2] += med

    def overlaps():
        d = x[:, None, :] - x[nb]
        d = d - torch.round(d / L) * L
        dist = torch.where(has, d.norm(dim=2), torch.ones_like(nb, dtype=F64))
        return d, dist, torch.where(has, r[:, None] + r[nb] - dist, torch.zeros_like(dist))

    vol = r ** 3
    for _ in range(120):
        d, dist, ov = overlaps()
        hit = ov > 0
        f = vol[nb] / (vol[nb] + vol[:, None])
        move = (d * (torch.where(hit, ov, torch.zeros_like(ov)) * f / dist)[:, :, None]).sum(1)
        x = x + 1.5 * move / hit.sum(1).clamp(min=1)[:, None]
        x[:, 2] = torch.maximum(x[:, 2], r)
    tol = 1e-3 * float(r.min())
    for _ in range(40):
        _, _, ov = overlaps()
        larger = (r[:, None] > r[nb]) | ((r[:, None] == r[nb]) & (nb > torch.arange(m, device=DEV)[:, None]))
        r = r - torch.where(larger, (ov - tol).clamp(min=0), torch.zeros_like(ov)).amax(1) * (1 + 1e-9)
    x[:, :2] = torch.remainder(x[:, :2], 12 * a)
    return x, r, 12 * a


def _packing(c, seed):
    """Absolute positions (FP64 [n, 3]), radii (FP64) and initial velocities."""
    gen = _gen(seed, 0)
    r0, kind, n = c["r"], c["packing"], c["n"]
    ext = [c["nx"] * c["h"], c["ny"] * c["h"], c["nz"] * c["h"]]
    foot = [ext[0] * c["fx"], ext[1] * c["fy"]]
    if kind == "bed":
        x, r, L = _bed_tile(gen, r0)
        tx, ty = (max(1, int((e - 4 * r0) / L)) for e in ext[:2])
        if ext[0] < L + 4 * r0 or ext[1] < L + 4 * r0 or ext[2] < x[:, 2].max() + 3 * r0:  # a box below one tile
            keep = (x[:, 0] < ext[0] - 4 * r0) & (x[:, 1] < ext[1] - 4 * r0) & (x[:, 2] < ext[2] - 3 * r0)
            x, r = x[keep], r[keep]
        m = x.shape[0]
        reps = min(tx * ty, -(-n // m))
        at = torch.arange(reps, device=DEV)
        off = torch.stack([2 * r0 + (at % tx) * L, 2 * r0 + (at // tx) * L, torch.zeros_like(at, dtype=F64)], 1).to(F64)
        x = (x[None] + off[:, None]).reshape(-1, 3)[:n]
        r = r.repeat(reps)[:n]
        return x, r, torch.zeros_like(x)
    # "dense" and "wet" are stable packings (what touches or is bridged stays so over a window), "rough" is not
    jitter = {"loose": 0.2, "rough": 0.01, "dense": 0.002, "wet": 0.004}.get(kind, 0.05) * r0
    lo = {"rough": 0.985, "dense": 0.985, "wet": 0.985, "loose": 1.25}.get(kind, 1.1) * r0
    if kind in ("cubic", "loose"):
        s = c["nn"] * r0 if kind == "cubic" else (4 / 3 * math.pi * r0 ** 3 / 0.3) ** (1 / 3)
        mx, my = (max(1, int((f - 2 * lo) / s) + 1) for f in foot)
        mz = max(1, int((0.95 * ext[2] - 2 * lo) / s))
        n = min(n, mx * my * mz)
        t = torch.arange(n, device=DEV)
        g = torch.stack([t % mx, t // mx % my, t // (mx * my)], 1)
    else:  # FCC sites: half-lattice coordinates with an even sum, x fastest, then y, then z
        s = c["nn"] * r0 / math.sqrt(2.0)
        mx, my = (max(2, int((f - 2 * lo) / s) + 1) for f in foot)
        mx -= mx % 2
        mz = max(1, int((0.95 * ext[2] - 2 * lo) / s))
        n = min(n, mx // 2 * my * mz)
        t = torch.arange(n, device=DEV)
        j, k = t // (mx // 2) % my, t // (mx // 2 * my)
        g = torch.stack([2 * (t % (mx // 2)) + (j + k) % 2, j, k], 1)
    x = g.to(F64) * s
    start = torch.tensor([lo if c["fx"] > 0.25 else 0.5 * (ext[0] - mx * s), lo if c["fy"] > 0.25 else 0.5 * (ext[1] - my * s),
                          lo], device=DEV, dtype=F64)
    x = x + start + _uniform(gen, (n, 3), -jitter, jitter)
    v0 = {"rough": 0.05, "dense": 0.005, "wet": 0.005, "loose": 0.01}.get(kind, 0.0)
    v = _uniform(gen, (n, 3), -v0, v0) if v0 else torch.zeros_like(x)
    return x, torch.full((n,), r0, device=DEV, dtype=F64), v


def _axes(c, comp):
    n = [c["nx"], c["ny"], c["nz"]]
    return [(torch.arange(n[a] + (a == comp), device=DEV, dtype=F64) + (0.0 if a == comp else 0.5)) * c["h"]
            for a in range(3)]


def _fluid(c, seed, amp=None):
    """Face velocities (float32 [z, y, x]), the wall-normal ones zero on the walls."""
    gen = _gen(seed, 1)
    n = [c["nx"], c["ny"], c["nz"]]
    amp = c["amp"] if amp is None else amp
    kind = c.get("fluid", "noise")
    if kind == "modes":  # a sum of random divergence-free modes, RMS speed amp / 2
        modes = 8 if c["nx"] < 300 else 32
        ext = torch.tensor([m * c["h"] for m in n], dtype=F64)
        cpu = torch.Generator().manual_seed(int(seed) & 0x7FFFFFFF)
        kv = torch.randint(1, 5, (modes, 3), generator=cpu) * (2 * torch.randint(0, 2, (modes, 3), generator=cpu) - 1)
        kv = 2 * math.pi * kv / ext
        ph = torch.rand(modes, generator=cpu, dtype=F64) * 2 * math.pi
        av = torch.randn(modes, 3, generator=cpu, dtype=F64)
        kh = kv / kv.norm(dim=1, keepdim=True)
        av = av - (av * kh).sum(1, keepdim=True) * kh
        av = av / av.norm(dim=1, keepdim=True) * (0.5 * amp / math.sqrt(modes / 2))
    out = []
    for comp in range(3):
        ax = _axes(c, comp)
        shape = (len(ax[2]), len(ax[1]), len(ax[0]))
        if kind == "modes":
            f = torch.zeros(shape, device=DEV, dtype=torch.float32)
            for m in range(modes):
                px, py, pz = (torch.remainder(float(kv[m, a]) * ax[a], 2 * math.pi).float() for a in range(3))
                f += float(av[m, comp]) * torch.sin(px + float(ph[m]) + py[:, None] + pz[:, None, None])
        elif kind == "shear":
            f = torch.zeros(shape, device=DEV, dtype=torch.float32)
            if comp == 0:
                f += (amp * ax[2]).float()[:, None, None]
        else:
            f = _uniform(gen, shape, -amp, amp, torch.float32)
        side = f.select(2 - comp, 0), f.select(2 - comp, n[comp])
        for s in side:
            s.zero_()
        out.append(f.contiguous())
    return out


def _problem(c, seed):
    """What a simulation starts from: grid, parameters, the canonical encoding
    of the granules and the fluid fields."""
    x, r, v = _packing(c, seed)
    r = r.float()
    n = x.shape[0]
    rmax = float(r.max())
    k = max(1, int(math.floor(c["h"] / (2 * rmax) * (1 - 1e-12))))
    grid = SimpleNamespace(nx=c["nx"], ny=c["ny"], nz=c["nz"], dx=c["h"], origin=(0.0, 0.0, 0.0), k_contact=k)
    params = SimpleNamespace(rho_s=2650.0, rho_f=1000.0, k_n=c["k_n"], zeta=0.3, kt_over_cn=1.0, mu_fric=0.5,
                             c_drag=0.22, g=(0.0, 0.0, -9.8), dt_sub=c["dt"], dt_fluid=c["K"] * c["dt"],
                             virtual_mass=1, walls=1, sigma=c["sigma"], bridge_frac=1e-4, moisture=0.0,
                             moisture_peak=0.3)
    nc = torch.tensor([c["nx"] * k, c["ny"] * k, c["nz"] * k], device=DEV)
    s = x / (c["h"] / k)
    cell = torch.minimum(s.floor().long().clamp(min=0), nc - 1)
    q = torch.round((s - cell) * FRAC).long().clamp(1024, FRAC - 1024)
    u, vf, wf = _fluid(c, seed)
    zc = _axes(c, 3)
    p = (params.rho_f * 9.8 * (c["nz"] * c["h"] - zc[2])).float()[:, None, None].expand(c["nz"], c["ny"], c["nx"])
    lo, hi = x.amin(0) - rmax, x.amax(0) + rmax
    ins = [(zc[a] >= lo[a]) & (zc[a] <= hi[a]) for a in range(3)]
    inside = ins[2][:, None, None] & ins[1][None, :, None] & ins[0][None, None, :]
    if c["packing"] == "wet":  # moisture on both sides of the capillary factor's peak
        t = ((zc[2] - lo[2]) / (hi[2] - lo[2])).clamp(0, 1)
        within = (0.15 + 0.3 * t)[:, None, None].expand(inside.shape)
    else:
        phi = {"loose": 0.3, "cubic": 0.39, "bed": 0.6}.get(c["packing"], 0.55)
        within = torch.full_like(inside, 1.0 - phi, dtype=F64)
    af = torch.where(inside, within, torch.ones_like(within)).float()
    flat = lambda t: t.contiguous().reshape(-1)
    return SimpleNamespace(n=n, grid=grid, params=params, K=c["K"], cell=cell.int(), q=q.int(), r=r, v=v.float(),
                           u=flat(u), vf=flat(vf), wf=flat(wf), p=flat(p), alpha_f=flat(af))


def _target(p, seed):
    """The target cloud of the differentiable window: the initial positions
    plus normal noise of half a radius."""
    x0 = _absolute(p)
    return x0 + 0.5 * p.r.double()[:, None] * torch.randn(x0.shape, generator=_gen(seed, 2), device=DEV, dtype=F64)


def _projection_inputs(c, seed):
    """A sediment-like alpha_s (a bed with bumps, beyond the densest packing in
    places), alpha_f* off by up to the ratio limits, random face velocities."""
    gen = _gen(seed, 3)
    ax = [(torch.arange(m, device=DEV, dtype=F64) + 0.5) / m for m in (c["nx"], c["ny"], c["nz"])]
    Z, Y, X = ax[2][:, None, None], ax[1][None, :, None], ax[0][None, None, :]
    bed = (1.5 - 4.5 * Z).clamp(0, 1) + 0 * X + 0 * Y
    for b in _uniform(gen, (4, 4), 0.1, 0.9).tolist():
        s = 0.1 + 0.2 * b[3]
        bed = bed + 0.6 * torch.exp(-((X - b[0]) ** 2 + (Y - b[1]) ** 2 + (Z - b[2]) ** 2) / (2 * s * s))
    a_s = (0.85 * bed / bed.max() + _uniform(gen, bed.shape, -0.03, 0.03)).clamp(0, 0.85)
    a_star = (1.0 - a_s) * _uniform(gen, bed.shape, 0.3, 1.8)
    n = (c["nx"], c["ny"], c["nz"])
    vel = []
    for comp in range(3):
        shape = [n[2] + (comp == 2), n[1] + (comp == 1), n[0] + (comp == 0)]
        f = _uniform(gen, shape, -0.5, 0.5, torch.float32)
        for side in range(2):
            if not c["open"] >> (2 * comp + side) & 1:
                f.select(2 - comp, side * n[comp]).zero_()
        vel.append(f.contiguous())
    return a_s.contiguous(), a_star.float().contiguous(), vel


# ------------------------------------------------------------------ prepare and run

def prepare(case, seed):
    c = case
    s = SimpleNamespace(case=c, kind=c["kind"])
    if c["kind"] == "project":
        s.a_s, s.a_star, s.vel = _projection_inputs(c, seed)
        s.grid = gic.GicGrid(c["nx"], c["ny"], c["nz"], 1, c["h"], (0.0, 0.0, 0.0))
        s.params = gic.make_proj_params(c["dt"], 1000.0, [c["open"] >> k & 1 for k in range(6)], tol=c["tol"])
        s.ws = torch.empty(gic.gic_project_workspace_size(s.grid), dtype=torch.uint8, device=DEV)
        s.p = [torch.empty_like(s.a_s) for _ in range(2)]
        s.out = [torch.empty_like(f) for f in s.vel]
        s.disp = [torch.empty_like(f) for f in s.vel]
        return s
    p = _problem(c, seed)
    prec = gic.GIC_FP32 if c["bits"] == 32 else gic.GIC_FP64
    if c["kind"] == "host":
        pin = lambda t: t.cpu().pin_memory()
        s.precision = prec
        s.inputs = [pin(t) for t in (p.cell, p.q, p.r, p.v, p.u, p.vf, p.wf, p.p, p.alpha_f)]
        s.grid, s.params = gic.make_grid(p.grid), gic.make_params(p.params)
        host = lambda shape, dt: torch.empty(shape, dtype=dt, pin_memory=True)
        s.x, s.v = host((p.n, 3), F64), host((p.n, 3), F64)
        s.alpha = host(p.p.numel(), F64)
        s.Fs = [host(f.numel(), torch.float32) for f in (p.u, p.vf, p.wf)]
        s.sums = host(2, F64)
        s.ws = torch.empty(gic.gic_window_host_workspace_size(s.grid, p.n, prec), dtype=torch.uint8, device=DEV)
        return s
    s.sim = Simulator.from_problem(p, prec, DEV, verlet=c["kind"] != "parts")
    s.init = s.sim.A.clone()
    if c["kind"] == "grad":
        real = s.sim.real
        s.v0 = p.v.to(real)
        s.c_drag = torch.tensor(p.params.c_drag, dtype=real, device=DEV)
        s.mu = torch.tensor(p.params.mu_fric, dtype=real, device=DEV)
        s.target = _target(p, seed)
    return s


def run(state):
    s = state
    if s.kind == "project":
        gic.gic_project(s.grid, s.params, s.a_s, s.a_star, *s.vel, s.p[0], s.p[1], s.out, s.disp, s.ws)
        return {"p": s.p, "v": s.out, "dx": s.disp}
    if s.kind == "host":
        gic.gic_window_forward_host(s.grid, s.params, s.precision, *s.inputs, s.case["K"], s.x, s.v, s.alpha, s.Fs,
                                    s.sums, s.ws)
        return {"x": s.x, "v": s.v.float(), "alpha_s": s.alpha, "Fs": s.Fs, "sums": s.sums}
    sim = s.sim
    if s.kind == "grad":
        v0, c, mu = (t.detach().requires_grad_() for t in (s.v0, s.c_drag, s.mu))
        x = GicWindow.apply(v0, c, mu, sim, s.init, s.case["K"], 10)
        loss = ((x - s.target) ** 2).sum(dim=1).mean()
        loss.backward()
        return {"x": x.detach(), "g_v0": v0.grad, "g_c_drag": c.grad, "g_mu": mu.grad}
    # a fluid step from the saved state; FP32 states keep their velocities as float
    sim.load_state(s.init)
    sim.run(s.case["K"])
    x, v = sim.positions()
    return {"x": x, "v": v.to(sim.real), "alpha_s": sim.alpha_s, "Fs": list(sim.Fs), "sums": sim.sums}


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    c = case
    if c["kind"] == "project":  # alpha_s, alpha_f*, v* in; two pressures, v' and dx out; two solves
        n = c["nx"] * c["ny"] * c["nz"]
        return {"bytes": 64.0 * n, "flops": 4000.0 * n}
    cells = c["nx"] * c["ny"] * c["nz"]
    w = 1 if c["bits"] == 32 else 2
    n, K = c["n"], c["K"]
    # a substep: the state in and out and the share of fluid samples and F_s deposits; the fields once, F_s and alpha_s out
    fields = cells * (32.0 * w + 8)
    b = {"window": 90.0, "host": 90.0, "grad": 280.0, "parts": 353.0}[c["kind"]] * w * K * n + fields
    if c["kind"] == "host":
        b += 88.0 * n
    flops = {"window": 400.0, "host": 400.0, "grad": 1600.0, "parts": 600.0}[c["kind"]] * K * n
    return {"bytes": b, "flops": flops}


# ------------------------------------------------------------------ the method in 64 bits

def _absolute(p):
    return (p.cell.double() + p.q.double() / FRAC) * (p.grid.dx / p.grid.k_contact)


class _Exact:
    """Alg. 2 in FP64 torch operations on absolute positions, differentiable."""

    def __init__(self, c, p):
        self.c, self.p = c, p
        self.h, self.n3 = c["h"], [c["nx"], c["ny"], c["nz"]]
        self.r = p.r.double()
        P = p.params
        self.V = 4.0 / 3.0 * math.pi * self.r ** 3
        self.m, self.ma = P.rho_s * self.V, 0.5 * P.rho_f * self.V
        self.c_drag = torch.tensor(P.c_drag, dtype=F64, device=DEV)
        self.mu = torch.tensor(P.mu_fric, dtype=F64, device=DEV)
        self.g = torch.tensor(P.g, dtype=F64, device=DEV)
        shape = lambda a: [self.n3[2] + (a == 2), self.n3[1] + (a == 1), self.n3[0] + (a == 0)]
        self.vel = [f.double() for f in (p.u, p.vf, p.wf)]
        pr = p.p.double().reshape(shape(3))
        self.gp = []
        for a in range(3):
            ax = 2 - a
            d = torch.diff(pr, dim=ax) / self.h
            self.gp.append(torch.cat([d.narrow(ax, 0, 1), d, d.narrow(ax, d.shape[ax] - 1, 1)], ax).reshape(-1))
        self.af = p.alpha_f.double()
        self.Fs = [torch.zeros_like(f) for f in self.vel]
        self.pairs_at = None
        self.skin = 0.1 * float(self.r.max())

    def stencil(self, x, comp):
        """The eight sample indices and weights of grid `comp` (3: centres)."""
        i0, w = [], []
        for a in range(3):
            ns = self.n3[a] + (a == comp)
            s = x[:, a] / self.h - (0.0 if a == comp else 0.5)
            i = s.detach().floor()
            t = s - i
            i = i.long()
            t = torch.where(i < 0, torch.zeros_like(t), torch.where(i > ns - 2, torch.ones_like(t), t))
            i0.append(i.clamp(0, ns - 2))
            w.append(t)
        sx, sy = self.n3[0] + (comp == 0), self.n3[1] + (comp == 1)
        base = i0[0] + sx * (i0[1] + sy * i0[2])
        for k in range(8):
            a, b, d = k & 1, k >> 1 & 1, k >> 2
            yield base + a + sx * (b + sy * d), ((w[0] if a else 1 - w[0]) * (w[1] if b else 1 - w[1]) *
                                                 (w[2] if d else 1 - w[2]))

    def gather(self, x, comp, fields):
        out = [0.0] * len(fields)
        for i, w in self.stencil(x, comp):
            out = [o + w * f[i] for o, f in zip(out, fields)]
        return out

    def reach(self):
        r = float(self.r.max())
        return 2 * r * (1.1 if self.c["sigma"] > 0 else 1.0)

    def find_pairs(self, x):
        if self.pairs_at is not None and float((x - self.pairs_at).norm(dim=1).max()) < self.skin / 2:
            return
        self.pairs_at = x.clone()
        R = self.reach() + self.skin
        lo = x.amin(0)
        cell = ((x - lo) / R).floor().long() + 1
        M = cell.amax(0) + 2
        key = cell[:, 0] + M[0] * (cell[:, 1] + M[1] * cell[:, 2])
        key, order = torch.sort(key)
        xs, rs = x[order], self.r[order]
        uniq, count = torch.unique_consecutive(key, return_counts=True)
        start = torch.cumsum(count, 0) - count
        most = int(count.max())
        at = torch.arange(x.shape[0], device=DEV)
        I, J = [], []
        extra = self.skin + (0.2 * float(self.r.max()) if self.c["sigma"] > 0 else 0.0)
        for o in range(27):
            d = (o % 3 - 1) + M[0] * ((o // 3 % 3 - 1) + M[1] * (o // 9 - 1))
            if o < 13:
                continue
            u = torch.searchsorted(uniq, key + d).clamp(max=uniq.numel() - 1)
            hit = uniq[u] == key + d
            first = start[u]
            num = torch.where(hit, count[u], torch.zeros_like(first))
            for k in range(most):
                i = at[num > k]
                j = first[i] + k
                if o == 13:
                    keep = j > i
                    i, j = i[keep], j[keep]
                near = ((xs[i] - xs[j]) ** 2).sum(1) < (rs[i] + rs[j] + extra) ** 2
                I.append(order[i[near]])
                J.append(order[j[near]])
        self.I, self.J = torch.cat(I), torch.cat(J)

    def law(self, d, n, overlap, dv, meff):
        """Spring and dashpot along n, Coulomb-capped tangential dashpot."""
        P = self.p.params
        cn = 2 * P.zeta * torch.sqrt(P.k_n * meff)
        vn = (dv * n).sum(1)
        Fn = P.k_n * overlap - cn * vn
        t = dv - vn[:, None] * n
        t2 = (t * t).sum(1)
        some = t2 > 0
        vt = torch.where(some, torch.sqrt(torch.where(some, t2, torch.ones_like(t2))), torch.zeros_like(t2))
        kt = P.kt_over_cn * cn
        cap = self.mu * Fn.abs()
        slip = kt * vt > cap
        a = torch.where(slip, cap / torch.where(slip, vt, torch.ones_like(vt)), kt)
        return Fn[:, None] * n - a[:, None] * t

    def contact(self, x, v):
        P = self.p.params
        F = torch.zeros_like(x)
        with torch.no_grad():
            self.find_pairs(x.detach())
            d2 = ((x[self.I] - x[self.J]) ** 2).sum(1)
            R = self.r[self.I] + self.r[self.J]
            touch = d2 < R * R
            reach = d2 < (1.1 * R) ** 2
        i, j = self.I[touch], self.J[touch]
        rel = x[i] - x[j]
        d = rel.norm(dim=1)
        f = self.law(d, rel / d[:, None], self.r[i] + self.r[j] - d, v[i] - v[j], self.m[i] * self.m[j] / (self.m[i] + self.m[j]))
        F = F.index_add(0, i, f).index_add(0, j, -f)
        if P.sigma > 0:
            b = reach & ~touch
            i, j = self.I[b], self.J[b]
            rel = x[i] - x[j]
            d = rel.norm(dim=1)
            s = d - self.r[i] - self.r[j]
            R = 2 * self.r[i] * self.r[j] / (self.r[i] + self.r[j])
            Vs = P.bridge_frac * (self.V[i] + self.V[j]) / 2
            vr = (Vs / R ** 3) ** (1 / 3)
            af, = self.gather(x, 3, [self.af])
            dry = af < 1
            sr = P.moisture + torch.where(dry, af / torch.where(dry, 1 - af, torch.ones_like(af)), torch.full_like(af, 1e30))
            sm = (sr[i] + sr[j]) / 2
            inside = (sm > 0) & (sm < 1) & (s < R * (vr + 0.1 * vr * vr)) & (s > 0)
            sm = torch.where(inside, sm, torch.full_like(sm, 0.5))
            s = torch.where(inside, s, R)
            cp = 2 * P.moisture_peak - 0.5
            t = sm / (cp + torch.sqrt(cp * cp + (1 - 2 * cp) * sm))
            y = 2 * Vs / (math.pi * R * s * s)
            st = 2 * math.pi * P.sigma * R * (y / (torch.sqrt(1 + y) * (torch.sqrt(1 + y) + 1)))
            f = torch.where(inside, -4 * t * (1 - t) * st / d, torch.zeros_like(d))[:, None] * rel
            F = F.index_add(0, i, f).index_add(0, j, -f)
        for a in range(3):
            for side in range(2):
                gap = x[:, a] if side == 0 else self.n3[a] * self.h - x[:, a]
                k = torch.nonzero(gap.detach() < self.r).reshape(-1)
                if k.numel():
                    n = torch.zeros((k.numel(), 3), dtype=F64, device=DEV)
                    n[:, a] = 1.0 if side == 0 else -1.0
                    F = F.index_add(0, k, self.law(None, n, self.r[k] - gap[k], v[k], self.m[k]))
        return F

    def substep(self, x, v, transfer=True):
        P = self.p.params
        Fc = self.contact(x, v)
        both = [self.gather(x, a, [self.vel[a], self.gp[a]]) for a in range(3)]
        uf, gp = (torch.stack([b[k] for b in both], 1) for k in range(2))
        dv = uf - v
        s2 = (dv * dv).sum(1, keepdim=True)
        sp = torch.where(s2 > 0, torch.sqrt(torch.where(s2 > 0, s2, torch.ones_like(s2))), torch.zeros_like(s2))
        Ff = self.c_drag * math.pi * (self.r ** 2)[:, None] * P.rho_f * sp * dv - self.V[:, None] * gp
        af = self.g - gp / P.rho_f
        m, ma = self.m[:, None], self.ma[:, None]
        acc = (Fc + Ff + m * self.g + ma * af) / (m + ma)
        v2 = v + P.dt_sub * acc
        x2 = x + P.dt_sub * v2
        if transfer:
            fe = -(P.dt_sub / P.dt_fluid) * (Ff + ma * (af - acc))
            for a in range(3):
                for i, w in self.stencil(x, a):
                    self.Fs[a].index_add_(0, i, w * fe[:, a])
        return x2, v2

    def volume(self, x):
        out = torch.zeros(self.n3[0] * self.n3[1] * self.n3[2], dtype=F64, device=DEV)
        for i, w in self.stencil(x, 3):
            out.index_add_(0, i, w * self.V / self.h ** 3)
        return out


def _exact_projection(c, seed):
    a_s, a_star, vel = _projection_inputs(c, seed)
    h, dt, rho = c["h"], c["dt"], 1000.0
    ap = 1.0 - a_s.clamp(max=0.740)
    opened = [c["open"] >> k & 1 for k in range(6)]
    vel = [f.double() for f in vel]
    beta = []
    for a in range(3):
        ax = 2 - a
        m = ap.shape[ax]
        first, final = ap.narrow(ax, 0, 1), ap.narrow(ax, m - 1, 1)
        mid = 0.5 * (ap.narrow(ax, 1, m - 1) + ap.narrow(ax, 0, m - 1))
        beta.append(torch.cat([first * opened[2 * a], mid, final * opened[2 * a + 1]], ax))

    def grad(p):  # face differences, p = 0 beyond every side
        out = []
        for a in range(3):
            z = torch.zeros_like(p.narrow(2 - a, 0, 1))
            out.append(torch.diff(torch.cat([z, p, z], 2 - a), dim=2 - a))
        return out

    def div(f):
        return sum(torch.diff(f[a], dim=2 - a) for a in range(3))

    def apply(p):
        return -div([b * g for b, g in zip(beta, grad(p))])

    diag = sum(b.narrow(2 - a, 0, ap.shape[2 - a]) + b.narrow(2 - a, 1, ap.shape[2 - a]) for a, b in enumerate(beta))

    def solve(b):
        p, r = torch.zeros_like(b), b.clone()
        z = r / diag
        d, rz, b2 = z.clone(), (r * z).sum(), (b * b).sum()
        for it in range(6000):
            y = apply(d)
            al = rz / (d * y).sum()
            p += al * d
            r = r - al * y if it % 50 != 49 else b - apply(p)
            if it % 25 == 24 and float((r * r).sum()) <= 1e-27 * float(b2):
                break
            z = r / diag
            rz2 = (r * z).sum()
            d = z + rz2 / rz * d
            rz = rz2
        return p

    p1 = solve(-(rho * h / dt) * div([b * f for b, f in zip(beta, vel)]))
    p2 = solve(-(rho * h * h / dt ** 2) * ap * (1 - (a_star.double() / ap).clamp(0.5, 1.5)))
    out, disp = [], []
    for a, (g1, g2) in enumerate(zip(grad(p1), grad(p2))):
        f, d = vel[a] - dt / rho * g1 / h, (-(dt ** 2) / rho * g2 / h).clamp(-h, h)
        for side in range(2):
            if not opened[2 * a + side]:
                for t in (f, d):
                    t.select(2 - a, side * (f.shape[2 - a] - 1)).zero_()
        out.append(f)
        disp.append(d)
    return {"p": [p1, p2], "v": out, "dx": disp}


def exact(case, seed):
    c = case
    if c["kind"] == "project":
        return _exact_projection(c, seed)
    if c["n"] * c["K"] > 330_000_000:
        return None
    p = _problem(c, seed)
    E = _Exact(c, p)
    x, v = _absolute(p), p.v.double()
    if c["kind"] == "grad":
        if c["bits"] == 32:  # the parameters as the program holds them
            E.c_drag, E.mu = E.c_drag.float().double(), E.mu.float().double()
        leaves = v0, cd, mu = [t.requires_grad_() for t in (v, E.c_drag, E.mu)]
        E.c_drag, E.mu, v = cd, mu, v0
        for _ in range(c["K"]):
            x, v = E.substep(x, v, transfer=False)
        loss = ((x - _target(p, seed)) ** 2).sum(dim=1).mean()
        g = torch.autograd.grad(loss, leaves, allow_unused=True)
        g = [torch.zeros_like(t) if q is None else q for q, t in zip(g, leaves)]
        return {"x": x.detach(), "g_v0": g[0], "g_c_drag": g[1], "g_mu": g[2]}
    with torch.no_grad():
        for _ in range(c["K"]):
            x, v = E.substep(x, v)
        alpha = E.volume(x)
        total = E.V.sum()
        return {"x": x, "v": v, "alpha_s": alpha, "Fs": E.Fs, "sums": torch.stack([total, total])}
