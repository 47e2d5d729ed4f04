"""What a user of the framework has it do, as cases that can be timed and
checked: calls of the package's public entry points over the sizes, options
and precisions of the method's workloads.

A case names its kind and sizes.  ``prepare`` makes the inputs on the GPU and
the objects a user's program keeps (lattice, batch, solver), ``run`` is one
pass, ``work`` counts the bytes and floating-point operations a pass cannot do
without, and ``exact`` computes the same outputs in FP64 with plain torch and
numpy.  Fields that the FP32 lattice carries are read out in FP32.
"""
import math

import numpy as np
import torch

from paper_1601_02708_gb300 import (FEM, LBM, Bimolecular, Hybrid, LBMBatch, inputs,
                                    outlet_breakthrough, species_from_invariants)

# D2Q9: rest, E, N, W, S, NE, NW, SW, SE
E = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
W = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]
CHANNEL = (1, 2, 0, 0)  # Dirichlet west, Neumann east, periodic in y
BLOCK = (1, 1, 1, 1)    # four Dirichlet sides


def listed():
    return [
        # The lattice half of one Schwarz iteration of the plain hybrid run
        # (256 x 64, no pores, 10 substeps, data on the device): rollback,
        # substeps with time-interpolated inlet data, trace at the interface.
        # The smallest call, bound by launches and latency.
        dict(name="plain_block", kind="block", nx=256, ny=64, precision=32, porosity=1.0,
             channel=True, n=10),
        # The lattice half of one Schwarz iteration of a pore block (512 x 512,
        # four Dirichlet sides, dissolving, 50 substeps).
        dict(name="pore_block", kind="block", nx=512, ny=512, precision=32, porosity=0.55,
             channel=False, n=50),
        # An ordinary stretch of a dissolving channel run at an odd, ragged
        # size, edge data from the host, fields read out at its end.
        dict(name="channel_ragged", kind="channel", nx=1531, ny=977, precision=32,
             porosity=0.6, walls="bounce", dissolve=True, n=20),
        # The same at the size of the large single-lattice run: the largest.
        dict(name="channel_large", kind="channel", nx=4096, ny=4096, precision=32,
             porosity=0.6, walls="bounce", dissolve=True, n=20),
        # FP64 populations, the mode that reproduces the dissolving mask exactly.
        dict(name="channel_fp64", kind="channel", nx=1024, ny=1024, precision=64,
             porosity=0.6, walls="bounce", dissolve=True, n=10),
        # Pore walls of the maximum-entropy kind on a fixed mask.
        dict(name="channel_walls", kind="channel", nx=1200, ny=900, precision=32,
             porosity=0.6, walls="maxent", dissolve=False, n=10),
        # Independent pore geometries of uneven size advanced together.
        dict(name="batch", kind="batch", count=24, smin=64, smax=768, precision=32, n=25),
        # Gradients of the outlet breakthrough with the whole history kept.
        dict(name="gradient", kind="gradient", nx=512, ny=512, precision=32, n=500, stride=0),
        # The same from checkpoints, on a smaller odd lattice.
        dict(name="gradient_checkpointed", kind="gradient", nx=331, ny=203, precision=32,
             n=225, stride=15),
        # The continuum half of a coarse step around a pore block: five Schwarz
        # iterations of the 400 x 100 mesh, each with new ring data.
        dict(name="continuum", kind="continuum", nex=400, ney=100, iterations=5),
        # One whole coarse step of the plain hybrid run, FP64.
        dict(name="hybrid_plain", kind="hybrid", precision=64, eta=10, iterations=3),
        # The two invariants of an instantaneous reaction A + 2 B -> C, then
        # the species.
        dict(name="bimolecular", kind="bimolecular", nx=1024, ny=768, porosity=0.6, n=20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["block", "block", "channel", "channel", "channel", "batch", "gradient",
                       "gradient", "continuum", "hybrid", "bimolecular"])
    if kind == "block":
        pores = rng.random() < 0.7
        return dict(kind=kind, nx=_log_int(rng, 64, 2048), ny=_log_int(rng, 64, 2048),
                    precision=rng.choice([32, 32, 64]),
                    porosity=round(rng.uniform(0.4, 0.8), 3) if pores else 1.0,
                    channel=not pores, n=_log_int(rng, 5, 50))
    if kind == "channel":
        walls = rng.choice(["bounce", "bounce", "bounce", "maxent", "maxent_lattice"])
        precision = 64 if rng.random() < 0.25 else 32
        hi = 1400 if precision == 64 or walls == "maxent" else 3600
        return dict(kind=kind, nx=_log_int(rng, 64, hi), ny=_log_int(rng, 64, hi),
                    precision=precision, porosity=round(rng.uniform(0.4, 0.8), 3), walls=walls,
                    dissolve=walls == "bounce" and rng.random() < 0.7, n=rng.randint(4, 20))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(3, 32), smin=64,
                    smax=rng.choice([200, 400, 800]), precision=rng.choice([32, 32, 64]),
                    n=rng.randint(5, 25))
    if kind == "gradient":
        n = _log_int(rng, 50, 500)
        return dict(kind=kind, nx=_log_int(rng, 64, 640), ny=_log_int(rng, 64, 640),
                    precision=rng.choice([32, 32, 64]), n=n,
                    stride=rng.choice([0, 0, int(math.ceil(math.sqrt(n)))]))
    if kind == "continuum":
        ney = rng.randint(20, 110)
        return dict(kind=kind, nex=4 * ney, ney=ney, iterations=rng.randint(2, 6))
    if kind == "hybrid":
        return dict(kind=kind, precision=rng.choice([32, 64]), eta=rng.randint(4, 20),
                    iterations=rng.randint(2, 5))
    return dict(kind=kind, nx=_log_int(rng, 64, 2048), ny=_log_int(rng, 64, 2048),
                porosity=round(rng.uniform(0.4, 0.8), 3), n=rng.randint(4, 20))


# ---- inputs ---------------------------------------------------------------------

def _pores(nx, ny, porosity, seed):
    """uint8 [ny, nx] mask on the GPU: random overlapping disks of radius
    U[8, 24], as many as leave ``porosity`` open on average; the first and last
    columns stay fluid."""
    solid = torch.zeros(ny * nx, dtype=torch.uint8, device="cuda")
    rng = np.random.default_rng([seed, nx, ny])
    if porosity < 1.0:
        m = max(1, round(-math.log(porosity) * nx * ny / (math.pi * (8 * 8 + 8 * 24 + 24 * 24) / 3)))
        disks = np.stack([rng.uniform(0, nx, m), rng.uniform(0, ny, m), rng.uniform(8, 24, m)])
        off = torch.arange(-25, 26, device="cuda")
        for part in torch.from_numpy(disks).cuda().split(2048, dim=1):
            cx, cy, r = (v[:, None, None] for v in part)
            x, y = cx.floor().long() + off[None, None, :], cy.floor().long() + off[None, :, None]
            inside = ((x - cx) ** 2 + (y - cy) ** 2 <= r * r) & (x >= 1) & (x <= nx - 2) & \
                (y >= 0) & (y <= ny - 1)
            solid[(y * nx + x)[inside]] = 1
    return solid.view(ny, nx)


def _flow(nx, ny, solid, seed, mean=0.0):
    """float64 [2, ny, nx]: 16 Fourier modes of a stream function, at most 0.05
    fast, plus a mean flow along x; zero in the solids."""
    rng = np.random.default_rng([seed, nx, ny, 1])
    k = rng.integers(-8, 9, (2, 16))
    k[0, (k[0] == 0) & (k[1] == 0)] = 1
    amp = rng.normal(size=16) / np.hypot(k[0], k[1])
    phase = rng.uniform(0, 2 * math.pi, 16)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()
    kx, ky, amp, phase = dev(k[0]), dev(k[1]), dev(amp), dev(phase)
    a = 2 * math.pi / nx * torch.arange(nx, device="cuda", dtype=torch.float64)[:, None] * kx
    b = 2 * math.pi / ny * torch.arange(ny, device="cuda", dtype=torch.float64)[:, None] * ky + phase
    c, s = torch.cos(a).T, torch.sin(a).T
    gy, gx = amp * ky / ny, amp * kx / nx
    vel = torch.stack([(gy * torch.cos(b)) @ c - (gy * torch.sin(b)) @ s,
                       -((gx * torch.cos(b)) @ c - (gx * torch.sin(b)) @ s)])
    vel *= 0.05 / vel.square().sum(0).max().sqrt()
    vel[0] += mean
    return vel * (solid == 0)


def _smooth(nx, ny, seed):
    """A smooth float64 [ny, nx] field in [0.1, 0.9]."""
    rng = np.random.default_rng([seed, nx, ny, 2])
    p = rng.uniform(0, 2 * math.pi, 2)
    m = rng.integers(1, 4, 2)
    x = torch.arange(nx, device="cuda", dtype=torch.float64) / nx
    y = torch.arange(ny, device="cuda", dtype=torch.float64) / ny
    return 0.5 + 0.4 * torch.sin(2 * math.pi * m[1] * y + p[1])[:, None] * \
        torch.cos(2 * math.pi * m[0] * x + p[0])


def _pore_inputs(case, nx, ny, seed, edges, dissolve, k=1e-3):
    """Arguments of one reacting lattice and its edge data (start, end).  With
    dissolution one solid node in fifty is partly used up, so that nodes
    dissolve during a pass as they do in the middle of a long run."""
    porosity = case.get("porosity", 0.6)
    solid = _pores(nx, ny, porosity, seed)
    args = dict(edges=edges, vel=_flow(nx, ny, solid, seed), u0=_smooth(nx, ny, seed) * (solid == 0))
    if porosity < 1.0:
        args.update(solid=solid, react_mode=1, k=k)
    if dissolve:
        gen = torch.Generator(device="cuda").manual_seed(seed)
        u = torch.rand(2, ny, nx, device="cuda", dtype=torch.float64, generator=gen)
        args.update(dissolution=True, mineral=torch.where(u[0] < 0.02, 1e-4 + u[1], 1.0))
    t = torch.arange(2 * (nx + ny), device="cuda", dtype=torch.float64)
    a = 0.8 + 0.2 * torch.sin(0.02 * t + 0.1 * (seed % 60))
    return args, a, a + 0.05 * torch.cos(0.03 * t)


def _trace_points(nx, ny):
    """Interface points a third of the way in, off the nodes."""
    t = torch.linspace(0.3, ny - 1.7, 2 * ny // 3, device="cuda", dtype=torch.float64)
    return torch.stack([torch.full_like(t, nx / 3 + 0.21), t], 1)


def _batch_sizes(case, seed):
    """Sides at the quantiles of a log-uniform law on [smin, smax], in mixed
    order; porosity and tau drawn per member."""
    n = case["count"]
    q = (np.arange(n) + 0.5) / n
    side = np.rint(case["smin"] * (case["smax"] / case["smin"]) ** q).astype(int)
    np.random.default_rng(n).shuffle(side)
    rng = np.random.default_rng([seed, n])
    return [dict(side=int(s), porosity=float(p), tau=float(t), seed=1000 * (seed % 100000) + i)
            for i, (s, p, t) in enumerate(zip(side, rng.uniform(0.4, 0.8, n), rng.uniform(0.6, 1.2, n)))]


def _gradient_inputs(case, seed):
    nx, ny = case["nx"], case["ny"]
    solid = _pores(nx, ny, 0.6, seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    real = torch.float64 if case["precision"] == 64 else torch.float32
    kf = (1e-3 * (0.8 + 0.4 * torch.rand(ny, nx, device="cuda", dtype=torch.float64, generator=gen))).to(real)
    args = dict(edges=CHANNEL, solid=solid, vel=_flow(nx, ny, solid, seed, mean=0.15),
                u0=_smooth(nx, ny, seed) * (solid == 0), react_mode=2, k_field=kf)
    return args, kf, torch.tensor(1.0 + 0.01 * (seed % 7), dtype=real, device="cuda")


def _continuum_inputs(case, seed):
    """Mesh of [0, 4] x [0, 1] with a hole, its Dirichlet nodes (inlet, then
    the hole's ring), the state and one vector of Dirichlet data an iteration,
    converging as the Schwarz iterates do."""
    nex, ney = case["nex"], case["ney"]
    h = 1.0 / ney
    i0, i1, j0, j1 = (round(v * ney) for v in (1.7, 2.3, 0.2, 0.8))
    act = np.ones((ney, nex), np.uint8)
    act[j0:j1, i0:i1] = 0
    nxn = nex + 1
    ring = [j * nxn + i for j in range(j0, j1 + 1) for i in range(i0, i1 + 1)
            if i in (i0, i1) or j in (j0, j1)]
    inlet = [j * nxn for j in range(ney + 1)]
    rng = np.random.default_rng([seed, nex, ney])
    p = rng.uniform(0, 2 * math.pi, 3)
    x, y = np.meshgrid(np.arange(nxn) * h, np.arange(ney + 1) * h)
    d0 = (0.7 + 0.2 * np.sin(3 * x + p[0]) * np.cos(2 * y + p[1])).reshape(-1)
    dirichlet = np.array(inlet + ring)
    t = np.arange(len(dirichlet))
    data = [d0[dirichlet] - 0.02 * np.sin(0.05 * t + p[2]) * (1 + 0.3 ** (i + 1))
            for i in range(case["iterations"])]
    # the block's lattice spacing and diffusivity with 32 lattice nodes an
    # element, 50 substeps a coarse step
    hl = h / 32
    mesh = dict(nex=nex, ney=ney, x0=0.0, y0=0.0, hx=h, hy=h, D=0.2 / 3 * hl * hl, v=(0.0, 0.0),
                theta=0.5, dt=50.0, supg=False, elem_active=act, dirichlet=dirichlet, d0=d0)
    s = np.linspace(0, 1, 8 * ney)
    edge = np.stack([np.full_like(s, (i0 - 2) * h), ((j0 - 2) + (j1 - j0 + 4) * s) * h], 1)
    return mesh, d0, data, edge


def _hybrid_layout(case, seed):
    """The plain hybrid's layout with the pulse's place and width from the seed."""
    lay = inputs.hybrid_plain_layout(1)
    rng = np.random.default_rng([seed, 3])
    at, wide = rng.uniform(0.45, 0.6), rng.uniform(0.002, 0.006)
    L, F = lay["lbm"], lay["fem"]
    xs = 0.5 + np.arange(L["nx"]) * lay["h"]
    L["u0"] = np.tile(np.exp(-(xs - at) ** 2 / wide), (L["ny"], 1))
    xn = (np.arange((F["nex"] + 1) * (F["ney"] + 1)) % (F["nex"] + 1)) * F["hx"]
    F["d0"] = np.exp(-(xn - at) ** 2 / wide)
    F["dt"] = float(case["eta"])
    lay["eta"], lay["max_iter"] = case["eta"], case["iterations"]
    return lay


def _bimolecular_inputs(case, seed):
    nx, ny = case["nx"], case["ny"]
    solid = _pores(nx, ny, case["porosity"], seed)
    fluid = solid == 0
    a, b = _smooth(nx, ny, seed) * fluid, (1.0 - _smooth(nx, ny, seed)) * fluid
    return dict(edges=CHANNEL, solid=solid, vel=_flow(nx, ny, solid, seed)), a, b


# ---- prepare and run --------------------------------------------------------------

def _real(precision):
    return torch.float64 if precision == 64 else torch.float32


def prepare(case, seed):
    return _KINDS[case["kind"]][0](case, seed)


def run(state):
    return _KINDS[state["kind"]][1](state)


def work(case):
    return _KINDS[case["kind"]][2](case)


def exact(case, seed):
    return _KINDS[case["kind"]][3](case, seed)


def _block_args(case, seed):
    edges = CHANNEL if case["channel"] else BLOCK
    return _pore_inputs(case, case["nx"], case["ny"], seed, edges, case["porosity"] < 1.0, k=5e-4)


def _block_prepare(case, seed):
    nx, ny, real = case["nx"], case["ny"], _real(case["precision"])
    args, ua, ub = _block_args(case, seed)
    lat = LBM(nx, ny, 0.8 if case["channel"] else 0.7, precision=case["precision"], **args)
    pts = _trace_points(nx, ny)
    return dict(kind="block", lat=lat, n=case["n"], ua=ua, ub=ub, start=lat.save(), pts=pts,
                precision=case["precision"], dissolves="dissolution" in args,
                trace=torch.empty(len(pts), dtype=torch.float64, device="cuda"),
                u=torch.empty(ny, nx, dtype=real, device="cuda"),
                solid=torch.empty(ny, nx, dtype=torch.uint8, device="cuda"))


def _block_run(s):
    lat = s["lat"]
    lat.restore(s["start"])
    lat.substeps(s["n"], s["n"], s["ua"], s["ub"])
    lat.trace(s["pts"], out=s["trace"])
    out = dict(u=lat.concentration(out=s["u"], precision=s["precision"]),
               trace=s["trace"] if s["precision"] == 64 else s["trace"].float())
    if s["dissolves"]:
        out["solid"] = lat.solid(out=s["solid"])
    return out


def _lattice_work(nodes, fluid, size, n, fields=1, surface=0.0):
    """Populations in and out, velocity, mask and concentration once; 105
    operations a fluid node and substep (moments 8, collision 97)."""
    b = fluid * nodes * (fields * 18 + 2) * size + nodes * (1 + fields * size)
    return dict(bytes=b + 24.0 * surface * nodes, flops=105.0 * fields * fluid * nodes * n)


def _block_work(case):
    nodes = case["nx"] * case["ny"]
    return _lattice_work(nodes, case["porosity"], case["precision"] // 8, case["n"],
                         surface=0.0 if case["channel"] else 0.045)


def _block_exact(case, seed):
    nx, ny = case["nx"], case["ny"]
    args, ua, ub = _block_args(case, seed)
    ref = _Lattice(nx, ny, 0.8 if case["channel"] else 0.7, **args)
    ref.substeps(case["n"], case["n"], ua, ub)
    out = dict(u=ref.u, trace=ref.trace(_trace_points(nx, ny)))
    if "dissolution" in args:
        out["solid"] = None
    return out


def _channel_args(case, seed):
    return _pore_inputs(case, case["nx"], case["ny"], seed, CHANNEL, case["dissolve"])


def _channel_prepare(case, seed):
    nx, ny = case["nx"], case["ny"]
    args, ua, ub = _channel_args(case, seed)
    lat = LBM(nx, ny, 0.7, precision=case["precision"], walls=case["walls"], **args)
    return dict(kind="channel", lat=lat, n=case["n"], ua=ua.cpu().numpy(), ub=ub.cpu().numpy(),
                q=np.zeros(2 * (nx + ny)), precision=case["precision"], dissolves=case["dissolve"],
                u=torch.empty(ny, nx, dtype=_real(case["precision"]), device="cuda"),
                solid=torch.empty(ny, nx, dtype=torch.uint8, device="cuda"),
                mineral=torch.empty(ny, nx, dtype=torch.float64, device="cuda"))


def _channel_run(s):
    lat = s["lat"]
    lat.substeps(s["n"], s["n"], s["ua"], s["ub"], s["q"])
    out = dict(u=lat.concentration(out=s["u"], precision=s["precision"]))
    if s["dissolves"]:
        out.update(solid=lat.solid(out=s["solid"]), mineral=lat.mineral(out=s["mineral"]))
    return out


def _channel_work(case):
    nodes = case["nx"] * case["ny"]
    w = _lattice_work(nodes, case["porosity"], case["precision"] // 8, case["n"],
                      surface=0.045 if case["dissolve"] else 0.0)
    if case["dissolve"]:
        w["bytes"] += 9.0 * nodes  # mask and mineral read out
    return w


def _channel_exact(case, seed):
    args, ua, ub = _channel_args(case, seed)
    ref = _Lattice(case["nx"], case["ny"], 0.7, walls=case["walls"] != "bounce", **args)
    ref.substeps(case["n"], case["n"], ua, ub)
    out = dict(u=ref.u)
    if case["dissolve"]:
        out.update(solid=None, mineral=ref.mineral)
    return out


def _batch_prepare(case, seed):
    stream = torch.cuda.Stream()
    members, ua, ub, u = [], [], [], []
    for m in _batch_sizes(case, seed):
        args, a, b = _pore_inputs(m, m["side"], m["side"], m["seed"], CHANNEL, True)
        torch.cuda.synchronize()
        members.append(LBM(m["side"], m["side"], m["tau"], precision=case["precision"],
                           stream=stream.cuda_stream, **args))
        ua.append(a)
        ub.append(b)
        u.append(torch.empty(m["side"], m["side"], dtype=_real(case["precision"]), device="cuda"))
    return dict(kind="batch", batch=LBMBatch(members), stream=stream, n=case["n"], ua=ua, ub=ub,
                u=u, precision=case["precision"])


def _batch_run(s):
    s["batch"].substeps(s["n"], s["n"], s["ua"], s["ub"])
    return [m.concentration(out=u, precision=s["precision"])
            for m, u in zip(s["batch"].members, s["u"])]


def _batch_work(case):
    q = (np.arange(case["count"]) + 0.5) / case["count"]
    nodes = float(((case["smin"] * (case["smax"] / case["smin"]) ** q) ** 2).sum())
    return _lattice_work(nodes, 0.6, case["precision"] // 8, case["n"], surface=0.045)


def _batch_exact(case, seed):
    out = []
    for m in _batch_sizes(case, seed):
        args, a, b = _pore_inputs(m, m["side"], m["side"], m["seed"], CHANNEL, True)
        ref = _Lattice(m["side"], m["side"], m["tau"], **args)
        ref.substeps(case["n"], case["n"], a, b)
        out.append(ref.u)
    return out


def _gradient_prepare(case, seed):
    args, kf, cin = _gradient_inputs(case, seed)
    lat = LBM(case["nx"], case["ny"], 0.7, precision=case["precision"], **args)
    return dict(kind="gradient", lat=lat, k=kf.requires_grad_(), c=cin.requires_grad_(),
                start=lat.save(), n=case["n"], stride=case["stride"], precision=case["precision"])


def _gradient_run(s):
    J = outlet_breakthrough(s["lat"], s["k"], s["c"], s["n"], s["start"], stride=s["stride"])
    gk, gc = torch.autograd.grad(J, [s["k"], s["c"]])
    return dict(J=J.detach().to(s["k"].dtype), k=gk, c=gc)


def _gradient_work(case):
    nodes, size = case["nx"] * case["ny"], case["precision"] // 8
    # the forward state in and out, the rate and its gradient; a forward and a
    # reverse step (105 and 110 operations) a fluid node and substep
    return dict(bytes=0.6 * nodes * (2 * 18 + 2 + 2) * size + nodes,
                flops=0.6 * nodes * case["n"] * 215.0)


def _gradient_exact(case, seed):
    if case["nx"] * case["ny"] * case["n"] > 2 ** 28:
        return None
    args, kf, cin = _gradient_inputs(case, seed)
    k = kf.double().requires_grad_()
    c = cin.double().requires_grad_()
    args["k_field"] = k
    ny = case["ny"]
    ref = _Lattice(case["nx"], ny, 0.7, **args)
    ud = torch.zeros(2 * (case["nx"] + ny), dtype=torch.float64, device="cuda")
    west = torch.zeros_like(ud)
    west[:ny] = 1.0
    fluid_out = (~ref.solid[:, -1]).double()

    def stretch(F, k, c, steps):
        ref.k, J = k, 0.0
        for _ in range(steps):
            F, u = ref.step(F, ud + c * west, 0.0)
            J = J + (u[:, -1] * fluid_out).sum()
        return F, J

    from torch.utils.checkpoint import checkpoint
    F, J, left = ref.F, 0.0, case["n"]
    while left:
        m = min(left, 25)
        F, j = checkpoint(stretch, F, k, c, m, use_reentrant=False)
        J, left = J + j, left - m
    gk, gc = torch.autograd.grad(J, [k, c])
    return dict(J=J.detach(), k=gk, c=gc)


def _continuum_prepare(case, seed):
    mesh, d0, data, edge = _continuum_inputs(case, seed)
    dev = lambda a: torch.from_numpy(a).cuda()
    fem = FEM(**mesh)
    return dict(kind="continuum", fem=fem, d0=dev(d0), data=[dev(v) for v in data], edge=dev(edge),
                d=torch.empty(fem.n, dtype=torch.float64, device="cuda"),
                at=torch.empty(len(edge), dtype=torch.float64, device="cuda"))


def _continuum_run(s):
    fem = s["fem"]
    for values in s["data"]:
        fem.set(s["d0"])
        fem.step(values)
        fem.interpolate(s["edge"], out=s["at"])
    return dict(d=fem.get(s["d"]), at=s["at"])


def _continuum_work(case):
    n = (case["nex"] + 1) * (case["ney"] + 1)
    # the operator's 9 + 9 coefficients once, the state in and out; a right-hand
    # side and about 8 iterations of two products and ten vector operations
    return dict(bytes=n * 8.0 * (18 + 2 * case["iterations"]),
                flops=case["iterations"] * n * (18 + 8 * 56.0))


def _continuum_exact(case, seed):
    mesh, d0, data, edge = _continuum_inputs(case, seed)
    ref = _Continuum(**mesh)
    d = ref.step(np.where(ref.touched, d0, 0.0), data[-1])
    return dict(d=d, at=ref.interpolate(d, edge))


def _hybrid_prepare(case, seed):
    lay = _hybrid_layout(case, seed)
    L = lay["lbm"]
    run_ = Hybrid(lay, precision=case["precision"])
    real = _real(case["precision"])
    return dict(kind="hybrid", run=run_, real=real, precision=case["precision"],
                start=run_.lbm.save(), d0=run_.fem.get(torch.empty(run_.fem.n, dtype=torch.float64, device="cuda")),
                u=torch.empty(L["ny"], L["nx"], dtype=real, device="cuda"),
                d=torch.empty(run_.fem.n, dtype=torch.float64, device="cuda"))


def _hybrid_run(s):
    # from the same instant every time: the pulse would leave the domain
    s["run"].lbm.restore(s["start"])
    s["run"].fem.set(s["d0"])
    s["run"].coarse_step()
    return dict(d=s["run"].fem.get(s["d"]).to(s["real"]),
                u=s["run"].lbm.concentration(out=s["u"], precision=s["precision"]))


def _hybrid_work(case):
    w = _lattice_work(256 * 64, 1.0, case["precision"] // 8, case["eta"] * case["iterations"])
    return dict(bytes=w["bytes"] + 41 * 11 * 8.0 * 20,
                flops=w["flops"] + case["iterations"] * 41 * 11 * (18 + 4 * 56.0))


def _hybrid_exact(case, seed):
    lay = _hybrid_layout(case, seed)
    L, F = dict(lay["lbm"]), lay["fem"]
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    nx, ny, eta = L.pop("nx"), L.pop("ny"), case["eta"]
    ref = _Lattice(nx, ny, L.pop("tau"), edges=L["edges"], vel=dev(L["vel"]), u0=dev(L["u0"]))
    fem = _Continuum(**F)
    s0, s1 = lay["lbm_slots"]
    ua, ub = (torch.zeros(2 * (nx + ny), dtype=torch.float64, device="cuda") for _ in range(2))
    dn, F0 = F["d0"], ref.F
    ua[s0:s1] = dev(fem.interpolate(dn, lay["lbm_points"]))
    trace = ref.trace(dev(lay["gamma_lattice_xy"]))
    for _ in range(case["iterations"]):
        d = fem.step(dn, np.concatenate([lay["fixed_values"], trace.cpu().numpy()]))
        ub[s0:s1] = dev(fem.interpolate(d, lay["lbm_points"]))
        ref.F = F0
        ref.substeps(eta, eta, ua, ub)
        trace = ref.trace(dev(lay["gamma_lattice_xy"]))
    return dict(d=d, u=ref.u)


COEFFS = (1.0, 2.0, 1.0)


def _bimolecular_prepare(case, seed):
    nx, ny = case["nx"], case["ny"]
    args, a, b = _bimolecular_inputs(case, seed)
    run_ = Bimolecular(nx, ny, 0.7, COEFFS, a.cpu().numpy(), b.cpu().numpy(), precision=32, **args)
    field = lambda dt: torch.empty(ny, nx, dtype=dt, device="cuda")
    da = torch.zeros(2 * (nx + ny), dtype=torch.float64, device="cuda")
    da[:ny] = 1.0
    return dict(kind="bimolecular", run=run_, n=case["n"], da=da, db=torch.zeros_like(da),
                alpha=field(torch.float64), beta=field(torch.float64),
                species=[field(torch.float64) for _ in range(3)])


def _bimolecular_run(s):
    r = s["run"]
    r.substeps(s["n"], 1, (s["da"], s["da"]), (s["db"], s["db"]))
    a, b = r.alpha.concentration(out=s["alpha"]), r.beta.concentration(out=s["beta"])
    return [v.float() for v in species_from_invariants(a, b, COEFFS, out=s["species"])]


def _bimolecular_work(case):
    nodes = case["nx"] * case["ny"]
    w = _lattice_work(nodes, case["porosity"], 4, case["n"], fields=2)
    return dict(bytes=w["bytes"] + 12.0 * nodes, flops=w["flops"])


def _bimolecular_exact(case, seed):
    nx, ny = case["nx"], case["ny"]
    args, a, b = _bimolecular_inputs(case, seed)
    u = []
    for u0, west in ((a, 1.0), (b, 0.0)):
        ref = _Lattice(nx, ny, 0.7, u0=u0, **args)
        d = torch.zeros(2 * (nx + ny), dtype=torch.float64, device="cuda")
        d[:ny] = west
        ref.substeps(case["n"], 1, d, d)
        u.append(ref.u)
    nA, nB, nC = COEFFS
    excess = u[0] - nA / nB * u[1]
    uA = excess.clamp(min=0)
    return [uA, nB / nA * (-excess).clamp(min=0), nC / nA * (u[0] - uA)]


_KINDS = {
    "block": (_block_prepare, _block_run, _block_work, _block_exact),
    "channel": (_channel_prepare, _channel_run, _channel_work, _channel_exact),
    "batch": (_batch_prepare, _batch_run, _batch_work, _batch_exact),
    "gradient": (_gradient_prepare, _gradient_run, _gradient_work, _gradient_exact),
    "continuum": (_continuum_prepare, _continuum_run, _continuum_work, _continuum_exact),
    "hybrid": (_hybrid_prepare, _hybrid_run, _hybrid_work, _hybrid_exact),
    "bimolecular": (_bimolecular_prepare, _bimolecular_run, _bimolecular_work, _bimolecular_exact),
}


# ---- FP64 reference in plain torch and numpy -----------------------------------------

class _Lattice:
    """The lattice's update as formulas on whole FP64 arrays: collide, stream
    with halfway bounce-back, boundary data, moments, dissolution."""

    def __init__(self, nx, ny, tau, edges, vel, u0, solid=None, react_mode=0, k=0.0, k_field=None,
                 dissolution=False, mineral=None, walls=False):
        self.nx, self.ny, self.omega, self.edges, self.walls = nx, ny, 1.0 / tau, edges, walls
        dev = dict(device="cuda")
        self.solid = torch.zeros(ny, nx, dtype=torch.bool, **dev) if solid is None else solid != 0
        self.react, self.k = react_mode, k if k_field is None else k_field.double()
        self.dissolves, self.pending = dissolution, torch.zeros_like(self.solid)
        self.mineral = mineral.clone() if dissolution else None
        x, y = torch.arange(nx, **dev)[None, :], torch.arange(ny, **dev)[:, None]
        self.out = []  # the source x - e_i of pull i lies outside
        for cx, cy in E:
            o = torch.zeros(ny, nx, dtype=torch.bool, **dev)
            if edges[0] != 0:
                o = o | (x - cx < 0) | (x - cx >= nx)
            if edges[2] != 0:
                o = o | (y - cy < 0) | (y - cy >= ny)
            self.out.append(o)
        some = torch.stack(self.out).any(0)
        self.edge_nodes = (some & ~self.solid).reshape(-1).nonzero()[:, 0]
        self.some_out = some
        vx, vy = vel
        self.P = [W[i] * (1 + 3 * (cx * vx + cy * vy) + 4.5 * (cx * vx + cy * vy) ** 2
                          - 1.5 * (vx * vx + vy * vy)) for i, (cx, cy) in enumerate(E)]
        self._masks()
        self.u = u0 * (~self.solid)
        self.F = self._collide([p * self.u for p in self.P], self.u)
        if dissolution:
            self._dissolve(self.u)

    def _shift(self, a, i):
        return torch.roll(a, (E[i][1], E[i][0]), (0, 1))  # value at x - e_i

    def _masks(self):
        post = self.solid & ~self.pending
        self.bounce = [self._shift(self.solid, i) & ~self.out[i] for i in range(9)]
        links = [self._shift(post, i) & ~self.out[i] for i in range(9)]
        self.wsolid = sum(W[i] * links[i] for i in range(1, 9))
        self.post = post

    def _rate(self):
        return self.k * (self.wsolid > 0).double() if self.react == 1 else self.k if self.react == 2 else 0.0

    def _collide(self, f, u):
        kr = self._rate()
        return [f[i] + self.omega * (self.P[i] * u - f[i]) - W[i] * kr * u for i in range(9)]

    def step(self, F, up, q):
        f = [torch.where(self.bounce[i], F[OPP[i]], self._shift(F[i], i)) if i else F[0]
             for i in range(9)]
        if self.walls:
            f = self._wall(f)
        f = self._edges(f, up, q)
        u = sum(f) * (~self.solid)
        F = self._collide(f, u)
        if self.dissolves:
            F = [torch.where(self.solid, 0.0, v) for v in F]
        return F, u

    def substeps(self, n, eta, ua, ub, q=0.0):
        for j in range(1, n + 1):
            self.F, self.u = self.step(self.F, (1 - j / eta) * ua + j / eta * ub, q)
            if self.dissolves:
                self._dissolve(self.u)

    def _edges(self, f, up, q):
        """Maximum-entropy data: on a Dirichlet side the unknown populations
        share u - (known) in proportion to their weights, on the east Neumann
        side the outward moment is q."""
        at = self.edge_nodes
        if not len(at):
            return f
        nx, ny = self.nx, self.ny
        x, y = at % nx, at // nx
        g = torch.stack([v.reshape(-1)[at] for v in f])
        unknown = torch.stack([o.reshape(-1)[at] for o in self.out])
        w = torch.tensor(W, dtype=torch.float64, device="cuda")[:, None]
        wu = (w * unknown).sum(0)
        known = g * ~unknown
        slot = torch.full_like(at, -1)
        for s, on, k in ((3, y == ny - 1, 2 * ny + nx + x), (2, y == 0, 2 * ny + x),
                         (1, x == nx - 1, ny + y), (0, x == 0, y)):
            if self.edges[s] == 1:
                slot = torch.where(on, k, slot)
        dirichlet = (up[slot.clamp(min=0)] - known.sum(0)) / wu
        cx = torch.tensor([e[0] for e in E], dtype=torch.float64, device="cuda")[:, None]
        neumann = ((known * cx).sum(0) - q).clamp(min=0) / wu
        g = torch.where(unknown, w * torch.where(slot >= 0, dirichlet, neumann), g)
        return [v.reshape(-1).index_copy(0, at, g[i]).view(ny, nx) for i, v in enumerate(f)]

    def _wall(self, f):
        """Zero-flux maximum-entropy walls: unknowns w_i exp(-1 - g e_i.n)."""
        at = (sum(self.bounce[1:]) > 0) & ~self.solid & ~self.some_out
        at = at.reshape(-1).nonzero()[:, 0]
        g = torch.stack([v.reshape(-1)[at] for v in f])
        link = torch.stack([b.reshape(-1)[at] for b in self.bounce])
        w = torch.tensor(W, dtype=torch.float64, device="cuda")[:, None]
        c = torch.tensor(E, dtype=torch.float64, device="cuda")
        m = torch.round(-36 * (w * link).T @ c)
        length = m.square().sum(1).sqrt()
        d = c @ m.T
        a = d / length.clamp(min=1)
        neg = link & (d < 0)
        flux = (torch.where(neg, 0.0, a * g)).sum(0)  # carried into the wall
        root = neg.any(0) & (flux > 0)
        b = torch.where(neg, -a, 0.0)
        t = torch.zeros_like(flux)
        goal = torch.log(torch.where(root, flux, 1.0))
        for _ in range(100):
            e = torch.where(neg, w * b * torch.exp(t * b - 1), 0.0)
            L = e.sum(0)
            step = torch.where(root, (torch.log(L) - goal) * L / (b * e).sum(0), 0.0)
            t = t - step
            if not bool((step.abs() > 1e-15 * (1 + t.abs())).any()):
                break
        new = torch.where(root, w * torch.exp(t * b - 1), 0.0)
        g = torch.where(neg & (length > 0), new, g)
        return [v.reshape(-1).index_copy(0, at, g[i]).view(self.ny, self.nx) for i, v in enumerate(f)]

    def _dissolve(self, u):
        """Each solid node loses what its fluid neighbours' sinks take from it;
        one that has nothing left is solid for one more streaming."""
        fluid = ~self.solid
        r = torch.where(fluid & (self.wsolid > 0), self._rate() * u / self.wsolid.clamp(min=1e-3), 0.0)
        take = sum(W[i] * torch.where(self.out[i], 0.0, self._shift(r, i)) for i in range(1, 9))
        live = self.solid & ~self.pending
        near = sum(self._shift(~self.post, i) & ~self.out[i] for i in range(1, 9)) > 0
        self.mineral = torch.where(live & near, self.mineral - take, self.mineral)
        done = live & near & (self.mineral <= 0)
        if bool(self.pending.any()) or bool(done.any()):
            self.solid = self.solid & ~self.pending
            self.pending = done
            self._masks()
            self.edge_nodes = (self.some_out & ~self.solid).reshape(-1).nonzero()[:, 0]

    def trace(self, xy):
        x1, y1 = xy.floor().long().T
        if self.edges[0] != 0:
            x1 = x1.clamp(max=self.nx - 2)
        if self.edges[2] != 0:
            y1 = y1.clamp(max=self.ny - 2)
        gx, gy = (xy - torch.stack([x1, y1], 1)).T
        at = lambda dx, dy: self.u[(y1 + dy) % self.ny, (x1 + dx) % self.nx]
        return (at(0, 0) * (1 - gx) + at(1, 0) * gx) * (1 - gy) + \
            (at(0, 1) * (1 - gx) + at(1, 1) * gx) * gy


class _Continuum:
    """Q1 elements and the trapezoidal rule, assembled by quadrature-free
    element matrices and solved by block elimination along x."""

    def __init__(self, nex, ney, x0, y0, hx, hy, D, v, theta, dt, supg, elem_active, dirichlet, d0):
        self.nex, self.ney, self.hx, self.hy, self.x0, self.y0 = nex, ney, hx, hy, x0, y0
        m = lambda h: h / 6 * np.array([[2.0, 1], [1, 2]])
        k = lambda h: 1 / h * np.array([[1.0, -1], [-1, 1]])
        c = 0.5 * np.array([[-1.0, 1], [-1, 1]])
        tau, (vx, vy) = 0.0, v
        if supg and vx:  # flow along x
            pe = vx * hx / (2 * D)
            tau = hx / (2 * vx) * (1 / math.tanh(pe) - 1 / pe)
        M = np.einsum("ab,cd->cadb", m(hx), m(hy)) + tau * vx * np.einsum("ab,cd->cadb", c.T, m(hy))
        K = vx * np.einsum("ab,cd->cadb", c, m(hy)) + D * (
            np.einsum("ab,cd->cadb", k(hx), m(hy)) + np.einsum("ab,cd->cadb", m(hx), k(hy))) + \
            tau * vx * vx * np.einsum("ab,cd->cadb", k(hx), m(hy))
        nxn, nyn = nex + 1, ney + 1
        act = np.ones((ney, nex)) if elem_active is None else elem_active.astype(float)
        # [column i][offset di + 1] blocks over y of A and B
        A, B = (np.zeros((nxn, 3, nyn, nyn)) for _ in range(2))
        touched = np.zeros((nyn, nxn), bool)
        j = np.arange(ney)
        for cy in range(2):
            for cx in range(2):
                touched[cy:cy + ney, cx:cx + nex] |= act > 0
                for dy in range(2):
                    for dx in range(2):
                        a = M[cy, cx, dy, dx] + theta * dt * K[cy, cx, dy, dx]
                        b = M[cy, cx, dy, dx] - (1 - theta) * dt * K[cy, cx, dy, dx]
                        for i in range(nex):
                            A[i + cx, dx - cx + 1, j + cy, j + dy] += a * act[:, i]
                            B[i + cx, dx - cx + 1, j + cy, j + dy] += b * act[:, i]
        self.touched = touched.reshape(-1)
        fixed = ~touched
        self.dirichlet = np.asarray(dirichlet)
        fixed.reshape(-1)[self.dirichlet] = True
        for i in range(nxn):
            rows = np.nonzero(fixed[:, i])[0]
            A[i][:, rows, :] = 0.0
            B[i][:, rows, :] = 0.0
            A[i, 1, rows, rows] = 1.0
        self.A, self.B = A, B

    def step(self, d, values):
        nxn, nyn = self.nex + 1, self.ney + 1
        X = d.reshape(nyn, nxn).T
        b = np.einsum("iyz,iz->iy", self.B[:, 1], X)
        b[1:] += np.einsum("iyz,iz->iy", self.B[1:, 0], X[:-1])
        b[:-1] += np.einsum("iyz,iz->iy", self.B[:-1, 2], X[1:])
        full = b.T.copy().reshape(-1)
        full[self.dirichlet] = values
        b = full.reshape(nyn, nxn).T.copy()
        C, g = np.zeros((nxn, nyn, nyn)), np.zeros((nxn, nyn))
        for i in range(nxn):
            D = self.A[i, 1].copy()
            r = b[i].copy()
            if i:
                D -= self.A[i, 0] @ C[i - 1]
                r -= self.A[i, 0] @ g[i - 1]
            s = np.linalg.solve(D, np.concatenate([self.A[i, 2], r[:, None]], 1))
            C[i], g[i] = s[:, :-1], s[:, -1]
        for i in range(nxn - 2, -1, -1):
            g[i] -= C[i] @ g[i + 1]
        return np.ascontiguousarray(g.T).reshape(-1)

    def interpolate(self, d, xy):
        px, py = (xy[:, 0] - self.x0) / self.hx, (xy[:, 1] - self.y0) / self.hy
        i = np.clip(np.floor(px).astype(int), 0, self.nex - 1)
        j = np.clip(np.floor(py).astype(int), 0, self.ney - 1)
        gx, gy = px - i, py - j
        d = d.reshape(self.ney + 1, self.nex + 1)
        return (d[j, i] * (1 - gx) + d[j, i + 1] * gx) * (1 - gy) + \
            (d[j + 1, i] * (1 - gx) + d[j + 1, i + 1] * gx) * gy
