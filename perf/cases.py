"""Workloads of the DSMC-LBM library as a program uses them: what is timed when the library's
speed is measured, and the values its deterministic parts have to give.

Every case is one pass through the public calls of the binding (which are the C ABI's):
hybrid steps of one channel, of a batch of channels, host-buffer steps, DSMC steps alone,
LB steps alone, the two mappings, and the gradient of the differentiated LBM. Sizes are
those of the named workloads, tests and benchmark of this repository and odd sizes between.
A pass that advances particles ends with the snapshot a program takes of them: the live
particles of every bin (the slots past a cell's count are scratch and are zeroed in the copy),
with the counts, the collision state, the moment sums and the populations.

`exact` restates the LB step, DSMC2LB, the LB2DSMC coefficients and the interface loss in FP64
torch. The particle trajectories have no such value: their draws, pairs and rounding are the
method's own.
"""
import math

import numpy as np
import torch

from paper_1512_08042_gb300 import binding as B
from paper_1512_08042_gb300 import workloads as W

DEV = "cuda:0"


# ---------------------------------------------------------------------------------------
# cases

def listed():
    return [
        # the paper's quasi-1D channel (64 cells, FP64, mapping at two cells): a few thousand
        # particles, so launches and latency are all of it
        dict(name="hybrid_64x1_fp64", kind="hybrid", ncx=64, ncy=1, ncz=0, ppc=100, lb_ratio=1, lattice=39,
             real_bytes=8, kn=0.1, kn_end=0.0, bgk=0, nsteps=20),
        # the Sec. 4 proof of concept: D3Q19 without regularisation, equilibrium DSMC2LB on one row
        dict(name="hybrid_poc_d3q19_fp64", kind="hybrid", ncx=64, ncy=64, ncz=0, ppc=50, lb_ratio=1,
             lattice=19, real_bytes=8, kn=0.05, kn_end=0.0, bgk=1, nsteps=20),
        # the ordinary 2D channel, many steps in one call
        dict(name="hybrid_64x256", kind="hybrid", ncx=64, ncy=256, ncz=0, ppc=50, lb_ratio=2, lattice=39,
             real_bytes=4, kn=0.05, kn_end=0.0, bgk=0, nsteps=20),
        # the same channel driven by a host program: lists in and strip moments out every step
        dict(name="host_step_64x256", kind="host", ncx=64, ncy=256, ncz=0, ppc=50, lb_ratio=2, lattice=39,
             real_bytes=4, kn=0.05, kn_end=0.0, bgk=0, nsteps=1),
        # the largest channel: 105M particles, Kn varying along it
        dict(name="hybrid_512x4096_knvar", kind="hybrid", ncx=512, ncy=4096, ncz=0, ppc=50, lb_ratio=2,
             lattice=39, real_bytes=4, kn=0.005, kn_end=0.5, bgk=0, nsteps=20),
        # full 3D
        dict(name="hybrid_64x256x8", kind="hybrid", ncx=64, ncy=256, ncz=8, ppc=50, lb_ratio=2, lattice=39,
             real_bytes=4, kn=0.05, kn_end=0.0, bgk=0, nsteps=20),
        # the ensemble of uneven channels
        dict(name="ensemble_64", kind="ensemble", n=64, shape_seed=1000, nsteps=10),
        # DSMC alone at sizes that divide nothing, in a dense, collisional gas
        dict(name="dsmc_131x509", kind="dsmc", ncx=131, ncy=509, ncz=0, ppc=37, lb_ratio=1, lattice=39,
             real_bytes=4, kn=0.02, kn_end=0.0, bgk=0, nsteps=10),
        # LB alone: the ordinary lattice and the largest
        dict(name="lbm_128x512", kind="lbm", ncx=64, ncy=256, ncz=0, ppc=10, lb_ratio=2, lattice=39,
             real_bytes=4, kn=0.05, kn_end=0.0, bgk=0, nsteps=10),
        dict(name="lbm_1024x8192", kind="lbm", ncx=512, ncy=4096, ncz=0, ppc=10, lb_ratio=2, lattice=39,
             real_bytes=4, kn=0.05, kn_end=0.0, bgk=0, nsteps=4),
        # the differentiated LBM: loss and gradients through checkpointed steps
        dict(name="gradient_256x128", kind="gradient", ncx=128, ncy=64, ncz=0, ppc=10, lb_ratio=2, lattice=39,
             real_bytes=4, kn=0.1, kn_end=0.0, bgk=0, nsteps=100, ckpt=50, coupled=0),
        # the two mappings on a strip of 2048 cells
        dict(name="mappings_512x4", kind="mappings", ncx=512, ncy=8, ncz=0, ppc=50, lb_ratio=2, lattice=39,
             real_bytes=4, kn=0.05, kn_end=0.0, bgk=0, nsteps=1),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _channel(rng, max_cells, three_d=True):
    """A channel of at most max_cells cells: height, streamwise cells, layers, particles per cell,
    resolution, lattice, precision and Kn of the ranges above."""
    real_bytes = 8 if rng.random() < 0.25 else 4
    if real_bytes == 8:
        max_cells = min(max_cells, 8192)
    total = _log(rng, 512, max_cells)
    ncx = int(max(16, min(512, _log(rng, 16, min(512.0, total / 4)))))
    ncz = rng.choice([2, 3, 5, 8]) if three_d and rng.random() < 0.25 else 0
    ncy = int(max(4, total / ncx / max(1, ncz)))
    kn = _log(rng, max(0.005, 1.0 / ncx), 0.5)
    lattice = 19 if rng.random() < 0.25 else 39
    c = dict(ncx=ncx, ncy=ncy, ncz=ncz, ppc=rng.randint(20, 100), lb_ratio=rng.choice([1, 2]), lattice=lattice,
             real_bytes=real_bytes, kn=kn, kn_end=0.0, bgk=int(lattice == 19 and rng.random() < 0.5))
    c["ppc"] = min(c["ppc"], 100_000_000 // (ncx * ncy * max(1, ncz)))
    if ncz == 0 and rng.random() < 0.2:
        c["kn_end"] = min(0.5, 4 * kn)
    return c


def draw(rng):
    kind = rng.choice(["hybrid", "hybrid", "hybrid", "host", "dsmc", "dsmc", "ensemble", "lbm", "gradient",
                       "mappings"])
    if kind == "ensemble":
        return dict(kind=kind, n=rng.randint(8, 64), shape_seed=rng.randint(1, 10 ** 6), nsteps=rng.randint(1, 20))
    if kind == "gradient":
        return dict(kind=kind, ncx=rng.randint(12, 128), ncy=rng.randint(6, 80), ncz=0, ppc=10,
                    lb_ratio=rng.choice([1, 2]), lattice=rng.choice([39, 39, 19]), real_bytes=rng.choice([4, 4, 8]),
                    kn=_log(rng, 0.05, 0.5), kn_end=0.0, bgk=0, nsteps=rng.randint(10, 100), ckpt=rng.randint(10, 50),
                    coupled=rng.randint(0, 1))
    if kind == "mappings":
        return dict(kind=kind, ncx=int(_log(rng, 16, 512)), ncy=rng.randint(6, 12), ncz=0, ppc=rng.randint(20, 100),
                    lb_ratio=rng.choice([1, 2]), lattice=rng.choice([39, 39, 19]), real_bytes=rng.choice([4, 4, 8]),
                    kn=0.05, kn_end=0.0, bgk=0, nsteps=1)
    c = _channel(rng, 2_000_000 if kind in ("hybrid", "dsmc") else 200_000, three_d=kind != "host")
    c["kind"] = kind
    c["nsteps"] = 1 if kind == "host" else rng.randint(1, 20)
    if kind == "lbm":
        c["ppc"], c["kn_end"] = 10, 0.0
    return c


# ---------------------------------------------------------------------------------------
# inputs

def _cfg(case, seed):
    c = case
    cfg = W.config(ncx=c["ncx"], ncy=c["ncy"], ncz=c["ncz"], ppc=c["ppc"], lb_ratio=c["lb_ratio"],
                   lattice=c["lattice"], real_bytes=c["real_bytes"], kn=c["kn"], seed=1 + int(seed) % (1 << 40),
                   lb_collision=c["bgk"], d2l_mode=c["bgk"])
    if c["kn_end"] > 0:
        cfg.update(kn_profile=1, kn_end=c["kn_end"])
    if c["bgk"]:
        cfg["coupling"] = "buffer_row"
    return cfg


def _params(case):
    """Lattice size, relaxation time and force increment of a case (Eq. tau, the no-slip parabola)."""
    c = case
    nx, ny = c["ncx"] * c["lb_ratio"], c["ncy"] * c["lb_ratio"]
    nz = c["ncz"] * c["lb_ratio"] if c["ncz"] >= 2 else 1
    r = math.sqrt(1.5) if c["lattice"] == 39 else math.sqrt(3.0)
    tau = math.sqrt(math.pi / 8.0) * r * c["kn"] * nx + 0.5
    return nx, ny, nz, tau, 8.0 * (tau - 0.5) * 0.1 / (r * r) / (nx * nx)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _populations(case, seed):
    """Populations around rest, w rho (1 + 0.05 U), rho = 1 + 0.02 U, U in (-1, 1), rounded to the
    state precision."""
    nx, ny, nz, _, _ = _params(case)
    g = _gen(seed)
    q = case["lattice"]
    w = torch.as_tensor(_lattice(q)[1], dtype=torch.float32, device=DEV).view(q, 1)
    rho = 1.0 + 0.02 * (2.0 * torch.rand(1, nx * ny * nz, generator=g, device=DEV) - 1.0)
    f = 2.0 * torch.rand(q, nx * ny * nz, generator=g, device=DEV) - 1.0
    f.mul_(0.05).add_(1.0).mul_(rho).mul_(w)
    return f.to(torch.float32 if case["real_bytes"] == 4 else torch.float64)


def _sums(case, seed):
    """Cumulative moment sums of 100 samples of a slowly drifting gas per cell, and the sample
    count: counts around ppc, velocities of unit variance, third moments to match."""
    g = _gen(seed + 7)
    n = case["ncx"] * case["ncy"]
    s = 100
    u = 0.05 * torch.randn(n, 3, generator=g, device=DEV, dtype=torch.float64)
    cov = torch.eye(3, device=DEV, dtype=torch.float64) + 0.0
    cov = cov + 0.03 * torch.randn(n, 3, 3, generator=g, device=DEV, dtype=torch.float64)
    cov = 0.5 * (cov + cov.transpose(1, 2))
    third = 0.02 * torch.randn(n, 10, generator=g, device=DEV, dtype=torch.float64)
    num = (s * case["ppc"] * (1.0 + 0.02 * torch.randn(n, generator=g, device=DEV, dtype=torch.float64))).round()
    cols = [torch.ones_like(num)] + [u[:, i] for i in range(3)]
    m2 = lambda i, j: cov[:, i, j] + u[:, i] * u[:, j]  # noqa: E731
    cols += [m2(i, j) for i, j in _PAIRS]
    cols += [third[:, k] + u[:, i] * m2(j, l) + u[:, j] * m2(i, l) + u[:, l] * m2(i, j) -
             2.0 * u[:, i] * u[:, j] * u[:, l] for k, (i, j, l) in enumerate(_TRIPLES)]
    return (torch.stack(cols, 1) * num[:, None]).contiguous(), s


def _node_params(case, seed):
    """Per-node force increments and relaxation times around the channel's, interface nodes
    (a strip of 8 rows) and targets."""
    nx, ny, _, tau, gs = _params(case)
    real = torch.float32 if case["real_bytes"] == 4 else torch.float64
    g = _gen(seed + 3)
    gn = (gs * (1.0 + 0.1 * torch.randn(nx * ny, generator=g, device=DEV))).to(real)
    tn = (tau * (1.0 + 0.02 * torch.randn(nx * ny, generator=g, device=DEV))).to(real)
    rows = min(8, ny)  # across the channel, as the coupling strip
    y0 = ny // 2 - rows // 2
    nodes = torch.arange(y0 * nx, (y0 + rows) * nx, device=DEV)
    # a denser gas with a plane profile, and the scatter of sampled moments
    x = (torch.arange(nx, device=DEV, dtype=torch.float32) + 0.5) / nx
    targets = 0.05 * torch.randn(nodes.numel(), 20, generator=g, device=DEV)
    targets[:, 0] += 1.2
    targets[:, 2] += (1.2 * x * (1.0 - x)).repeat(rows)
    return gn, tn, nodes.to(torch.int32), targets.to(real)


def _strip_nodes(case):
    """Half of the cell rows of a mapping case, as cells and the nodes they hold."""
    c = case
    r, nx, rows = c["lb_ratio"], c["ncx"] * c["lb_ratio"], c["ncy"] // 2
    cells = torch.arange(rows * c["ncx"], device=DEV, dtype=torch.int32)
    nodes = torch.arange(rows * r * nx, device=DEV, dtype=torch.int32)
    return nodes, cells


class State:
    pass


_STREAMS = []


def _stream():
    """The program's one stream: its contexts' calls run one after another on it."""
    if not _STREAMS:
        _STREAMS.append(torch.cuda.Stream(torch.device(DEV)))
    return _STREAMS[0]


def _context(cfg):
    h = B.Hybrid(cfg, device=DEV, stream=_stream())
    return h, torch.arange(int(h.L.bin), device=DEV)[None, :]


def prepare(case, seed):
    st = State()
    st.case, kind = case, case["kind"]
    if kind == "ensemble":
        cfgs = [dict(c, seed=c["seed"] + 1000 * (1 + int(seed) % (1 << 40)))
                for c in W.ensemble_configs(case["n"], seed=case["shape_seed"])]
        st.batch = B.Batch(cfgs, device=DEV, stream=_stream())
        sites = [W.coupling_sites(c) for c in cfgs]
        st.nodes, st.cells = [s[0] for s in sites], [s[1] for s in sites]
        # views of the replicas' state that the program reads after every call
        reps = st.batch.replicas
        st.views = {k: [getattr(h, k)().reshape(-1) for h in reps] for k in ("acc", "crmax", "rem", "nbar_sum")}
        st.f = [[h.f(half).reshape(-1) for h in reps] for half in (0, 1)]
        st.batch.hybrid_step(st.nodes, st.cells, nsteps=8, use_graph=False)  # past the first samples
        return st
    cfg = _cfg(case, seed)
    if kind in ("hybrid", "host", "dsmc"):
        st.h, st.slot = _context(cfg)
        nodes, cells = W.coupling_sites(cfg)
        if kind == "host":
            st.nodes, st.cells = torch.from_numpy(nodes).pin_memory(), torch.from_numpy(cells).pin_memory()
            st.out = torch.zeros(case["nsteps"], max(1, len(cells)), 20, dtype=torch.float64).pin_memory()
            st.status = torch.zeros(case["nsteps"], dtype=torch.int32).pin_memory()
            nodes, cells = torch.from_numpy(nodes).to(DEV), torch.from_numpy(cells).to(DEV)
        else:
            nodes = st.nodes = torch.from_numpy(nodes).to(DEV)
            cells = st.cells = torch.from_numpy(cells).to(DEV)
        if kind == "dsmc":
            st.h.dsmc_step(4)
        else:  # past the first, noisy samples
            st.h.hybrid_step(nodes, cells, nsteps=8, use_graph=False)
        return st
    if kind == "lbm":
        st.h = B.Hybrid(cfg, device=DEV, stream=_stream())
        st.h.f().copy_(_populations(case, seed).view(st.h.f().shape))
        torch.cuda.synchronize()
        return st
    if kind == "gradient":
        st.h = B.Hybrid(cfg, device=DEV, stream=_stream())
        st.f0 = _populations(case, seed).view(st.h.f().shape).requires_grad_(True)
        st.g, st.tau, st.nodes, st.targets = _node_params(case, seed)
        st.g.requires_grad_(True)
        st.tau.requires_grad_(True)
        if case["coupled"]:
            st.acc, st.nsamples = _sums(case, seed)
            st.acc.requires_grad_(True)
            st.d2l = _strip_nodes(case)[0]
        return st
    st.h = B.Hybrid(cfg, device=DEV, stream=_stream())
    st.nodes, st.cells = _strip_nodes(case)
    acc, s = _sums(case, seed)
    st.h.acc().copy_(acc)
    st.h.f().copy_(_populations(case, seed).view(st.h.f().shape))
    st.h.set_counters(nsamples=s)
    # views of what the mappings write: the listed cells' Grad records (FP64: rho, the new count, a2,
    # a3, u, C), counts and bins, and the populations
    n, b, es, half = st.cells.numel(), int(st.h.L.bin), case["real_bytes"], st.h.current()[0]
    off = int(st.h.L.map_scratch)
    rec = st.h.arena[off:off + 176 * n].view(torch.float64).view(n, 22)
    off = int(st.h.L.count[half])
    st.counts = st.h.arena[off:off + 4 * n].view(torch.int32)
    off = int(st.h.L.part[half])
    st.particles = st.h.arena[off:off + n * b * 8 * es].view(st.h.real).view(n, b, 8)[:, :, :5]
    st.slot = torch.arange(b, device=DEV, dtype=torch.int32)[None, :, None]
    st.out = dict(f=st.h.f(), rho=rec[:, 0], coefficients=rec[:, 2:], counts=st.counts)
    return st


# ---------------------------------------------------------------------------------------
# one pass

def _snapshot(h, slot, f=True):
    """The state after a call, on the context's stream: live particle records (x, y, vx, vy, vz,
    in 3D z), counts, collision state, moment sums and populations."""
    with torch.cuda.stream(h.stream):
        nrec = 6 if h.three_d() else 5
        counts = h.counts()
        nc, b = int(h.L.ncells), int(h.L.bin)
        off = int(h.L.part[h.current()[0]])
        es = 4 if h.real == torch.float32 else 8
        rec = h.arena[off:off + nc * b * 8 * es].view(h.real).view(nc, b, 8)
        live = (slot < counts[:, None])[:, :, None]
        out = dict(particles=torch.where(live, rec[:, :, :nrec], 0.0), counts=counts, crmax=h.crmax(), rem=h.rem(),
                   nbar_sum=h.nbar_sum(), acc=h.acc())
        if f:
            out["f"] = h.f()
    return out


def run(st):
    case = st.case
    kind = case["kind"]
    if kind == "hybrid":
        st.h.hybrid_step(st.nodes, st.cells if st.cells.numel() else None, nsteps=case["nsteps"])
        return _snapshot(st.h, st.slot)
    if kind == "dsmc":
        st.h.dsmc_step(case["nsteps"])
        return _snapshot(st.h, st.slot, f=False)
    if kind == "host":
        # the moments of the coupled cells and the status word, in host memory after the wait
        st.h.hybrid_step_host(st.nodes, st.cells, st.out, st.status, nsteps=case["nsteps"])
        st.h.host_wait(0)
        return dict(moments=st.out, status=st.status, f=st.h.f(), acc=st.h.acc(), crmax=st.h.crmax(), rem=st.h.rem(),
                    nbar_sum=st.h.nbar_sum())
    if kind == "ensemble":
        st.batch.hybrid_step(st.nodes, st.cells, nsteps=case["nsteps"])
        # the ensemble's result: every replica's moment sums, collision state and populations
        with torch.cuda.stream(st.batch.stream):
            out = {k: torch.cat(v) for k, v in st.views.items()}
            out["f"] = torch.cat(st.f[st.batch.replicas[0].current()[1]])
        return out
    if kind == "lbm":
        st.h.lbm_step(case["nsteps"])
        return st.h.f()
    if kind == "gradient":
        if case["coupled"]:
            loss = B.coupled_interface_loss(st.h, st.acc, st.nsamples, st.d2l, st.g, st.tau, st.f0, st.nodes,
                                            st.targets, case["nsteps"], case["ckpt"])
            ga, gg, gt, gf = torch.autograd.grad(loss, (st.acc, st.g, st.tau, st.f0))
            return dict(loss=loss.detach(), g=gg, tau=gt, f0=gf, acc=ga)
        loss = B.interface_loss(st.h, st.g, st.tau, st.f0, st.nodes, st.targets, case["nsteps"], case["ckpt"])
        gg, gt, gf = torch.autograd.grad(loss, (st.g, st.tau, st.f0))
        return dict(loss=loss.detach(), g=gg, tau=gt, f0=gf)
    st.h.map_dsmc_to_lbm(st.nodes)
    st.h.map_lbm_to_dsmc(st.cells)
    with torch.cuda.stream(st.h.stream):  # the regenerated particles of the listed cells
        particles = torch.where(st.slot < st.counts[:, None, None], st.particles, 0.0)
    return dict(st.out, particles=particles)


# ---------------------------------------------------------------------------------------
# the work of a pass

def work(case):
    """Every step reads and writes the particles (position and velocity), the per-cell state and
    the populations once; a gradient step reads the populations and the adjoint and writes the
    adjoint, beside the forward step."""
    kind = case["kind"]
    if kind == "ensemble":
        tot = dict(bytes=0.0, flops=0.0)
        for c in W.ensemble_configs(case["n"], seed=case["shape_seed"]):
            w = work(dict(kind="host", ncx=c["ncx"], ncy=1, ncz=0, ppc=c["ppc"], lb_ratio=1, lattice=39, real_bytes=4,
                          kn=c["kn"], kn_end=0.0, bgk=0, nsteps=case["nsteps"]))
            tot = {k: tot[k] + w[k] for k in tot}
        return tot
    rb, q, n = case["real_bytes"], case["lattice"], case["nsteps"]
    nx, ny, nz, _, _ = _params(case)
    nodes = nx * ny * nz
    cells = case["ncx"] * case["ncy"] * max(1, case["ncz"])
    lb_bytes, lb_flops = nodes * (2 * q * rb + (rb if case["kn_end"] > 0 else 0)), nodes * q * 25.0
    if kind == "lbm":
        return dict(bytes=n * lb_bytes, flops=n * lb_flops)
    if kind == "gradient":
        step = nodes * (2 * q * rb + 2 * rb) + nodes * (3 * q * rb + 6 * rb)
        return dict(bytes=n * step, flops=n * 4 * lb_flops)
    if kind == "mappings":
        m = (case["ncy"] // 2) * case["ncx"]
        mn = m * case["lb_ratio"] ** 2
        return dict(bytes=m * 160 + 2 * mn * q * rb + m * (176 + 5 * rb * case["ppc"]) + cells * 8,
                    flops=mn * q * 60.0 + m * (q * 60.0 + case["ppc"] * 200.0))
    comps = 6 if case["ncz"] >= 2 else 5
    part, per_cell = cells * case["ppc"], 2 * (2 * rb + 4 + 4 + 160)
    bytes_, flops = n * (part * 2 * comps * rb + cells * per_cell), n * part * 80.0
    if kind != "dsmc":
        bytes_, flops = bytes_ + n * lb_bytes, flops + n * lb_flops
    if kind != "host":  # the snapshot
        bytes_ += part * comps * rb
    return dict(bytes=bytes_, flops=flops)


# ---------------------------------------------------------------------------------------
# FP64 values

_PAIRS = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]
_TRIPLES = [(0, 0, 0), (0, 0, 1), (0, 0, 2), (0, 1, 1), (0, 1, 2), (0, 2, 2), (1, 1, 1), (1, 1, 2), (1, 2, 2), (2, 2, 2)]


def _shell(base):
    """All distinct signed permutations of a speed."""
    out = set()
    for p in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        for s in range(8):
            out.add(tuple(base[p[i]] * (1 - 2 * (s >> i & 1)) for i in range(3)))
    return out


def _lattice(q):
    """Speeds and weights by Gauss-Hermite shells, in the library's row order (its public table)."""
    e = B.lattice(q)[0]
    if q == 39:
        shells = [((0, 0, 0), 1 / 12), ((1, 0, 0), 1 / 12), ((1, 1, 1), 1 / 27), ((2, 0, 0), 2 / 135),
                  ((2, 2, 0), 1 / 432), ((3, 0, 0), 1 / 1620)]
    else:
        shells = [((0, 0, 0), 1 / 3), ((1, 0, 0), 1 / 18), ((1, 1, 0), 1 / 36)]
    table = {v: w for b, w in shells for v in _shell(b)}
    return e, np.array([table[tuple(int(x) for x in v)] for v in e])


class _LB:
    """The LB step in FP64: pull by an index table (wall sources point at the wall densities
    appended to the populations), moments and series by matrices."""

    def __init__(self, case):
        self.bgk, self.q = case["bgk"], case["lattice"]
        nx, ny, nz, self.tau0, self.g0 = _params(case)
        e, w = _lattice(self.q)
        r = math.sqrt(1.5) if self.q == 39 else math.sqrt(3.0)
        t = lambda a: torch.as_tensor(np.asarray(a), dtype=torch.float64, device=DEV)  # noqa: E731
        xi = r * e
        cols = [np.ones(self.q)] + [xi[:, i] for i in range(3)] + [xi[:, i] * xi[:, j] for i, j in _PAIRS]
        cols += [xi[:, i] * xi[:, j] * xi[:, k] for i, j, k in _TRIPLES]
        self.mono = t(np.stack(cols, 1))  # raw moments of a population
        mult2 = [1, 2, 2, 1, 2, 1]
        mult3 = [1, 3, 3, 3, 6, 3, 1, 3, 3, 1]
        her = [np.ones(self.q)] + [xi[:, i] for i in range(3)]
        her += [0.5 * m * (xi[:, i] * xi[:, j] - (i == j)) for m, (i, j) in zip(mult2, _PAIRS)]
        for m, (i, j, k) in zip(mult3, _TRIPLES):
            h = xi[:, i] * xi[:, j] * xi[:, k] - xi[:, i] * (j == k) - xi[:, j] * (i == k) - xi[:, k] * (i == j)
            her.append(m * h / 6.0 * (self.q == 39))
        self.her, self.w = t(np.stack(her, 1)), t(w)
        n = nx * ny * nz
        self.n, rows = n, ny * nz
        x = torch.arange(nx, device=DEV).view(1, 1, nx)
        y = torch.arange(ny, device=DEV).view(1, ny, 1)
        z = torch.arange(nz, device=DEV).view(nz, 1, 1)
        idx = torch.empty(self.q, n, dtype=torch.int64, device=DEV)
        left, right = [], []
        for a in range(self.q):
            ex, ey, ez = (int(v) for v in e[a])
            row = ((z - ez) % nz) * ny + (y - ey) % ny
            sx = (x - ex).expand(nz, ny, nx)
            i = a * n + row * nx + sx
            dest = (z * ny + y).expand(nz, ny, nx)
            i = torch.where(sx < 0, self.q * n + a * 2 * rows + dest, i)
            i = torch.where(sx >= nx, self.q * n + (a * 2 + 1) * rows + dest, i)
            idx[a] = i.reshape(-1)
            src = (a * n + row * nx).reshape(-1)
            left += [src + k for k in range(-ex)]
            right += [src + nx - ex + k for k in range(ex)]
        self.idx, self.left, self.right = idx, torch.stack(left), torch.stack(right)
        self.inv_flux = 1.0 / float(sum(w[a] * e[a, 0] for a in range(self.q) if e[a, 0] > 0))

    def pull(self, f):
        flat = f.reshape(-1)
        walls = torch.stack([flat[self.left].sum(0), flat[self.right].sum(0)]) * self.inv_flux
        src = torch.cat([flat, (self.w[:, None, None] * walls[None]).reshape(-1)])
        return src[self.idx.reshape(-1)].view(self.q, self.n)

    def step(self, f, g=None, tau=None):
        g = self.g0 if g is None else g
        tau = self.tau0 if tau is None else tau
        om, of = 1.0 - 1.0 / tau, 1.0 - 0.5 / tau
        fs = self.pull(f)
        m = self.mono.t() @ fs
        rho = m[0]
        u = [m[1] / rho, m[2] / rho + 0.5 * g, m[3] / rho]
        gv = [0.0, g, 0.0]
        a1 = [0.0, -0.5 * rho * g, 0.0]
        ke, omr = (1.0 - om, 0.0 * om) if self.bgk else (1.0, om)
        rk = ke * rho
        out = [rk] + [rk * u[i] + omr * a1[i] + of * rho * gv[i] for i in range(3)]
        for k, (i, j) in enumerate(_PAIRS):
            neq = m[4 + k] - rho * (u[i] * u[j] + (i == j))
            out.append(rk * u[i] * u[j] + omr * neq + of * rho * (gv[i] * u[j] + gv[j] * u[i]))
        for k, (i, j, l) in enumerate(_TRIPLES):
            sym = u[i] * (j == l) + u[j] * (i == l) + u[l] * (i == j)
            sa = a1[i] * (j == l) + a1[j] * (i == l) + a1[l] * (i == j)
            neq = m[10 + k] - rho * (u[i] * u[j] * u[l] + sym) - sa
            force = gv[i] * u[j] * u[l] + gv[j] * u[i] * u[l] + gv[l] * u[i] * u[j]
            out.append(rk * u[i] * u[j] * u[l] + omr * neq + of * rho * force)
        out = self.w[:, None] * (self.her @ torch.stack([o.expand(self.n) for o in out]))
        return out + om * fs if self.bgk else out

    def grad_coefficients(self, f):
        """rho, u and the comoving a2, a3 of populations f [q, n] (20 rows)."""
        m = self.mono.t() @ f
        rho = m[0]
        u = [m[1 + i] / rho for i in range(3)]
        p2 = {ij: m[4 + k] / rho for k, ij in enumerate(_PAIRS)}
        raw = lambda i, j: p2[(min(i, j), max(i, j))]  # noqa: E731
        rows = [rho] + u + [raw(i, j) - u[i] * u[j] - float(i == j) for i, j in _PAIRS]
        rows += [m[10 + k] / rho - u[i] * raw(j, l) - u[j] * raw(i, l) - u[l] * raw(i, j) + 2.0 * u[i] * u[j] * u[l]
                 for k, (i, j, l) in enumerate(_TRIPLES)]
        return torch.stack(rows)

    def from_sums(self, acc, nsamples, ppc, cells):
        """DSMC2LB: populations [q, n] of the listed cells from their cumulative sums."""
        s = acc[cells]
        n = s[:, 0]
        rho, m = n / (nsamples * ppc), s / n[:, None]
        u = [m[:, 1 + i] for i in range(3)]
        a = [rho] + [rho * v for v in u]
        a += [rho * (m[:, 4 + k] - float(i == j)) for k, (i, j) in enumerate(_PAIRS)]
        a += [rho * (m[:, 10 + k] - u[i] * float(j == l) - u[j] * float(i == l) - u[l] * float(i == j))
              for k, (i, j, l) in enumerate(_TRIPLES)]
        return self.w[:, None] * (self.her @ torch.stack(a))


def _cell_of(case, nodes):
    nx, r = case["ncx"] * case["lb_ratio"], case["lb_ratio"]
    nodes = nodes.long()
    return (nodes // nx // r) * case["ncx"] + (nodes % nx) // r


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("lbm", "gradient", "mappings"):
        return None
    lb = _LB(case)
    nx, ny, nz, _, _ = _params(case)
    shape = (case["lattice"], nz, ny, nx) if case["ncz"] >= 2 else (case["lattice"], ny, nx)
    f = _populations(case, seed).double().view(lb.q, lb.n)
    if kind == "lbm":
        for _ in range(case["nsteps"]):
            f = lb.step(f)
        return f.view(shape)
    acc, ns = _sums(case, seed)
    if kind == "mappings":
        nodes, cells = _strip_nodes(case)
        at = nodes.long()
        f[:, at] = lb.from_sums(acc, ns, case["ppc"], _cell_of(case, nodes))
        g4 = f.view(lb.q, case["ncy"], case["lb_ratio"], case["ncx"], case["lb_ratio"]).mean((2, 4))
        c = lb.grad_coefficients(g4.reshape(lb.q, -1)[:, cells.long()])
        a = c[4:] if lb.q == 39 else torch.cat([c[4:10], torch.zeros_like(c[10:])])
        big = a.abs().max(0).values
        coef = torch.cat([a, c[1:4], (1.0 + 30.0 * big)[None]]).t().contiguous()
        return dict(f=f.view(shape), rho=c[0], coefficients=coef, counts=None, particles=None)
    # the states of the forward steps are kept, and the steps differentiated one at a time in reverse
    g, tau, nodes, targets = _node_params(case, seed)
    g, tau, targets = g.double(), tau.double(), targets.double()
    at = nodes.long()
    if case["coupled"]:
        d2l = _strip_nodes(case)[0]
        cells = _cell_of(case, d2l)
        acc = acc.requires_grad_(True)
        mapped = lb.from_sums(acc, ns, case["ppc"], cells)
        f[:, d2l.long()] = mapped.detach()
    states = [f]
    for _ in range(case["nsteps"]):
        states.append(lb.step(states[-1], g, tau))
    last = states[-1].requires_grad_(True)
    loss = ((lb.grad_coefficients(last[:, at]).t() - targets) ** 2).sum()
    lam, = torch.autograd.grad(loss, last)
    gg, gt = torch.zeros_like(g), torch.zeros_like(tau)
    for k in reversed(range(case["nsteps"])):
        s, a, b = (v.detach().clone().requires_grad_(True) for v in (states[k], g, tau))
        lam, da, db = torch.autograd.grad(lb.step(s, a, b), (s, a, b), lam)
        gg += da
        gt += db
    out = dict(loss=loss.detach(), g=gg, tau=gt)
    if case["coupled"]:
        # the mapping replaced the listed nodes: their adjoint goes to the sums of the cells, at a
        # fixed sample count
        ga, = torch.autograd.grad(mapped, acc, lam[:, d2l.long()])
        lam[:, d2l.long()] = 0.0
        out["acc"] = ga
    out["f0"] = lam.view(shape)
    return out
