"""The collide's pools of a block share one SM's memory: bins and shapes whose full pools exceed it run
with smaller ones, and warps whose cells do not fit theirs take them one at a time. Both block
shapes, with crowded cells that overflow any pool, against the oracle (events and counts equal,
particles to 1e-5 in FP32 and 1e-12 in FP64, the tolerance of the collide's other edges); the tuners and
the batch at such sizes."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1512_08042_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU-only machines, never run there
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1512_08042_gb300 import binding as B  # noqa: E402
from paper_1512_08042_gb300 import build as BUILD  # noqa: E402

BUILD.build()

# (real bytes, layers, particles per cell, capacity factor): eight pools of four cells exceed an SM's
# memory in all but the first two, four of them in the last
SIZES = [(4, 0, 50, 2.5), (4, 3, 50, 2.5), (8, 3, 100, 2.5), (8, 0, 140, 1.6), (4, 3, 190, 1.25), (8, 3, 240, 1.05)]


@pytest.mark.parametrize("warps", [4, 8])
@pytest.mark.parametrize("size", range(len(SIZES)))
def test_crowded_cells_in_both_shapes_match_the_oracle(size, warps):
    real_bytes, ncz, ppc, cf = SIZES[size]
    cfg = W.config(ncx=7, ncy=5, ncz=ncz, ppc=ppc, capacity_factor=cf, kn=0.1, real_bytes=real_bytes, seed=31 + size)
    h, o = B.Hybrid(cfg), O.Oracle(cfg)
    ncells, room = int(h.L.ncells), int(h.L.bin) - 16
    # cells filled almost to their bins beside ordinary, nearly empty and empty ones
    counts = np.resize(np.array([room, room, room, room - 3, ppc // 2, 1, 0, ppc // 3, ppc // 2, ppc // 4, 2]), ncells)
    rng = np.random.default_rng(7 + size)
    cell = np.repeat(np.arange(ncells), counts)
    n = cell.size
    real = np.float32 if real_bytes == 4 else np.float64
    x = (cell % 7 + 0.1 + 0.8 * rng.random(n)).astype(real)
    y = (cell // 7 % 5 + 0.1 + 0.8 * rng.random(n)).astype(real)
    z = (cell // 35 + 0.1 + 0.8 * rng.random(n)).astype(real) if ncz else None
    v = [(0.03 * rng.standard_normal(n)).astype(real) for _ in range(3)]  # few leave their cells
    cs = np.zeros(ncells + 1, np.uint32)
    cs[1:] = np.cumsum(counts)
    h.set_fuse("always")
    h.set_collide_block(warps)
    h.load_particles(x, y, *v, cs, z=z)
    o.set_particles(x, y, *v, cs, z=z)
    h.dsmc_step(3)  # two fused passes and a plain collide
    o.dsmc_step(3)
    assert h.sync_status()[1] == 0
    hc, oc = h.counters(), o.counters()
    for k in ("candidates", "collisions", "wall_hits"):
        assert hc[k] == oc[k], k
    assert np.array_equal(h.cell_start().cpu().numpy().astype(np.uint32), o.get(O.A_CELL_START))
    tol = 1e-5 if real_bytes == 4 else 1e-12
    gp, op = h.particles(), o.particles()
    for k in op:
        assert np.allclose(gp[k].cpu().numpy(), op[k], rtol=tol, atol=tol), k
    h.close()


def test_tuner_takes_both_shapes_where_full_pools_do_not_fit():
    cfg = W.config(ncx=8, ncy=6, ncz=3, ppc=100, real_bytes=8, kn=0.1, seed=5)
    a, b = B.Hybrid(cfg), B.Hybrid(cfg)
    w, fuse = a.tune_collide()
    assert w in (4, 8) and a.collide_block() == w and fuse in ("always", "never")
    b.hybrid_step(nsteps=192)
    a.sync()
    b.sync()
    for k, v in a.particles().items():
        assert torch.equal(v, b.particles()[k]), k
    a.close()
    b.close()


def test_batch_runs_where_full_pools_do_not_fit():
    cfgs = [W.config(ncx=12, ncy=2, ppc=140, capacity_factor=1.6, real_bytes=8, kn=0.1, seed=1),
            W.config(ncx=9, ncy=3, ppc=30, real_bytes=8, kn=0.05, seed=2)]
    sites = [W.coupling_sites(c, strip_cells=1) for c in cfgs]
    nodes, cells = [s[0] for s in sites], [s[1] for s in sites]
    b = B.Batch(cfgs)
    assert b.blocks()["collide"] == 256
    b.hybrid_step(nodes, cells, nsteps=3)
    b.tune(nodes, cells)
    b.sync()
    for g, c, dn, dc in zip(b.replicas, cfgs, nodes, cells):
        h = B.Hybrid(c)
        h.hybrid_step(torch.from_numpy(dn).cuda(), torch.from_numpy(dc).cuda(), nsteps=3 + 77)
        h.sync()
        for k, v in h.particles().items():
            assert torch.equal(v, g.particles()[k]), k
        h.close()
    b.close()
