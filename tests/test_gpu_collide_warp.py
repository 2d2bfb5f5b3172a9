"""The collide at the edges of its warp-sized work: a warp takes four cells, keeps the first 64
arrivals of a cell in registers (FP32), settles eight NTC candidates of a cell at a time and
falls back to one cell at a time when the four cells' particles do not fit its pool. Integers,
pairs and particles against the oracle as in the parity tests (FP32 bit for bit up to the
libm-free series, FP64 to 1e-12)."""
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

# (cells across, along, ppc, Kn, counts per cell): few particles and many candidates, so that
# most windows hold candidates of one particle; one particle per cell; counts on both sides of
# the 64 held arrivals; a crowd that overflows the pool of its warp; cells that end inside a warp
CASES = [
    (7, 3, 3, 0.01, [2, 3, 2, 4, 3, 0, 2]),
    (6, 5, 4, 0.05, [1, 1, 0, 1, 9]),
    (13, 5, 60, 0.05, [63, 64, 65, 72, 60, 31, 33]),
    (6, 7, 40, 0.02, [96, 96, 96, 90, 1, 0, 5, 2]),
    (9, 3, 100, 0.01, [100, 130, 90, 200, 256, 64]),
]


@pytest.mark.parametrize("real_bytes", [4, 8])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_collide_matches_the_oracle_at_the_edges_of_a_warps_work(case, real_bytes):
    ncx, ncy, ppc, kn, pattern = CASES[case]
    cfg = W.config(ncx=ncx, ncy=ncy, ppc=ppc, kn=kn, real_bytes=real_bytes, seed=17 + case, capacity_factor=2.5)
    ncells = ncx * ncy
    counts = np.resize(np.array(pattern), ncells)
    rng = np.random.default_rng(5 + case)
    cell = np.repeat(np.arange(ncells), counts)
    n = cell.size
    real = np.float32 if real_bytes == 4 else np.float64
    x = (cell % ncx + 0.02 + 0.96 * rng.random(n)).astype(real)
    y = (cell // ncx + 0.02 + 0.96 * rng.random(n)).astype(real)
    v = [(0.3 * rng.standard_normal(n)).astype(real) for _ in range(3)]  # few leave their cells
    cs = np.zeros(ncells + 1, np.uint32)
    cs[1:] = np.cumsum(counts)
    h, o = B.Hybrid(cfg), O.Oracle(cfg)
    h.set_fuse("always")
    h.load_particles(x, y, *v, cs)
    o.set_particles(x, y, *v, cs)
    h.dsmc_step(1)
    o.dsmc_step(1)
    h.dsmc_step(2)  # a fused pass between
    o.dsmc_step(2)
    hc, oc = h.counters(), o.counters()
    for k in ("candidates", "collisions", "wall_hits"):
        assert hc[k] == oc[k], k
    assert np.array_equal(h.cell_start().cpu().numpy().astype(np.uint32), o.get(O.A_CELL_START))
    tol = 1e-5 if real_bytes == 4 else 1e-12
    gp, op = h.particles(), o.particles()
    for k in op:
        g = gp[k].cpu().numpy()
        assert np.allclose(g, op[k], rtol=tol, atol=tol), k
    assert np.allclose(h.crmax().cpu().numpy(), o.get(O.A_CRMAX), rtol=tol)
    assert oc["candidates"] > 0 or case == 1
