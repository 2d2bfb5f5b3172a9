"""DSMC2LB takes consecutive list entries of one cell together (two nodes per cell and axis): lists in
which entries of one cell do not follow one another, of odd length, with repeated cells, an index
out of range and a cell without samples between them give the populations the oracle gives."""
import numpy as np
import pytest

from conftest import lb_err

from oracle import oracle as O
from paper_1512_08042_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU-only machines, never run there
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1512_08042_gb300 import binding as B  # noqa: E402
from paper_1512_08042_gb300 import build as BUILD  # noqa: E402

BUILD.build()


@pytest.mark.parametrize("real_bytes,lattice,eq", [(4, 39, 0), (8, 39, 0), (4, 19, 1)])
@pytest.mark.parametrize("order", ["rows", "shuffled", "single", "odd"])
def test_map_dsmc_to_lbm_lists(real_bytes, lattice, eq, order):
    cfg = W.config(ncx=7, ncy=5, ppc=20, lb_ratio=2, real_bytes=real_bytes, lattice=lattice, d2l_mode=eq, seed=4)
    h, o = B.Hybrid(cfg), O.Oracle(cfg)
    h.dsmc_step(2)
    o.dsmc_step(2)
    nn = int(h.d["nnodes"])
    nodes = np.arange(nn, dtype=np.int32)
    if order == "shuffled":
        nodes = np.random.default_rng(2).permutation(nodes).astype(np.int32)
    elif order == "single":
        nodes = nodes[33:34]
    elif order == "odd":
        nodes = nodes[1:nn - 4]
        nodes[10] = nn + 3  # out of range: skipped and flagged, the entry after it still mapped
    h.map_dsmc_to_lbm(torch.from_numpy(nodes.copy()).cuda())
    o.map_dsmc_to_lbm(nodes)
    h.sync()
    w = O.lattice(lattice)[1]
    # the tolerance of the mapping's parity test: FP64 coefficients, the series in the state
    # precision
    assert lb_err(h.f().cpu().numpy(), o.f(), w) < (2e-6 if real_bytes == 4 else 1e-12)
    rc, bits = h.sync_status()
    assert bool(bits & B.ST_BAD_INPUT) == (order == "odd")
    h.close()
