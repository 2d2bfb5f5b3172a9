"""DSMC2LB takes consecutive list entries of one cell together (two nodes per cell and axis): lists in
which entries of one cell do not follow one another, of odd length, with an index out of range
between them, give every node exactly the populations that a list of that node alone gives."""
import numpy as np
import pytest

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
    a, b = B.Hybrid(cfg), B.Hybrid(cfg)
    for h in (a, b):
        h.dsmc_step(2)
    nn = int(a.d["nnodes"])
    nodes = np.arange(nn, dtype=np.int32)
    if order == "shuffled":
        nodes = np.random.default_rng(2).permutation(nodes).astype(np.int32)
    elif order == "single":
        nodes = nodes[33:34]
    elif order == "odd":
        nodes = nodes[1:nn - 4]
        nodes[10] = nn + 3  # out of range: skipped and flagged, the entry after it still mapped
    dev = torch.from_numpy(nodes.copy()).cuda()
    a.map_dsmc_to_lbm(dev)
    for k in range(len(nodes)):
        b.map_dsmc_to_lbm(dev[k:k + 1])
    a.sync()
    b.sync()
    assert torch.equal(a.f(), b.f())
    assert a.sync_status() == b.sync_status()
    assert bool(a.sync_status()[1] & B.ST_BAD_INPUT) == (order == "odd")
    a.close()
    b.close()
