"""DSMC2LB takes two entries of one cell together where they are neighbours along an axis: lists in rows,
shifted by one, along the other axes, shuffled, of odd length, with repeated nodes and with indices out
of range (among them the one that would be the neighbour above a 2D lattice), of fewer and of more
entries than the GPU has warps, give every node exactly the populations that lists of one entry give."""
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


def _order(nodes, nx, plane, order):
    if order == "rows":
        return nodes
    if order == "shifted":
        return nodes[1:]
    if order == "columns":
        return nodes.reshape(-1, plane // nx, nx).transpose(0, 2, 1).reshape(-1)
    if order == "layers":
        return nodes.reshape(-1, plane).T.reshape(-1)
    if order == "shuffled":
        return np.random.default_rng(3).permutation(nodes)
    out = nodes[:len(nodes) - 3].copy()  # "odd": of odd length, with repeats and invalid entries
    out[6:8] = out[4]
    out[11] = out[10] + plane * 64  # above any lattice here
    out[20] = -1
    out[31] = -7
    out[40:42] = (nodes[-plane], nodes[-plane] + plane)  # above the last layer
    return out


@pytest.mark.parametrize("real_bytes,lattice,ncz,ncx,ncy,lb_ratio", [
    (4, 39, 0, 20, 30, 2), (8, 39, 0, 20, 30, 2), (4, 19, 4, 10, 12, 2), (8, 19, 3, 7, 13, 2), (4, 39, 0, 64, 60, 2),
    (4, 39, 0, 40, 40, 1)])
@pytest.mark.parametrize("order", ["rows", "shifted", "columns", "layers", "shuffled", "odd"])
def test_lists_equal_single_entries(real_bytes, lattice, ncz, ncx, ncy, lb_ratio, order):
    cfg = W.config(ncx=ncx, ncy=ncy, ncz=ncz, ppc=20, lb_ratio=lb_ratio, real_bytes=real_bytes, lattice=lattice, seed=4)
    a, b = B.Hybrid(cfg), B.Hybrid(cfg)
    for h in (a, b):
        h.dsmc_step(2)
    nx, ny, nn = int(a.d["nx"]), int(a.d["ny"]), int(a.d["nnodes"])
    nodes = _order(np.arange(nn, dtype=np.int32), nx, nx * ny, order).astype(np.int32)
    dev = torch.from_numpy(np.ascontiguousarray(nodes)).cuda()
    a.map_dsmc_to_lbm(dev)
    for k in range(len(nodes)):
        b.map_dsmc_to_lbm(dev[k:k + 1])
    assert a.sync_status() == b.sync_status()
    assert bool(a.sync_status()[1] & B.ST_BAD_INPUT) == (order == "odd")
    assert torch.equal(a.f(), b.f())
    a.close()
    b.close()


def test_lists_of_a_slab_skip_its_ghost_rows():
    cfg = W.config(ncx=24, ncy=20, ppc=20, lb_ratio=2, seed=4, ncy_global=40, y0=10)
    a, b = B.Hybrid(cfg), B.Hybrid(cfg)
    for h in (a, b):
        h.dsmc_move()
        h.dsmc_merge()
        h.dsmc_collide()
    nodes = np.arange(int(a.d["nnodes"]), dtype=np.int32)
    dev = torch.from_numpy(nodes).cuda()
    a.map_dsmc_to_lbm(dev)
    for k in range(len(nodes)):
        b.map_dsmc_to_lbm(dev[k:k + 1])
    assert a.sync_status() == b.sync_status() and a.sync_status()[1] & B.ST_BAD_INPUT
    assert torch.equal(a.f(), b.f())
    a.close()
    b.close()
