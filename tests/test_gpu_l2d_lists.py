"""LB2DSMC takes its block shape from the list's length: lists on both sides of every line give each cell
the particles that lists of at most 100 cells, one shape in every precision and lattice, give, bit for
bit, with an index out of range flagged."""
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


@pytest.mark.parametrize("noisy", [False, True])
@pytest.mark.parametrize("real_bytes,lattice,ncz,lb_ratio", [
    (4, 39, 0, 2), (8, 39, 0, 1), (4, 19, 0, 1), (8, 19, 0, 2), (4, 19, 3, 1), (8, 39, 2, 2)])
def test_long_lists_equal_short_ones(real_bytes, lattice, ncz, lb_ratio, noisy):
    ncx, ncy = (42, 30) if not ncz else (21, 30)
    cfg = W.config(ncx=ncx, ncy=ncy, ncz=ncz, ppc=30, lb_ratio=lb_ratio, real_bytes=real_bytes, lattice=lattice, seed=9)
    a, b = B.Hybrid(cfg), B.Hybrid(cfg)
    ncells, nn = int(a.L.ncells), int(a.d["nnodes"])
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for h in (a, b):
        h.dsmc_step(3)
        if noisy:  # populations of three samples: most first trials are rejected
            h.map_dsmc_to_lbm(torch.arange(nn, dtype=torch.int32, device="cuda"))
    rng = np.random.default_rng(1)
    for n in (sms, sms + 1, 2 * sms, 2 * sms + 1, 4 * sms + 1, 5 * sms, ncells):
        cells = rng.permutation(ncells)[:n].astype(np.int32)
        cells[n // 2] = ncells + 5
        dev = torch.from_numpy(cells).cuda()
        a.map_lbm_to_dsmc(dev)
        for k in range(0, n, 100):
            b.map_lbm_to_dsmc(dev[k:k + 100])
        assert a.sync_status() == b.sync_status() and a.sync_status()[1] & B.ST_BAD_INPUT
        assert a.counters() == b.counters()
        assert torch.equal(a.counts(), b.counts())
        pa, pb = a.particles(), b.particles()
        for k, v in pa.items():
            assert torch.equal(v, pb[k]), (n, k)
    a.close()
    b.close()
