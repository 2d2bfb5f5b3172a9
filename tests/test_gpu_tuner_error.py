"""A tuner that fails leaves the shapes and modes it found: contexts on the default stream, which
cannot replay graphs, so that the tuner's first timed call is refused."""
import pytest

from paper_1512_08042_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU-only machines, never run there
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1512_08042_gb300 import binding as B  # noqa: E402
from paper_1512_08042_gb300 import build as BUILD  # noqa: E402

BUILD.build()


def _fused_passes(h):
    """Fused passes of a three-step call (none in two-pass mode)."""
    h.profile("fused")
    h.dsmc_step(3)
    h.profile_harvest()
    n = h.profile_read()[1]
    h.profile(-1)
    return n


def test_collide_tuner_restores_the_shape_and_the_mode():
    h = B.Hybrid(W.config(ncx=8, ncy=6, ppc=20, seed=1), stream=torch.cuda.default_stream())
    assert h.collide_block() == 4
    h.set_fuse("never")
    with pytest.raises(B.HybError):
        h.tune_collide()
    assert h.collide_block() == 4
    assert _fused_passes(h) == 0
    h.set_fuse("always")
    assert _fused_passes(h) == 2
    h.close()


def test_batch_tuner_restores_the_block_sizes():
    cfgs = [W.config(ncx=12, ncy=1, ppc=20, seed=1), W.config(ncx=16, ncy=1, ppc=30, seed=2)]
    sites = [W.coupling_sites(c) for c in cfgs]
    b = B.Batch(cfgs, stream=torch.cuda.default_stream())
    before = b.blocks()
    with pytest.raises(B.HybError):
        b.tune([s[0] for s in sites], [s[1] for s in sites])
    assert b.blocks() == before
    b.close()
