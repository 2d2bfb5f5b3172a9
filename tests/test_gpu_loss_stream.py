"""The differentiated LBM runs on its context's stream: inputs that the caller's stream is still to
write are waited for."""
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


def test_interface_loss_waits_for_inputs_of_the_callers_stream():
    cfg = W.config(ncx=16, ncy=8, ppc=10, lb_ratio=2, real_bytes=8, kn=0.3, ma=0.5, seed=3)
    h = B.Hybrid(cfg)
    n = int(h.d["nnodes"])
    base = torch.from_numpy(W.gen_populations(O.lattice(39)[1], n, seed=1)).cuda().view(h.f().shape)
    g = torch.full((n,), float(h.d["g_step"]), dtype=h.real, device="cuda")
    tau = torch.full((n,), float(h.d["tau"]), dtype=h.real, device="cuda")
    nodes = torch.arange(40, dtype=torch.int32, device="cuda")
    targets = torch.from_numpy(0.1 * np.ones((40, 20))).cuda()
    f = base * 1.01
    torch.cuda.synchronize()
    want = B.interface_loss(h, g, tau, f, nodes, targets, 3).item()
    f.zero_()
    torch.cuda.synchronize()
    work = torch.zeros(1 << 28, device="cuda")  # a few milliseconds of writes on the caller's stream
    for _ in range(20):
        work.add_(1.0)
    f.copy_(base).mul_(1.01)
    assert B.interface_loss(h, g, tau, f, nodes, targets, 3).item() == want
    h.close()
