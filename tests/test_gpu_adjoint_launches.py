"""The one-call sweeps of the differentiated LBM overlap their launches (in FP64 only up to one block per
SM): on lattices on both sides of that line they give what the single step calls give, bit for bit."""
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


@pytest.mark.parametrize("real_bytes", [4, 8])
@pytest.mark.parametrize("ncx,ncy,lattice", [(64, 300, 39), (64, 320, 39), (33, 640, 19), (40, 16, 39)])
def test_sweeps_equal_single_steps(ncx, ncy, lattice, real_bytes):
    h = B.Hybrid(W.config(ncx=ncx, ncy=ncy, ppc=1, real_bytes=real_bytes, lattice=lattice, kn=0.2, seed=2))
    n, steps = int(h.d["nnodes"]), 6
    rng = np.random.default_rng(ncx)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(h.real).cuda()  # noqa: E731
    f0 = dev(W.gen_populations(O.lattice(lattice)[1], n, seed=3)).view(h.f().shape)
    g = dev(h.d["g_step"] * (1 + 0.3 * rng.standard_normal(n)))
    tau = dev(h.d["tau"] * (1 + 0.1 * rng.standard_normal(n)))
    lam_T = dev(rng.standard_normal(f0.numel())).view(f0.shape)
    wall = torch.zeros(h.wall_scratch_size(), dtype=h.real, device="cuda")
    torch.cuda.synchronize()
    # forward: every state, by single steps and by one call
    states = [f0.clone()]
    for _ in range(steps):
        nxt = torch.empty_like(f0)
        h.lbm_step_nodes(states[-1], nxt, g, tau)
        states.append(nxt)
    a, b = f0.clone(), torch.empty_like(f0)
    ck = torch.empty((steps - 1,) + tuple(f0.shape), dtype=h.real, device="cuda")
    torch.cuda.synchronize()
    fT = h.lbm_steps_nodes(a, b, g, tau, steps, 1, ck)
    h.sync()
    assert torch.equal(fT, states[-1])
    for k in range(1, steps):
        assert torch.equal(ck[k - 1], states[k]), k
    # adjoint: from the last state back
    one = [torch.zeros_like(g), torch.zeros_like(tau)]
    lam, other = lam_T.clone(), torch.empty_like(lam_T)
    torch.cuda.synchronize()
    for k in reversed(range(steps)):
        h.lbm_adjoint_step(states[k], lam, other, g, tau, one[0], one[1], wall)
        lam, other = other, lam
    seg = [torch.zeros_like(g), torch.zeros_like(tau)]
    x, y = lam_T.clone(), torch.empty_like(lam_T)
    scratch = torch.empty((steps - 1,) + tuple(f0.shape), dtype=h.real, device="cuda")
    torch.cuda.synchronize()
    out = h.lbm_adjoint_segment(f0, scratch, steps, x, y, g, tau, seg[0], seg[1], wall)
    h.sync()
    assert torch.equal(out, lam)
    assert torch.equal(seg[0], one[0]) and torch.equal(seg[1], one[1])
    h.close()
