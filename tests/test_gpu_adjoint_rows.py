"""The adjoint LB step cuts a row of nodes into warp-sized segments and the warp next to a wall
sums that row's wall adjoint: rows of one and several segments, of full and partial ones, 2D and
3D. The FP64 gradient against central differences along random directions in the populations,
forces and relaxation times; the same tolerance as the gradient checks against the oracle."""
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


@pytest.mark.parametrize("ncx,ncy,ncz,lattice", [(6, 5, 0, 39), (31, 4, 0, 39), (32, 4, 0, 39), (33, 4, 0, 39),
                                                 (65, 3, 0, 39), (40, 5, 0, 19), (34, 4, 3, 39), (6, 3, 2, 19)])
def test_gradient_along_random_directions(ncx, ncy, ncz, lattice):
    cfg = W.config(ncx=ncx, ncy=ncy, ncz=ncz, ppc=10, real_bytes=8, lattice=lattice, kn=0.3, ma=0.5, seed=3)
    h = B.Hybrid(cfg)
    n, q = int(h.d["nnodes"]), int(h.d["q"])
    rng = np.random.default_rng(ncx)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    _, w, _ = O.lattice(lattice)
    f0 = dev(W.gen_populations(w, n, seed=ncx + 100)).view(h.f().shape)
    g = dev(h.d["g_step"] * (1 + 0.3 * rng.standard_normal(n)))
    tau = dev(h.d["tau"] * (1 + 0.1 * rng.standard_normal(n)))
    nodes = torch.arange(0, n, 3, dtype=torch.int32, device="cuda")
    targets = dev(0.1 * rng.standard_normal((nodes.numel(), 20)))

    def loss(f, gg, tt):
        return B.interface_loss(h, gg, tt, f, nodes, targets, 4, 3)

    leaves = [t.clone().requires_grad_(True) for t in (f0, g, tau)]
    grads = torch.autograd.grad(loss(*leaves), leaves)
    for i, scale in enumerate((1e-6, 1e-5, 1e-5)):
        x = [f0, g, tau]
        v = dev(rng.standard_normal(x[i].numel())).view(x[i].shape) * x[i].abs()
        up, dn = list(x), list(x)
        up[i], dn[i] = x[i] + scale * v, x[i] - scale * v
        want = float((loss(*up) - loss(*dn)) / (2 * scale))
        got = float((grads[i] * v).sum())
        size = float((grads[i] * v).abs().sum())
        assert abs(got - want) <= 1e-6 * size, (i, got, want, size)
    h.close()
