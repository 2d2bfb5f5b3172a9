"""The adjoint LB step needs the nodes next to a wall (three in D3Q39) in one warp. Rows whose width is
a little above a multiple of 32 with more segments than half a segment has nodes (962, 993, 994, 1025,
1026): the FP64 gradient of a loss next to the walls against central differences along random
directions next to the walls, at the tolerance of the other rows' check. The differences' error
is below it: their truncation is O(scale^2) and their rounding about 1e-15 / scale of the loss, which
is of the size of the gradient's terms."""
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


@pytest.mark.parametrize("ncx,lb_ratio,ncy,ncz,lattice", [
    (481, 2, 2, 0, 39), (993, 1, 3, 0, 39), (497, 2, 2, 0, 39), (1025, 1, 3, 0, 39), (513, 2, 2, 0, 39),
    (962, 1, 3, 2, 39), (993, 1, 3, 0, 19)])
def test_gradient_next_to_the_walls_of_wide_rows(ncx, lb_ratio, ncy, ncz, lattice):
    check_gradient_next_to_the_walls(ncx, lb_ratio, ncy, ncz, lattice)


@pytest.mark.parametrize("ncx,lb_ratio,ncy,ncz,lattice", [
    (6, 1, 22, 0, 39), (7, 1, 19, 0, 39), (12, 1, 7, 2, 39), (20, 1, 13, 0, 19), (25, 1, 6, 0, 39),
    (33, 1, 620, 0, 39), (21, 2, 310, 0, 19)])
def test_gradient_of_whole_rows_in_a_block(ncx, lb_ratio, ncy, ncz, lattice):
    # narrow rows go whole to a block, whose last one may have fewer (22 rows of 6 nodes: 21 and 1);
    # rows of 33 and 42 nodes only on lattices this large
    check_gradient_next_to_the_walls(ncx, lb_ratio, ncy, ncz, lattice)


def check_gradient_next_to_the_walls(ncx, lb_ratio, ncy, ncz, lattice):
    cfg = W.config(ncx=ncx, ncy=ncy, ncz=ncz, ppc=1, lb_ratio=lb_ratio, real_bytes=8, lattice=lattice, kn=0.3, ma=0.5,
                   seed=3)
    h = B.Hybrid(cfg)
    n, q, nx = int(h.d["nnodes"]), int(h.d["q"]), int(h.d["nx"])
    rng = np.random.default_rng(ncx)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    f0 = dev(W.gen_populations(O.lattice(lattice)[1], n, seed=ncx + 100)).view(h.f().shape)
    g = dev(h.d["g_step"] * (1 + 0.3 * rng.standard_normal(n)))
    tau = dev(h.d["tau"] * (1 + 0.1 * rng.standard_normal(n)))
    x = np.arange(n) % nx
    near = (x < 8) | (x >= nx - 8)
    nodes = dev(np.nonzero(near)[0][::3].astype(np.int32))
    targets = dev(0.1 * rng.standard_normal((nodes.numel(), 20)))

    def loss(f, gg, tt):
        return B.interface_loss(h, gg, tt, f, nodes, targets, 4, 3)

    leaves = [t.clone().requires_grad_(True) for t in (f0, g, tau)]
    grads = torch.autograd.grad(loss(*leaves), leaves)
    for i, scale in enumerate((1e-6, 1e-5, 1e-5)):
        p = [f0, g, tau]
        mask = np.tile(near, p[i].numel() // n)
        v = dev(mask * rng.standard_normal(p[i].numel())).view(p[i].shape) * p[i].abs()
        up, dn = list(p), list(p)
        up[i], dn[i] = p[i] + scale * v, p[i] - scale * v
        want = float((loss(*up) - loss(*dn)) / (2 * scale))
        got = float((grads[i] * v).sum())
        size = float((grads[i] * v).abs().sum())
        assert abs(got - want) <= 1e-6 * size, (i, got, want, size)
    h.close()
