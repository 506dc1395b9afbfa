"""The divergence of msmg_velocity divides by the cell sizes through a reciprocal and a
correction: the quotients are IEEE division's, bit for bit.

The balance ||div v - b|| is exactly zero when b holds the divergence that plain FP64
division gives for the returned face velocities.  b is the source itself where the cell term
is zero or the pressure is (cell 0 here; the term keeps the system non-singular).  The
pressure's steps are powers of two, so that a face velocity is a product the compiler may
fuse into the difference without changing it."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2403_19342_gb300 as p
    return p


@pytest.mark.parametrize("h", [(1.0 / 48, 1.0 / 40, 1.0 / 36), (20.0, 10.0, 2.0), (0.3, 7e-3, 1.1e5),
                               (1.9999999999999998, 1.0000000000000002, 0.1)])
@pytest.mark.parametrize("seed", [0, 1])
def test_divergence_has_the_bits_of_division(pkg, h, seed):
    shape = (36, 40, 48)
    g = torch.Generator(device="cuda").manual_seed(seed)
    rnd = lambda *s: torch.randn(*s, dtype=torch.float64, device="cuda", generator=g)
    W = torch.zeros(shape, dtype=torch.float64, device="cuda")
    W[0, 0, 0] = 1.0
    S = pkg.Solver(torch.exp(2.0 * rnd(3, *shape)),
                   pkg.Options(n_levels=2, block=(4, 4, 4), ratio=[], n_eig=[1], eig_tol=1e-6, cell_diag=W), h=h)
    p = torch.zeros_like(W)
    for ax in range(3):
        step = torch.sign(rnd(shape[ax])) * 2.0 ** torch.randint(-3, 4, (shape[ax],), device="cuda", generator=g).double()
        step[0] = 0.0
        view = [1, 1, 1]
        view[ax] = shape[ax]
        p = p + torch.cumsum(step, 0).view(view)
    v, _ = S.velocity(p, torch.zeros_like(p))
    div = torch.zeros_like(p)
    for d in range(3):
        ax = 2 - d                                # +d faces; no flow through the boundary
        vm = torch.zeros_like(p)
        vm.narrow(ax, 1, shape[ax] - 1).copy_(v[d].narrow(ax, 0, shape[ax] - 1))
        div = div + (v[d] - vm) / torch.full_like(p, h[d])   # (by a Python scalar PyTorch multiplies by 1 / h)
    _, bal = S.velocity(p, div)
    S.close()
    assert bal[1] > 0.0 and bal[0] == 0.0
