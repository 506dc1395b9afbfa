"""The coarsest GEMV launched beside the restriction before it and by itself (the choice
depends on how many of its CTAs fit): the iterates of the cooperative coarse cycle, which
has no such launch, bit for bit.

Blocks of 4^3: 3645 unknowns behind 729 parents (fits), 4000 behind 1000 (does not), 256
behind 64 (fits; with four right-hand sides too), 384 with 24 per parent."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2403_19342_gb300 as p
    return p


@pytest.mark.parametrize("N,n_eig", [(72, (4, 5)), (80, (4, 4)), (32, (4, 4)), (32, (12, 6))])
@pytest.mark.parametrize("n_rhs", [1, 4])
def test_same_bits_as_the_cooperative_cycle(pkg, N, n_eig, n_rhs):
    g = torch.Generator(device="cuda").manual_seed(N)
    shape = (N, N, N)
    kappa = torch.exp(torch.randn(shape, dtype=torch.float64, device="cuda", generator=g))
    F = torch.randn((n_rhs,) + shape, dtype=torch.float64, device="cuda", generator=g)
    F -= F.mean(dim=(1, 2, 3), keepdim=True)
    S = pkg.Solver(kappa, pkg.Options(n_levels=3, block=(4, 4, 4), ratio=[(2, 2, 2)], n_eig=list(n_eig), eig_tol=1e-6,
                                      precision=pkg.MIXED), n_rhs=n_rhs + 1)
    out = []
    for form in (0, 2):
        pkg.msmg_set_tuning(S.ctx, (0, 0, form, form))
        x, info, _ = S.solve(F if n_rhs > 1 else F[0].contiguous(), rtol=1e-8, max_iter=100)
        infos = info if isinstance(info, list) else [info]
        assert all(i["converged"] for i in infos)
        out.append((x, [i["iterations"] for i in infos]))
    S.close()
    assert torch.equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]
