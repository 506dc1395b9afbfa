"""Coarse-level steps of the V-cycle at the sizes where their code paths change: block sizes
with and without unrolled loops (4, 6, 7, 8; 3, 5, 9), basis widths that are not a multiple
of the four sums taken together and wider than the eight values a thread holds, levels with
few parents (four threads per row) and with many right-hand sides (one).

The fused coarse cycle forms every sum in the same order: equal bits.  Against the oracle's
V-cycle, FP64 rounding: 1e-9."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2403_19342_gb300 as p
    return p


@pytest.mark.parametrize("n_eig,ratio", [((4, 4), (2, 2, 2)), ((5, 9), (2, 2, 2)), ((6, 3), (2, 2, 2)),
                                         ((7, 11), (2, 1, 2)), ((8, 2), (1, 2, 2)), ((9, 1), (2, 2, 2)),
                                         ((3, 10), (4, 2, 2)), ((4, 6, 5), (2, 2, 2))])
def test_forms_agree(pkg, n_eig, ratio):
    shape = (32, 32, 32)
    rng = np.random.default_rng(sum(n_eig))
    kappa = np.exp(1.5 * rng.standard_normal(shape))
    nl = len(n_eig) + 1
    kw = dict(n_levels=nl, block=(4, 4, 4), ratio=[ratio] + [(2, 2, 2)] * (nl - 3), n_eig=list(n_eig))
    H = oracle.setup(kappa, (1 / 32,) * 3, oracle.Options(nu=[1] * (nl - 1), **kw))
    S = pkg.Solver(torch.tensor(kappa, device="cuda"), pkg.Options(eig_tol=1e-10, **kw), n_rhs=24)
    assert S.import_bases(H.basis[:nl - 1]) == 0
    F = rng.standard_normal((24,) + shape)
    F -= F.mean(axis=(1, 2, 3), keepdims=True)
    Ft = torch.tensor(F, device="cuda")
    z, x = [], []
    for form in (0, 2):
        pkg.msmg_set_tuning(S.ctx, (0, 0, form, form))
        z.append(S.apply_precond(Ft[0].contiguous()).cpu().numpy())
        x.append(S.solve(Ft, rtol=1e-8, max_iter=100)[0].clone())
    assert np.array_equal(z[0], z[1])
    assert torch.equal(x[0], x[1])
    one = S.solve(Ft[5].contiguous(), rtol=1e-8, max_iter=100)[0]
    assert torch.equal(one.reshape(-1), x[0][5].reshape(-1))
    ref = oracle.vcycle(H, F[0].ravel())
    assert np.linalg.norm(z[0].ravel() - ref) <= 1e-9 * np.linalg.norm(ref)
    S.close()
