"""Dense parts of the set-up at the edges of their blocks: the coarsest inverse (blocks of 32
pivots, tiles of 64, panels of 32 rows) and the coarse local eigenproblems (from 1 unknown to
96, where the work space no longer fits and Jacobi takes over; homogeneous fields with
multiple eigenvalues).

Tolerances: the V-cycle with the oracle's bases as the parity tests (1e-11, or ten times
eps cond of the coarsest operator); eigenvalues of matrices of norm at most 8 to 1e-12;
vectors orthonormal to 1e-12."""
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


@pytest.mark.parametrize("grid,L", [((2, 1, 1), 1), ((31, 1, 1), 1), ((4, 2, 1), 4), ((11, 3, 1), 1), ((4, 4, 4), 1),
                                    ((13, 5, 1), 1), ((4, 3, 2), 4), ((7, 6, 4), 1), ((5, 5, 5), 3)])
@pytest.mark.parametrize("wells", [False, True])
def test_coarsest_inverse(pkg, grid, L, wells):
    shape = tuple(2 * g for g in grid[::-1])
    rng = np.random.default_rng(sum(grid) + L)
    kappa = np.exp(2.0 * rng.standard_normal(shape))
    w = np.where(rng.uniform(size=shape) < 0.2, 10.0, 0.0) if wells else None
    if wells:
        w.flat[0] = 10.0
    oo = oracle.Options(n_levels=2, block=(2, 2, 2), ratio=[], n_eig=[L], nu=[1], cell_diag=w)
    h = tuple(1.0 / n for n in shape[::-1])
    H = oracle.setup(kappa, h, oo)
    S = pkg.Solver(torch.tensor(kappa, device="cuda"),
                   pkg.Options(n_levels=2, block=(2, 2, 2), ratio=[], n_eig=[L], eig_tol=1e-12,
                               cell_diag=None if w is None else torch.tensor(w, device="cuda")))
    assert S.import_bases([H.basis[0]]) == 0
    r = rng.standard_normal(shape)
    if not wells:
        r -= r.mean()
    z = S.apply_precond(torch.tensor(r, device="cuda")).cpu().numpy().ravel()
    zr = oracle.vcycle(H, r.ravel())
    ev = np.linalg.eigvalsh(H.A[-1].toarray())
    ev = ev[ev > 1e-12 * ev[-1]]
    slack = 10 * np.finfo(float).eps * ev[-1] / ev[0]
    assert np.linalg.norm(z - zr) <= max(1e-11, slack) * np.linalg.norm(zr)
    S.close()


@pytest.mark.parametrize("ratio,L,Ln", [((1, 1, 1), 1, 1), ((2, 1, 1), 1, 2), ((3, 1, 1), 1, 2), ((2, 2, 1), 3, 12),
                                        ((2, 2, 2), 4, 4), ((3, 3, 1), 5, 7), ((2, 2, 2), 6, 6), ((4, 2, 2), 4, 9),
                                        ((3, 5, 1), 4, 4), ((2, 2, 2), 11, 24), ((2, 2, 2), 12, 20)])
@pytest.mark.parametrize("homogeneous", [False, True])
def test_coarse_eigenpairs(pkg, ratio, L, Ln, homogeneous):
    block = (3, 3, 2)
    grid = (2 * ratio[0], ratio[1], ratio[2])
    shape = tuple(g * b for g, b in zip(grid, block))[::-1]
    rng = np.random.default_rng(L + Ln)
    kappa = np.ones(shape) if homogeneous else np.exp(1.5 * rng.standard_normal(shape))
    h = tuple(1.0 / n for n in shape[::-1])
    H = oracle.setup(kappa, h, oracle.Options(n_levels=3, block=block, ratio=[ratio], n_eig=[L, Ln], nu=[1, 1]))
    S = pkg.Solver(torch.tensor(kappa, device="cuda"),
                   pkg.Options(n_levels=3, block=block, ratio=[ratio], n_eig=[L, Ln], eig_tol=1e-12))
    assert S.setup_status == 0
    Psi, lam = (t.cpu().numpy() for t in S.export_basis(2))
    S.close()
    assert np.all(np.diff(lam, axis=1) >= -1e-12)
    for P in range(Psi.shape[0]):
        np.testing.assert_allclose(Psi[P] @ Psi[P].T, np.eye(Ln), rtol=0, atol=1e-12)
    # level 2's spectra depend on level 1's spans only, which a cluster at the cutoff leaves open
    lam_next, _, _ = oracle.level1_eigenpairs(H.T, H.S, block, min(L + 1, 18))
    if L == 18 or np.min(lam_next[:, min(L, 17)] - lam_next[:, L - 1]) > 1e-6:
        np.testing.assert_allclose(lam, H.lam[1], rtol=0, atol=1e-12)
