"""Level-2 local eigenpairs against LAPACK on the very matrices the set-up solves: the oracle
assembles each parent's matrix B^T A_P B (fine faces inside the parent only) from the bases
the GPU exported for level 1, so clusters at level 1's cutoff need no exception.  Multiple
eigenvalues (homogeneous fields), one unknown per parent up to 96 (where the tridiagonal
solver's work space no longer fits and Jacobi takes over).

Tolerances: the matrices have norm at most 8 and the exported basis is S-orthonormal to
1e-11, which moves an eigenvalue by 8e-11 at most: 1e-10 for the eigenvalues and, with the
solver's 1e-13 ||T||, for the residuals ||N psi - lam psi||; rows orthonormal to 1e-12."""
import numpy as np
import pytest
import torch

import oracle
from oracle.spectral import element_cells
from oracle.tpfa import assemble, interior_face_mask

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2403_19342_gb300 as p
    return p


@pytest.mark.parametrize("ratio,L,Ln", [((1, 1, 1), 1, 1), ((2, 1, 1), 1, 2), ((3, 1, 1), 1, 2), ((2, 2, 1), 3, 12),
                                        ((2, 2, 2), 4, 4), ((3, 3, 1), 5, 7), ((4, 2, 2), 4, 9), ((3, 5, 1), 4, 4),
                                        ((2, 2, 2), 11, 24), ((2, 2, 2), 12, 20)])
@pytest.mark.parametrize("homogeneous", [False, True])
def test_pairs_of_the_matrices_solved(pkg, ratio, L, Ln, homogeneous):
    block = (3, 3, 2)
    grid = (2 * ratio[0], ratio[1], ratio[2])
    shape = tuple(g * b for g, b in zip(grid, block))[::-1]
    rng = np.random.default_rng(L + Ln)
    kappa = np.ones(shape) if homogeneous else np.exp(1.5 * rng.standard_normal(shape))
    h = tuple(1.0 / n for n in shape[::-1])
    H = oracle.setup(kappa, h, oracle.Options(n_levels=3, block=block, ratio=[ratio], n_eig=[L, Ln], nu=[1, 1]))
    S = pkg.Solver(torch.tensor(kappa, device="cuda"),
                   pkg.Options(n_levels=3, block=block, ratio=[ratio], n_eig=[L, Ln], eig_tol=1e-12), h=h)
    assert S.setup_status == 0
    Phi, _ = S.export_basis(1)
    Psi, lam = (t.cpu().numpy() for t in S.export_basis(2))
    Phi = Phi.cpu().numpy()
    S.close()
    cells = element_cells(shape, block)
    parent_box = tuple(b * r for b, r in zip(block, ratio))
    A = assemble(H.T * interior_face_mask(shape, parent_box)).tocsr()
    elements = element_cells(grid[::-1], ratio)                  # element indices of each parent
    for P in range(Psi.shape[0]):
        B = np.zeros((int(np.prod(shape)), len(elements[P]) * L))
        for i, e in enumerate(elements[P]):
            B[cells[e], i * L:(i + 1) * L] = Phi[e].T
        N = B.T @ (A @ B)
        w = np.linalg.eigvalsh(0.5 * (N + N.T))
        np.testing.assert_allclose(lam[P], w[:Ln], rtol=0, atol=1e-10)
        np.testing.assert_allclose(Psi[P] @ Psi[P].T, np.eye(Ln), rtol=0, atol=1e-12)
        R = N @ Psi[P].T - Psi[P].T * lam[P][None, :]
        assert np.linalg.norm(R, axis=0).max() <= 1e-10
