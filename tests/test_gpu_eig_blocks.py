"""Level-1 subspace eigensolver over the element sizes its thread layout distinguishes (one
to four warps, four cells per thread, sizes that fill a warp or leave one cell over, odd
sizes) and block widths (K = 5 .. 16), against LAPACK on fields that stress it: a smooth
lognormal one, a high-contrast one whose weighted starting vectors are nearly dependent, a
homogeneous one with multiple eigenvalues.

Tolerances: eigenvalues of a symmetric matrix of norm at most 8 with residual 1e-12 are
accurate to 1e-12; 1e-10 leaves room for LAPACK's own rounding at contrast 1e6.  The basis is
S-orthonormal to the rounding of the Rayleigh-Ritz step (a Cholesky factor with pivots above
1e-3): 1e-11."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

BLOCKS = [(5, 13, 1), (4, 4, 5), (8, 4, 4), (43, 3, 1), (6, 6, 6), (8, 8, 6), (5, 11, 7), (8, 8, 8)]


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2403_19342_gb300 as p
    return p


def field(kind, shape, seed):
    rng = np.random.default_rng(seed)
    if kind == "homogeneous":
        return np.ones(shape)
    y = rng.standard_normal(shape)
    if kind == "smooth":
        return np.exp(0.5 * y)
    k = np.ones(shape)                            # one high block per element corner
    k[:, : shape[1] // 4, : shape[2] // 4] = 1e6
    k[:, -(shape[1] // 3):, -(shape[2] // 3):] = 1e4
    return k * np.exp(0.1 * y)


@pytest.mark.parametrize("block", BLOCKS)
@pytest.mark.parametrize("kind,L,mixed", [("smooth", 4, 0), ("smooth", 12, 1), ("contrast", 6, 1), ("contrast", 1, 0),
                                          ("contrast", 12, 0), ("homogeneous", 8, 1)])
def test_eigenpairs_against_lapack(pkg, block, kind, L, mixed):
    bx, by, bz = block
    shape = (bz, 2 * by, 2 * bx)                 # 2 x 2 x 1 elements
    if min(L + max(4, L // 2), 16) > min(bx, 4) * min(by, 4) * min(bz, 4):
        pytest.skip("more block vectors than starting modes")
    kappa = field(kind, shape, bx * by + L)
    S = pkg.Solver(torch.tensor(kappa, device="cuda"),
                   pkg.Options(n_levels=2, block=block, ratio=[], n_eig=[L], precision=mixed, eig_tol=1e-12))
    assert S.setup_status == 0 and S.info["eig_residual_max"] <= 1e-12
    Phi, lam = (t.cpu().numpy() for t in S.export_basis(1))
    S.close()
    h = (1.0 / shape[2], 1.0 / shape[1], 1.0 / shape[0])
    H = oracle.setup(kappa, h, oracle.Options(n_levels=2, block=block, ratio=[], n_eig=[L], nu=[1]))
    np.testing.assert_allclose(lam, H.lam[0], rtol=0, atol=1e-10)
    # S-orthonormality, S = sum_d kappa / h_d^2 per cell in element order
    s = kappa * sum(1.0 / v ** 2 for v in h)
    for e in range(4):
        ey, ex = divmod(e, 2)
        se = s[:, ey * by:(ey + 1) * by, ex * bx:(ex + 1) * bx].ravel()
        np.testing.assert_allclose((Phi[e] * se) @ Phi[e].T, np.eye(L), rtol=0, atol=1e-11)
