"""Fine kernels on groups of elements, at the shapes and sizes where the grouping changes: line
lengths with and without their own sweep (4, 6, 8; odd ones), one x-line per plane, 32 and 33
lines (the last keeps a warp per element), a last group that is not full, cell counts that
the bulk copies cannot take (odd), planes that are padded, the cell term, and element counts
from which FP64 and the restriction take groups.

Tolerances: FP64 V-cycles match the oracle's to 1e-9 (FP64 rounding).  An FP32 V-cycle has an
error e32, measured by the oracle with level 1 rounded as the kernels round it; the kernels
do the same operations in another summation order, so their error is of that size: 4 e32.
Batches and the fused prolongation do the same operations in the same order: equal bits."""
import numpy as np
import pytest
import torch

import fields
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2403_19342_gb300 as p
    return p


# (block, elements per direction, cell term)
FEW = [((4, 4, 5), (3, 3, 3), True), ((4, 4, 4), (3, 3, 3), False), ((6, 4, 5), (2, 5, 1), False),
       ((8, 4, 4), (2, 3, 3), True), ((5, 3, 7), (3, 3, 1), True), ((4, 1, 8), (3, 13, 1), False),
       ((1, 8, 6), (5, 2, 3), False), ((8, 32, 2), (2, 2, 1), False), ((2, 33, 2), (2, 1, 2), True),
       ((7, 7, 7), (2, 2, 1), False), ((8, 8, 6), (2, 1, 2), False)]
MANY = [((4, 2, 2), (14, 14, 14), True), ((3, 2, 2), (14, 12, 16), False), ((4, 4, 4), (14, 14, 14), False)]


def make(pkg, block, grid, wells, precision, n_eig, n_rhs):
    rng = np.random.default_rng(block[0] + 10 * grid[0])
    shape = tuple(b * e for b, e in zip(block[::-1], grid[::-1]))
    kappa = np.exp(1.5 * rng.standard_normal(shape))
    W = None
    if wells:
        W = 0.1 * rng.random(shape)       # everywhere: A is well conditioned, e32 is rounding alone
    nl = len(n_eig) + 1
    h = tuple(1.0 / k for k in shape[::-1])
    kw = dict(n_levels=nl, block=block, ratio=[(2, 2, 2)] * (nl - 2), n_eig=list(n_eig))
    H = oracle.setup(kappa, h, oracle.Options(nu=[1] * (nl - 1), cell_diag=W, **kw))
    S = pkg.Solver(torch.tensor(kappa, device="cuda"),
                   pkg.Options(precision=precision, eig_tol=1e-10, **kw,
                               cell_diag=None if W is None else torch.tensor(W, device="cuda")), h=h, n_rhs=n_rhs)
    assert S.import_bases(H.basis[:nl - 1]) == 0
    return H, S, shape


def check(pkg, block, grid, wells, mixed, n_eig):
    H, S, shape = make(pkg, block, grid, wells, pkg.MIXED if mixed else pkg.FP64, n_eig, 3)
    rng = np.random.default_rng(3)
    R = rng.standard_normal((3,) + shape)
    R -= R.mean(axis=(1, 2, 3), keepdims=True)
    # V-cycle, separate and fused prolongation
    zs = []
    for fused in (0, 1):
        pkg.msmg_set_tuning(S.ctx, (fused, fused, 0, 0))
        zs.append(S.apply_precond(torch.tensor(R[0], device="cuda")).cpu().numpy())
    assert np.array_equal(zs[0], zs[1])
    z64 = oracle.vcycle(H, R[0].ravel())
    nz = np.linalg.norm(z64)
    err = np.linalg.norm(zs[0].ravel() - z64) / nz
    tol = 4 * np.linalg.norm(oracle.vcycle_mixed(H, R[0].ravel()) - z64) / nz if mixed else 1e-9
    assert 0 < tol and err <= tol, (err, tol)
    # solves: three right-hand sides in one batch and one by one, the same bits
    F = torch.tensor(R, device="cuda")
    x, info, _ = S.solve(F, rtol=1e-9, max_iter=200)
    for j in range(3):
        xj, ij, _ = S.solve(F[j].contiguous(), rtol=1e-9, max_iter=200)
        assert torch.equal(xj.reshape(-1), x[j].reshape(-1))
        ij = ij if isinstance(ij, dict) else ij[0]
        assert ij["converged"] and ij["true_rel_residual"] <= 1.1e-9
    S.close()


@pytest.mark.parametrize("mixed", [True, False])
@pytest.mark.parametrize("block,grid,wells", FEW)
def test_few_elements(pkg, block, grid, wells, mixed):
    check(pkg, block, grid, wells, mixed, [9])


@pytest.mark.parametrize("mixed", [True, False])
@pytest.mark.parametrize("block,grid,wells", MANY)
def test_many_elements(pkg, block, grid, wells, mixed):
    check(pkg, block, grid, wells, mixed, [3, 3])
