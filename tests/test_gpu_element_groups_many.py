"""Fine kernels on groups at the element counts from which FP64 and the restriction take them
(2432): lines of 4, 6 and 8 and an odd one, planes that are padded (8 x 4), more than eight
cells per thread, and shapes on both sides of each kernel's own size rule (use_groups), in
both precisions.  2548 elements: the last group is not full.

Tolerances: an FP64 V-cycle matches the oracle's to 1e-9 (FP64 rounding).  An FP32 V-cycle
has the error of the oracle's V-cycle with level 1 rounded as the kernels round it, in
another summation order: four times that.  Solves reach their tolerance by the oracle's
matrix (10% for rounding); batches give the bits of single solves."""
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


def plain_bases(T, S, box, L, W=None):
    """Level-1 bases that need no eigensolve: the constant and the position along the element,
    S-orthonormal.  The V-cycle's kernels do not depend on what the bases are."""
    cells = oracle.element_cells(T.shape[1:], box)
    s = S.ravel()[cells]                                         # [m, nb]
    phi = np.empty((cells.shape[0], L, cells.shape[1]))
    pos = np.arange(cells.shape[1]) / cells.shape[1]
    for k in range(L):
        v = np.broadcast_to(pos ** k, s.shape).copy()
        for j in range(k):
            v -= (v * s * phi[:, j]).sum(axis=1, keepdims=True) * phi[:, j]
        phi[:, k] = v / np.sqrt((v * v * s).sum(axis=1, keepdims=True))
    return np.tile(np.arange(L, dtype=float), (cells.shape[0], 1)), phi, cells


# (block, cell term)
BLOCKS = [((4, 4, 5), True), ((6, 4, 5), False), ((8, 4, 4), False), ((5, 3, 7), True), ((6, 2, 8), False),
          ((6, 6, 4), False), ((8, 4, 2), True)]


@pytest.mark.parametrize("block,wells", BLOCKS)
def test_many_elements(pkg, monkeypatch, block, wells):
    monkeypatch.setattr(oracle.hierarchy, "level1_eigenpairs", plain_bases)
    grid, ratio = (14, 14, 13), (2, 2, 1)
    rng = np.random.default_rng(sum(block))
    shape = tuple(b * e for b, e in zip(block[::-1], grid[::-1]))
    kappa = np.exp(1.5 * rng.standard_normal(shape))
    W = 0.1 * rng.random(shape) if wells else None
    h = tuple(1.0 / k for k in shape[::-1])
    kw = dict(n_levels=3, block=block, ratio=[ratio], n_eig=[2, 2])
    H = oracle.setup(kappa, h, oracle.Options(nu=[1, 1], cell_diag=W, **kw))
    R = rng.standard_normal((3,) + shape)
    R -= R.mean(axis=(1, 2, 3), keepdims=True)
    z64 = oracle.vcycle(H, R[0].ravel())
    z32 = oracle.vcycle_mixed(H, R[0].ravel())
    nz = np.linalg.norm(z64)
    F = torch.tensor(R, device="cuda")
    for mixed in (False, True):
        S = pkg.Solver(torch.tensor(kappa, device="cuda"),
                       pkg.Options(precision=pkg.MIXED if mixed else pkg.FP64, eig_tol=1e-4,
                                   cell_diag=None if W is None else torch.tensor(W, device="cuda"), **kw), h=h, n_rhs=3)
        assert S.import_bases(H.basis[:2]) == 0
        for fused in (0, 1):
            pkg.msmg_set_tuning(S.ctx, (fused, fused, 0, 0))
            z = S.apply_precond(F[0].contiguous()).cpu().numpy().ravel()
            tol = 4 * np.linalg.norm(z32 - z64) / nz if mixed else 1e-9
            assert 0 < tol and np.linalg.norm(z - z64) <= tol * nz
        x, infos, _ = S.solve(F, rtol=1e-9, max_iter=200)
        for j in range(3):
            xj, ij, _ = S.solve(F[j].contiguous(), rtol=1e-9, max_iter=200)
            assert torch.equal(xj.reshape(-1), x[j].reshape(-1))
            assert ij["converged"] and ij["true_rel_residual"] <= 1.1e-9
        # the converged solution satisfies the oracle's operator: A x = b
        r = R[0].ravel() - H.A[0] @ x[0].cpu().numpy().ravel()
        if not wells:
            r -= r.mean()
        assert np.linalg.norm(r) <= 1.1e-9 * np.linalg.norm(R[0])
        S.close()
