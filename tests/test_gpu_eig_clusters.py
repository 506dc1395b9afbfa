"""Level-1 subspace eigensolve of elements whose wanted eigenvalues end inside a cluster: three
permeability layers in y plus a thin fourth below a full channel 1e5 times as permeable leave
eigenvalues 11 to 15 within 4e-4 of each other (L = 12, so the cutoff splits them).  A
filter of one degree on one interval can leave an unwanted vector undamped there, iteration
after iteration; with the degree varied the elements need about 16 (mixed) and 33 (FP64)
iterations, and 100 is the cap here.

Tolerance: residuals of at most eig_tol = 1e-8 on the symmetric form; eigenvalues of a
symmetric matrix of norm at most 8 are then within 1e-8 of the exact ones."""
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


@pytest.mark.parametrize("mixed", [True, False])
@pytest.mark.parametrize("layers", [(282.85560171, 282.85560171, 330.82258369, 330.82258369, 123.05305216, 123.05305216,
                                     123.05305216, 46.09138814),
                                    (282.9, 282.9, 330.8, 330.8, 123.1, 123.1, 123.1, 46.1)])
def test_cutoff_inside_a_cluster(pkg, mixed, layers):
    kappa = np.empty((8, 8, 16))
    kappa[:4] = np.array(layers)[None, :, None]
    kappa[4:] = 4.67695575e7
    h = (1.0 / 512,) * 3
    kw = dict(n_levels=2, block=(8, 8, 8), ratio=[], n_eig=[12])
    S = pkg.Solver(torch.tensor(kappa, device="cuda"),
                   pkg.Options(precision=pkg.MIXED if mixed else pkg.FP64, eig_tol=1e-8, eig_max_iter=100, **kw), h=h)
    info = S.info
    lam = S.export_basis(1)[1].cpu().numpy()
    status = S.setup_status
    S.close()
    assert status == 0 and info["eig_residual_max"] <= 1e-8, info
    assert info["eig_iterations_max"] <= 60
    H = oracle.setup(kappa, h, oracle.Options(nu=[1], **kw))
    np.testing.assert_allclose(lam, H.lam[0], rtol=0, atol=1.01e-8)
