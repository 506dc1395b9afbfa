"""Saturation sub-steps (Eq. (ES)) at the edges of their kernels: grids that are not a
multiple of the CTA size, one cell per direction in an element, 0 to 5 sub-steps (the two
maxima alternate), saturations outside the fluid model's range, face velocities on the
boundary (which carry no flow), viscosities whose fractional flow leaves FP32's range.

Tolerance: a sub-step is a few dozen FP64 operations on values of order 1 whose change is
at most ds_max = 1e-3, so 1e-13 absolute on S and 1e-13 relative on the time."""
import numpy as np
import pytest
import torch

from oracle import impes

pytestmark = pytest.mark.gpu

P_BH = 4000.0


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2403_19342_gb300 as p
    return p


def problem(shape, seed, lo=-0.2, hi=1.2):
    rng = np.random.default_rng(seed)
    S = rng.uniform(lo, hi, size=shape)
    phi = rng.uniform(0.05, 0.3, size=shape)
    p = P_BH + rng.normal(0, 50.0, size=shape)
    w = np.where(rng.uniform(size=shape) < 0.1, rng.uniform(0, 1.0, size=shape), 0.0)
    q = np.where(rng.uniform(size=shape) < 0.1, rng.uniform(0, 50.0, size=shape), 0.0)
    v = rng.normal(0, 30.0, size=(3,) + tuple(shape))     # boundary faces too: they must carry nothing
    v[:, rng.uniform(size=shape) < 0.1] = 0.0
    return S, phi, p, w, q, v


def solver(pkg, shape, block, h):
    nz, ny, nx = shape
    return pkg.Solver(torch.ones(shape, dtype=torch.float64, device="cuda"),
                      pkg.Options(n_levels=2, block=block, ratio=[], n_eig=[1], eig_tol=1e-10), h=h)


@pytest.mark.parametrize("shape,block", [((2, 2, 2), (1, 2, 2)), ((1, 1, 34), (2, 1, 1)), ((7, 6, 10), (5, 3, 7)),
                                         ((16, 20, 32), (4, 4, 4))])
@pytest.mark.parametrize("M", [0, 1, 2, 5])
def test_substeps_against_oracle(pkg, shape, block, M):
    h = (20.0, 10.0, 3.0)
    S, phi, p, w, q, v = problem(shape, 3 + M)
    t = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    sol = solver(pkg, shape, block, h)
    Sg = t(S)
    dt = pkg.msmg_impes_transport(sol.ctx, pkg.make_fluid(), t(v), t(p), t(w), P_BH, t(q), t(phi), Sg, M, 1e-3)
    Sr, dtr = impes.transport(S, v, p, w, P_BH, q, phi, h, M, 1e-3, impes.Fluid())
    np.testing.assert_allclose(Sg.cpu().numpy(), Sr, rtol=0, atol=1e-13)
    np.testing.assert_allclose(dt, dtr, rtol=1e-13)
    sol.close()


@pytest.mark.parametrize("mu_w,mu_o", [(1e-45, 3e-45), (1e60, 2e60), (0.3, 1e-50)])
def test_viscosities_outside_fp32_range(pkg, mu_w, mu_o):
    shape, h = (8, 8, 8), (1.0, 1.0, 1.0)
    S, phi, p, w, q, v = problem(shape, 9, 0.2, 0.8)
    t = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    sol = solver(pkg, shape, (4, 4, 4), h)
    Sg = t(S)
    dt = pkg.msmg_impes_transport(sol.ctx, pkg.make_fluid(mu_w, mu_o), t(v), t(p), t(w), P_BH, t(q), t(phi), Sg, 3, 1e-3)
    Sr, dtr = impes.transport(S, v, p, w, P_BH, q, phi, h, 3, 1e-3, impes.Fluid(mu_w, mu_o))
    np.testing.assert_allclose(Sg.cpu().numpy(), Sr, rtol=0, atol=1e-13)
    np.testing.assert_allclose(dt, dtr, rtol=1e-13)
    sol.close()


def test_not_a_number_stays_local(pkg):
    """A NaN or infinite saturation: the NaN cell and its neighbours become NaN, the infinite
    one is clipped by the fluid model, and the step length ignores NaN rates."""
    shape, h = (8, 8, 8), (1.0, 1.0, 1.0)
    S, phi, p, w, q, v = problem(shape, 11, 0.2, 0.8)
    S[4, 4, 4] = np.nan
    S[1, 1, 1] = np.inf
    t = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    sol = solver(pkg, shape, (4, 4, 4), h)
    Sg = t(S)
    dt = pkg.msmg_impes_transport(sol.ctx, pkg.make_fluid(), t(v), t(p), t(w), P_BH, t(q), t(phi), Sg, 1, 1e-3)
    r = impes.saturation_rate(S, v, p, w, P_BH, q, phi, h, impes.Fluid())
    top = np.nanmax(np.abs(r))
    np.testing.assert_allclose(dt, 1e-3 / top, rtol=1e-13)
    got, ref = Sg.cpu().numpy(), S + 1e-3 / top * r
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.isnan(got[4, 4, 4])
    fine = np.isfinite(ref)
    np.testing.assert_allclose(got[fine], ref[fine], rtol=0, atol=1e-13)
    sol.close()
