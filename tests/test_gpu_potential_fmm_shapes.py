"""Interpolated potential over the forms of its lists and of its evaluation: few
and many interpolation points, Gauss orders whose element rule exceeds a CTA,
one and several tiles of densities, a point count that is no multiple of a
warp.  Against the oracle at 1e-12 (only the order of the sums differs)."""
import numpy as np
import pytest

from gpu_common import lib, rel_err

pytestmark = pytest.mark.gpu
TOL64 = 1e-12


@pytest.mark.parametrize("kernel,p,m,q,order,R", [(0, 0, 1, 2, 4, 1), (0, 3, 2, 3, 18, 17), (1, 1, 3, 5, 6, 2),
                                                  (1, 2, 2, 8, 17, 16)])
def test_shapes_against_oracle(kernel, p, m, q, order, R):
    import torch
    from oracle import fmm, galerkin, geometry
    ibem = lib()
    ker = galerkin.HelmholtzKernel(3.0) if kernel else galerkin.LaplaceKernel()
    op = fmm.FMMOperator(galerkin.Discretisation(geometry.unit_sphere(), p, m, ker, n_regular=order), q, 1.6)
    rng = np.random.default_rng(1400 + order)
    w = rng.normal(size=(R, op.mesh.n_dofs)) + (1j * rng.normal(size=(R, op.mesh.n_dofs)) if kernel else 0.0)
    P = rng.normal(size=(37, 3))
    P *= (rng.uniform(1.05, 3.0, size=37) / np.linalg.norm(P, axis=1))[:, None]
    h = ibem.ibem_create(ibem.sphere_patches(), ibem.make_params(p, m, q_cheb=q, eta=1.6, kernel=kernel,
                                                                 kappa=3.0 if kernel else 0.0, gauss_regular=order))
    wd = torch.from_numpy(np.ascontiguousarray(np.stack([w.real, w.imag], -1) if kernel else w)).cuda()
    u = torch.full((R, 37, 2) if kernel else (R, 37), np.nan, dtype=torch.float64, device="cuda")
    counts = ibem.ibem_potential_fmm(h, wd, R, torch.from_numpy(P).cuda(), u)
    un = u.cpu().numpy()
    un = un[..., 0] + 1j * un[..., 1] if kernel else un
    assert rel_err(un, op.potential(w.T, P).T) < TOL64
    assert counts == tuple(np.sum(op.potential_counts, axis=0))
    ibem.ibem_destroy(h)
