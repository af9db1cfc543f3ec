"""Direct potentials through every grouping of densities (1, 2, 4, 8 and 16 per
lane, a second pass beyond 64) and ragged point counts, Laplace and Helmholtz,
against the oracle at 1e-12."""
import numpy as np
import pytest

from gpu_common import lib, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("nrhs,npts", [(1, 1), (3, 7), (5, 8), (9, 9), (20, 33), (40, 2), (64, 31), (70, 17)])
def test_groups_against_oracle(kernel, nrhs, npts):
    import torch
    from oracle import galerkin, geometry, solve
    ibem = lib()
    kappa = 3.0 if kernel else 0.0
    kern = galerkin.HelmholtzKernel(kappa) if kernel else galerkin.LaplaceKernel()
    disc = galerkin.Discretisation(geometry.unit_sphere(), 1, 1, kern)
    rng = np.random.default_rng(40 + nrhs + kernel)
    w = rng.normal(size=(nrhs, disc.mesh.n_dofs)) + (1j * rng.normal(size=(nrhs, disc.mesh.n_dofs)) if kernel else 0.0)
    P = rng.normal(size=(npts, 3))
    P *= (rng.uniform(1.2, 4.0, size=npts) / np.linalg.norm(P, axis=1))[:, None]
    u0 = solve.potential(disc, w.T, P).T
    h = ibem.ibem_create(ibem.sphere_patches(), ibem.make_params(1, 1, q_cheb=0, kernel=kernel, kappa=kappa))
    wd = torch.from_numpy(np.ascontiguousarray(np.stack([w.real, w.imag], -1) if kernel else w)).cuda()
    u = torch.full((nrhs, npts, 2) if kernel else (nrhs, npts), np.nan, dtype=torch.float64, device="cuda")
    ibem.ibem_potential(h, wd, nrhs, torch.from_numpy(P).cuda(), u)
    un = u.cpu().numpy()
    un = un[..., 0] + 1j * un[..., 1] if kernel else un
    for r in range(nrhs):
        assert rel_err(un[r], u0[r]) < 1e-12
    ibem.ibem_destroy(h)
