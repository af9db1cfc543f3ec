"""FP64 application: the shared launches of the coarse levels, the grouped
restriction and the sliced near rows, each right-hand side against the oracle
and against the same vector applied in other groupings (1e-12: only the order
of the sums differs)."""
import numpy as np
import pytest

from gpu_common import lib, rel_err

pytestmark = pytest.mark.gpu
TOL64 = 1e-12


def _apply(h, x, cplx):
    import torch
    ibem = lib()
    xd = torch.from_numpy(np.ascontiguousarray(np.stack([x.real, x.imag], -1) if cplx else x)).cuda()
    yd = torch.full_like(xd, np.nan)
    ibem.ibem_matvec(h, xd, yd, x.shape[0], 0)
    torch.cuda.synchronize()
    y = yd.cpu().numpy()
    return y[..., 0] + 1j * y[..., 1] if cplx else y


def _handle(p, m, q, kernel):
    ibem = lib()
    h = ibem.ibem_create(ibem.sphere_patches(), ibem.make_params(p, m, q_cheb=q, eta=1.6, kernel=kernel,
                                                                 kappa=3.0 if kernel else 0.0))
    ibem.ibem_assemble(h)
    return h


def _vectors(n, R, kernel):
    rng = np.random.default_rng(1100 + n + R)
    return rng.normal(size=(R, n)) + (1j * rng.normal(size=(R, n)) if kernel else 0.0)


@pytest.mark.parametrize("kernel,p,m,q", [(0, 0, 1, 4), (0, 1, 2, 5), (0, 0, 3, 3), (0, 0, 4, 4), (1, 0, 1, 4),
                                          (1, 1, 2, 3), (1, 0, 3, 4)])
def test_levels_against_oracle(kernel, p, m, q):
    from oracle import fmm, galerkin, geometry
    ker = galerkin.HelmholtzKernel(3.0) if kernel else galerkin.LaplaceKernel()
    op = fmm.FMMOperator(galerkin.Discretisation(geometry.unit_sphere(), p, m, ker), q, 1.6)
    h = _handle(p, m, q, kernel)
    x = _vectors(op.mesh.n_dofs, 2, kernel)
    y = _apply(h, x, bool(kernel))
    for r in range(2):
        assert rel_err(y[r], op.matvec(x[r])) < TOL64
    lib().ibem_destroy(h)


@pytest.mark.parametrize("kernel,p,m,q,R", [(0, 0, 3, 4, 5), (0, 1, 3, 6, 13), (0, 2, 3, 5, 64), (0, 3, 2, 6, 9),
                                            (0, 4, 2, 7, 3), (1, 0, 3, 4, 8), (1, 1, 3, 4, 4), (1, 2, 3, 6, 33),
                                            (1, 3, 2, 6, 14), (1, 4, 2, 5, 28), (1, 2, 2, 8, 64), (1, 1, 2, 9, 17)])
def test_groupings_agree(kernel, p, m, q, R):
    h = _handle(p, m, q, kernel)
    x = _vectors(lib().ibem_get_info(h).ndof, R, kernel)
    y = _apply(h, x, bool(kernel))
    for r in range(0, R, 3):
        assert rel_err(y[r], _apply(h, x[r:r + 1], bool(kernel))[0]) < TOL64, r
    lib().ibem_destroy(h)
