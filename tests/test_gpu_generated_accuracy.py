"""Accuracy of the double-float couplings against the native FP64 generation of every
far block.  Tolerances: 4/3 of the error of earlier, slower forms for the same
vectors, which may not be exceeded: generated and sliced with every float pair normalised
and a four-part phase reduction (3.36e-15 and 2.96e-15, 3.59e-15 and 1.62e-15), stored
with every far block kept and sums over blocks in FP64 (2.61e-16, 4.48e-16)."""
import numpy as np
import pytest

from gpu_common import lib

pytestmark = pytest.mark.gpu


def _applications(p, m, q, kappa, couplings):
    import torch
    ibem = lib()
    n = 6 * (2 ** m + p) ** 2
    x = torch.from_numpy(np.random.default_rng([5, m, int(kappa * 10)]).normal(size=(6, n, 2))).cuda()
    out = []
    for coupling in couplings:
        h = ibem.ibem_create(ibem.sphere_patches(), ibem.make_params(p, m, q_cheb=q, eta=1.6, kernel=1, kappa=kappa,
                                                                     fp64_coupling=coupling))
        ibem.ibem_assemble(h)
        y = torch.empty_like(x)
        ibem.ibem_matvec(h, x, y, 6)
        torch.cuda.synchronize()
        out.append(y)
        ibem.ibem_destroy(h)
    return [float((y - out[0]).norm() / out[0].norm()) for y in out[1:]]


@pytest.mark.parametrize("p,m,kappa,gen,sliced", [(1, 2, 8.0, 4.5e-15, 4.0e-15), (2, 3, 4.0, 4.8e-15, 2.2e-15)])
def test_error_against_native(p, m, kappa, gen, sliced):
    ibem = lib()
    err = _applications(p, m, 8, kappa, (ibem.IBEM_COUPLING_NATIVE, ibem.IBEM_COUPLING_GENERATE,
                                         ibem.IBEM_COUPLING_SLICED))
    assert err[0] < gen and err[1] < sliced, err


@pytest.mark.parametrize("p,m,q,kappa,tol", [(1, 3, 5, 8.0, 3.5e-16), (2, 4, 8, 1.0, 6.0e-16)])
def test_stored_error_against_native(p, m, q, kappa, tol):
    ibem = lib()
    err = _applications(p, m, q, kappa, (ibem.IBEM_COUPLING_NATIVE, ibem.IBEM_COUPLING_DF))
    assert err[0] < tol, err
