"""Accuracy of the generated and sliced double-float couplings against the native
FP64 generation of every far block.  Tolerances: 4/3 of what the arithmetic with
every float pair normalised and a four-part phase reduction gives for the same
vectors (3.36e-15 and 2.96e-15, 3.59e-15 and 1.62e-15), which the kernel values may
not be worse than."""
import numpy as np
import pytest

from gpu_common import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,m,kappa,gen,sliced", [(1, 2, 8.0, 4.5e-15, 4.0e-15), (2, 3, 4.0, 4.8e-15, 2.2e-15)])
def test_error_against_native(p, m, kappa, gen, sliced):
    import torch
    ibem = lib()
    n = 6 * (2 ** m + p) ** 2
    x = torch.from_numpy(np.random.default_rng([5, m, int(kappa * 10)]).normal(size=(6, n, 2))).cuda()
    out = []
    for coupling in (ibem.IBEM_COUPLING_NATIVE, ibem.IBEM_COUPLING_GENERATE, ibem.IBEM_COUPLING_SLICED):
        h = ibem.ibem_create(ibem.sphere_patches(), ibem.make_params(p, m, q_cheb=8, eta=1.6, kernel=1, kappa=kappa,
                                                                     fp64_coupling=coupling))
        ibem.ibem_assemble(h)
        y = torch.empty_like(x)
        ibem.ibem_matvec(h, x, y, 6)
        torch.cuda.synchronize()
        out.append(y)
        ibem.ibem_destroy(h)
    err = [float((y - out[0]).norm() / out[0].norm()) for y in out[1:]]
    assert err[0] < gen and err[1] < sliced, err
