"""Work space of the operator, whatever was called before it."""
import numpy as np
import pytest

from gpu_common import lib, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("R", [1, 5])
def test_right_hand_side_before_assembly(kernel, R):
    # ibem_rhs needs no assembly and sizes the work vectors before there are coupling matrices
    import torch
    ibem = lib()
    hs = [ibem.ibem_create(ibem.sphere_patches(), ibem.make_params(1, 2, q_cheb=4, eta=1.6, kernel=kernel,
                                                                   kappa=3.0 if kernel else 0.0)) for _ in range(2)]
    info = ibem.ibem_get_info(hs[0])
    tail = (2,) if kernel else ()
    g = torch.from_numpy(np.random.default_rng(1600).normal(size=(R, info.n_quad_points) + tail)).cuda()
    x = torch.from_numpy(np.random.default_rng(1601).normal(size=(R, info.ndof) + tail)).cuda()
    b = [torch.full_like(x, np.nan) for _ in hs]
    y = [torch.full_like(x, np.nan) for _ in hs]
    ibem.ibem_rhs(hs[0], g, R, b[0])
    for h, out in zip(hs, y):
        ibem.ibem_assemble(h)
        ibem.ibem_matvec(h, x, out, R)
    ibem.ibem_rhs(hs[1], g, R, b[1])
    torch.cuda.synchronize()
    for a in (b, y):
        assert rel_err(a[0].cpu().numpy(), a[1].cpu().numpy()) < 1e-13
    for h in hs:
        ibem.ibem_destroy(h)
