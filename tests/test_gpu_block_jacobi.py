"""Block-Jacobi over the sizes of its blocks (one to 64 dofs) and several columns at a
time: every column of a lock-step solve reaches its own true residual, in as many
iterations as alone (two more or less each: only the order of sums differs)."""
import numpy as np
import pytest

from gpu_common import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel,p,m", [(0, 0, 2), (0, 2, 3), (0, 4, 2), (1, 0, 1), (1, 1, 3), (1, 3, 2), (1, 4, 3)])
def test_columns_together_and_alone(kernel, p, m):
    import torch
    ibem = lib()
    h = ibem.ibem_create(ibem.sphere_patches(), ibem.make_params(p, m, q_cheb=6, eta=1.6, kernel=kernel,
                                                                 kappa=2.0 if kernel else 0.0))
    ibem.ibem_assemble(h)
    info = ibem.ibem_get_info(h)
    pts = torch.empty((info.n_quad_points, 3), dtype=torch.float64, device="cuda")
    ibem.ibem_quad_points(h, pts)
    src = torch.tensor([[0.3, 0.1, -0.2], [-0.4, 0.2, 0.3], [0.1, -0.5, 0.0]], dtype=torch.float64, device="cuda")
    d = torch.cdist(src, pts)
    g = 1.0 / d
    if kernel:
        g = torch.stack((torch.cos(2.0 * d) / d, torch.sin(2.0 * d) / d), dim=-1)
    b = torch.empty((3, info.ndof, 2) if kernel else (3, info.ndof), dtype=torch.float64, device="cuda")
    ibem.ibem_rhs(h, g.contiguous(), 3, b)

    def solve(rhs):
        w, r = torch.empty_like(rhs), torch.empty_like(rhs)
        n = rhs.shape[0]
        s = ibem.ibem_solve(h, rhs, w, n, rtol=1e-9, maxit=3000, precond=ibem.IBEM_PRECOND_BLOCK_JACOBI)
        ibem.ibem_matvec(h, w, r, n, 0)
        torch.cuda.synchronize()
        res = (r - rhs).reshape(n, -1).norm(dim=1) / rhs.reshape(n, -1).norm(dim=1)
        # the solver's own residual is recursive (CG); its drift stays far below the tolerance
        assert float(res.max()) < 2e-9
        return s
    alone = sum(solve(b[r:r + 1].contiguous()).iterations for r in range(3))
    assert abs(solve(b).iterations - alone) <= 2 * 3
    ibem.ibem_destroy(h)
