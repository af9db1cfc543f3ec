"""Batched coupling staged through shared memory: odd and even q, both kernels,
one and many right-hand sides and instances without a far field in one batch.
Each instance against its own FP64 operator, within the FP32 bound of the path."""
import numpy as np
import pytest

from gpu_common import lib, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("specs", [
    [(0, 0.0, 0, 3, 3, 1), (1, 1.0, 1, 3, 5, 3), (0, 0.0, 2, 2, 7, 17), (1, 4.0, 0, 2, 8, 2)],
    [(1, 3.0, 1, 1, 4, 5), (0, 0.0, 1, 3, 2, 7), (1, 2.0, 2, 3, 6, 1)],
    [(0, 0.0, 4, 2, 6, 33)],
])
def test_instances_against_fp64(specs):
    import torch
    ibem = lib()
    hs = []
    for kern, kappa, p, m, q, _ in specs:
        hs.append(ibem.ibem_create(ibem.sphere_patches(), ibem.make_params(p, m, q_cheb=q, eta=1.6, kernel=kern,
                                                                           kappa=kappa)))
        ibem.ibem_assemble(hs[-1])
    b = ibem.ibem_batch_create(hs, [s[5] for s in specs])
    off = ibem.ibem_batch_offsets(b, len(hs))
    x = torch.from_numpy(np.random.default_rng(1300 + len(specs)).normal(size=off[-1])).cuda()
    y = torch.full_like(x, np.nan)
    ibem.ibem_batch_matvec(b, x, y)
    for i, (h, s) in enumerate(zip(hs, specs)):
        xi = x[off[i]:off[i + 1]].contiguous()
        y64 = torch.empty_like(xi)
        ibem.ibem_matvec(h, xi, y64, s[5], 0)
        torch.cuda.synchronize()
        assert rel_err(y[off[i]:off[i + 1]].cpu().numpy(), y64.cpu().numpy()) < 2e-5, i
    ibem.ibem_batch_destroy(b)
    for h in hs:
        ibem.ibem_destroy(h)
