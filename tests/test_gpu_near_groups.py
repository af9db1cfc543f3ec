"""FP64 Helmholtz near product of several right-hand sides where they take fewer
threads than a CTA has (degree 4, four and five columns: 100 and 125 of 256) and the
widths around it: every column against the same column alone (another kernel) at
1e-12."""
import numpy as np
import pytest

from gpu_common import lib, rel_err

pytestmark = pytest.mark.gpu
TOL64 = 1e-12


def _apply(h, x):
    import torch
    xd = torch.from_numpy(np.ascontiguousarray(np.stack([x.real, x.imag], -1))).cuda()
    yd = torch.full_like(xd, np.nan)
    lib().ibem_matvec(h, xd, yd, x.shape[0], 0)
    y = yd.cpu().numpy()
    return y[..., 0] + 1j * y[..., 1]


@pytest.mark.parametrize("q", [0, 4])
def test_degree_4_columns(q):
    ibem = lib()
    h = ibem.ibem_create(ibem.sphere_patches(), ibem.make_params(4, 2, q_cheb=q, eta=1.6, kernel=1, kappa=3.0))
    ibem.ibem_assemble(h)
    rng = np.random.default_rng(1500 + q)
    x = rng.normal(size=(11, ibem.ibem_get_info(h).ndof)) + 1j * rng.normal(size=(11, ibem.ibem_get_info(h).ndof))
    alone = [_apply(h, x[r:r + 1])[0] for r in range(11)]
    for R in (4, 5, 6, 10, 11):
        for _ in range(3):
            y = _apply(h, x[:R])
            for r in range(R):
                assert rel_err(y[r], alone[r]) < TOL64, (R, r)
    ibem.ibem_destroy(h)
