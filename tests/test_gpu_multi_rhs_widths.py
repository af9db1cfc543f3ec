"""The FP32 operator with 16 to 256 right-hand sides at the edges of its tiles:
one and two MMAs per K block (more than 256 rows of moments), every even q, ragged
counts of right-hand sides, slices of the near rows and the per-thread transfers,
generated and stored coupling.  Against the FP64 operator; the BF16 rounding of K
and of the moments (2^-9 relative each) bounds the error as in the other tests of this path."""
import numpy as np
import pytest

from gpu_common import lib, rel_err

pytestmark = pytest.mark.gpu


def _apply(h, x, precision, cplx):
    import torch
    ibem = lib()
    xd = torch.from_numpy(np.ascontiguousarray(np.stack([x.real, x.imag], -1) if cplx else x)).cuda()
    yd = torch.empty_like(xd)
    ibem.ibem_matvec(h, xd, yd, x.shape[0], precision)
    torch.cuda.synchronize()
    y = yd.cpu().numpy()
    return y[..., 0] + 1j * y[..., 1] if cplx else y


@pytest.mark.parametrize("kernel,p,m,q,R", [(0, 0, 4, 2, 16), (0, 1, 3, 4, 31), (0, 2, 3, 10, 256), (0, 4, 2, 6, 33),
                                            (0, 3, 3, 8, 129), (1, 0, 3, 2, 129), (1, 1, 3, 4, 256), (1, 2, 3, 6, 17),
                                            (1, 3, 3, 8, 200), (1, 4, 2, 8, 97)])
def test_widths_against_fp64(kernel, p, m, q, R):
    ibem = lib()
    h = ibem.ibem_create(ibem.sphere_patches(), ibem.make_params(p, m, q_cheb=q, eta=1.6, kernel=kernel,
                                                                 kappa=3.0 if kernel else 0.0))
    ibem.ibem_assemble(h)
    n = ibem.ibem_get_info(h).ndof
    rng = np.random.default_rng(1000 + R + q)
    x = rng.normal(size=(R, n)) + (1j * rng.normal(size=(R, n)) if kernel else 0.0)
    y64 = np.concatenate([_apply(h, x[r:r + 8], 0, bool(kernel)) for r in range(0, R, 8)])
    modes = [ibem.IBEM_FP32_COUPLING_GENERATE] + ([ibem.IBEM_FP32_COUPLING_STORE] if kernel and q == 8 else [])
    for mode in modes:
        if kernel:
            ibem.ibem_set_fp32_coupling(h, mode)
        y = _apply(h, x, 1, bool(kernel))
        assert ibem.ibem_device_status(h) == ibem.IBEM_DEVICE_OK
        for r in range(R):
            assert rel_err(y[r], y64[r]) < 5e-3, (mode, r)
        assert np.array_equal(_apply(h, x, 1, bool(kernel)), y)
    ibem.ibem_destroy(h)
