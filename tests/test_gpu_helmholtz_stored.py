"""The stored double-float Helmholtz coupling (one of two mirrored
blocks, used for both directions, two right-hand sides per CTA and eight per pass) against the
native FP64 generation of every far block: all groupings of right-hand sides
and every storage width (q odd and even), at the 1e-12 parity tolerance; and
repeated applications bitwise."""
import numpy as np
import pytest

from gpu_common import lib, rel_err

pytestmark = pytest.mark.gpu


def _apply(h, x):
    import torch
    ibem = lib()
    xd = torch.from_numpy(np.ascontiguousarray(np.stack([x.real, x.imag], -1))).cuda()
    yd = torch.empty_like(xd)
    ibem.ibem_matvec(h, xd, yd, x.shape[0], 0)
    torch.cuda.synchronize()
    y = yd.cpu().numpy()
    return y[..., 0] + 1j * y[..., 1]


@pytest.mark.parametrize("q,nrhs", [(2, 1), (3, 4), (4, 2), (5, 3), (6, 1), (6, 7), (6, 8), (6, 9), (7, 5), (8, 13),
                                    (9, 2), (10, 6)])
def test_stored_equals_native(q, nrhs):
    ibem = lib()
    hs = [ibem.ibem_create(ibem.sphere_patches(), ibem.make_params(1, 2, q_cheb=q, eta=1.6, kernel=1, kappa=3.0,
                                                                   fp64_coupling=c))
          for c in (ibem.IBEM_COUPLING_DF, ibem.IBEM_COUPLING_NATIVE)]
    for h in hs:
        ibem.ibem_assemble(h)
    assert ibem.ibem_get_info(hs[0]).bytes_far > 0
    n = ibem.ibem_get_info(hs[0]).ndof
    rng = np.random.default_rng(900 + q)
    x = rng.normal(size=(nrhs, n)) + 1j * rng.normal(size=(nrhs, n))
    y, y0 = _apply(hs[0], x), _apply(hs[1], x)
    for r in range(nrhs):
        assert rel_err(y[r], y0[r]) < 1e-12
    assert np.array_equal(_apply(hs[0], x), y)
    # one column alone takes another grouping
    assert rel_err(_apply(hs[0], x[-1:]), y0[-1:]) < 1e-12
    for h in hs:
        ibem.ibem_destroy(h)
