"""Sliced coupling with waits that run out at any point of a row: the call comes
back with the timeout status or with the right result, and the handle goes on."""
import numpy as np
import pytest

from gpu_common import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [32, 64])
def test_short_waits(R):
    import torch
    ibem = lib()
    h = ibem.ibem_create(ibem.sphere_patches(), ibem.make_params(1, 3, q_cheb=8, eta=1.6, kernel=1, kappa=3.0,
                                                                 fp64_coupling=ibem.IBEM_COUPLING_SLICED))
    ibem.ibem_assemble(h)
    x = torch.from_numpy(np.random.default_rng(1700 + R).normal(size=(R, ibem.ibem_get_info(h).ndof, 2))).cuda()
    ref, y = torch.empty_like(x), torch.empty_like(x)
    ibem.ibem_matvec(h, x, ref, R)
    assert ibem.ibem_device_status(h) == ibem.IBEM_DEVICE_OK
    for limit in (0, 1, 2, 4, 16, 256, 1 << 26):
        ibem.ibem_set_wait_limit(h, limit)
        ibem.ibem_matvec(h, x, y, R)
        status = ibem.ibem_device_status(h)
        assert status in (ibem.IBEM_DEVICE_OK, ibem.IBEM_DEVICE_TIMEOUT)
        assert status == ibem.IBEM_DEVICE_TIMEOUT if limit == 0 else True
        if status == ibem.IBEM_DEVICE_OK:
            assert torch.equal(y, ref), limit
    assert status == ibem.IBEM_DEVICE_OK
    ibem.ibem_destroy(h)
