"""Network training kernels on batches that fill the chip and on some that do not: both
pixel tiles of the FP32 convolution and the tile heights of the weight gradient, against
the FP64 oracle."""
import numpy as np
import pytest

from gpu_common import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,n,H,W", [(8, 60, 35, 70), (8, 310, 12, 36), (8, 24, 13, 37), (16, 90, 10, 10)])
def test_gradients_of_large_batches(C, n, H, W):
    import torch
    from oracle import cnn
    ibem = lib()
    c = ibem.ibem_cnn_create(C, seed=H)
    p = ibem.ibem_cnn_params(c).astype(np.float64)
    rng = np.random.default_rng(1900 + H)
    x, t = (rng.normal(size=(n, 2, H, W)).astype(np.float32) for _ in range(2))
    xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    out = torch.full_like(xd, np.nan)
    ibem.ibem_cnn_forward(c, xd, out, ibem.IBEM_FP32)
    ref = cnn.forward(p, x.astype(np.float64), C)
    assert np.linalg.norm(out.cpu().numpy() - ref) < 1e-5 * np.linalg.norm(ref)
    loss0, g0 = cnn.loss_and_grad(p, x.astype(np.float64), t.astype(np.float64), C)
    loss, g = ibem.ibem_cnn_gradients(c, xd, td, ibem.IBEM_FP32)
    assert loss == pytest.approx(loss0, rel=1e-6)
    off = 0
    for ci, co in cnn.layer_channels(C):
        for k in (co * ci * 9, co):
            assert np.linalg.norm(g[off:off + k] - g0[off:off + k]) <= 1e-4 * np.linalg.norm(g0[off:off + k])
            off += k
    ibem.ibem_cnn_destroy(c)
