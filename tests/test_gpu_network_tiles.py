"""Network kernels at the edges of their pixel tiles (12 x 36 for FP32, 16 x 16
for BF16): images of one pixel, one below, at and one above a tile, against the
FP64 oracle network at the tolerances of the other tests of these entry points."""
import numpy as np
import pytest

from gpu_common import lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,n,H,W", [(8, 1, 1, 1), (8, 3, 11, 35), (32, 1, 12, 36), (32, 2, 13, 37), (16, 1, 25, 3),
                                     (8, 2, 2, 73), (32, 1, 24, 72)])
def test_forward_and_gradients(C, n, H, W):
    import torch
    from oracle import cnn
    ibem = lib()
    c = ibem.ibem_cnn_create(C, seed=H + W)
    p = ibem.ibem_cnn_params(c).astype(np.float64)
    rng = np.random.default_rng(1200 + H + W)
    x, t = (rng.normal(size=(n, 2, H, W)).astype(np.float32) for _ in range(2))
    xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    ref = cnn.forward(p, x.astype(np.float64), C)
    out = torch.full_like(xd, np.nan)
    for prec, tol in ((ibem.IBEM_FP32, 1e-5), (ibem.IBEM_BF16, 2e-2)):
        ibem.ibem_cnn_forward(c, xd, out, prec)
        torch.cuda.synchronize()
        assert np.linalg.norm(out.cpu().numpy() - ref) < tol * np.linalg.norm(ref)
    loss0, g0 = cnn.loss_and_grad(p, x.astype(np.float64), t.astype(np.float64), C)
    loss, g = ibem.ibem_cnn_gradients(c, xd, td, ibem.IBEM_FP32)
    assert loss == pytest.approx(loss0, rel=1e-6)
    off = 0
    for ci, co in cnn.layer_channels(C):
        for k in (co * ci * 9, co):
            assert np.linalg.norm(g[off:off + k] - g0[off:off + k]) <= 1e-4 * np.linalg.norm(g0[off:off + k])
            off += k
    again, g1 = ibem.ibem_cnn_gradients(c, xd, td, ibem.IBEM_FP32)
    assert again == loss and np.array_equal(g, g1)
    ibem.ibem_cnn_destroy(c)
