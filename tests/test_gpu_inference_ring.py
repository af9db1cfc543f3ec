"""Tensor-core inference (runs of 512 padded positions, one persistent CTA per SM) over
many runs per CTA: its ring of bands wraps, both accumulator sets are reused, images
end inside a run.  Against the same images one at a time and the oracle."""
import numpy as np
import pytest

from gpu_common import lib

pytestmark = pytest.mark.gpu


# 7 to 24 runs per SM; rings of 4, 4, 3, 2 and 1 bands
@pytest.mark.parametrize("n,H,W", [(96, 130, 130), (530, 16, 57), (40, 60, 240), (20, 100, 490), (4, 380, 1200)])
def test_inference_of_many_tiles(n, H, W):
    import torch
    from oracle import cnn
    ibem = lib()
    c = ibem.ibem_cnn_create(32, seed=5)
    p = ibem.ibem_cnn_params(c).astype(np.float64)
    x = torch.from_numpy(np.random.default_rng(1910 + W).normal(size=(n, 2, H, W)).astype(np.float32)).cuda()
    out, again = torch.full_like(x, np.nan), torch.full_like(x, np.nan)
    ibem.ibem_cnn_forward(c, x, out, ibem.IBEM_BF16)
    ibem.ibem_cnn_forward(c, x, again, ibem.IBEM_BF16)
    assert ibem.ibem_cnn_device_status(c) == ibem.IBEM_DEVICE_OK
    assert torch.equal(out, again)
    one = torch.full_like(x[:1], np.nan)
    for i in range(0, n, max(1, n // 40)):
        ibem.ibem_cnn_forward(c, x[i:i + 1].contiguous(), one, ibem.IBEM_BF16)
        assert torch.equal(one[0], out[i]), i
    i = n - 1
    ref = cnn.forward(p, x[i:i + 1, :, :, :].cpu().numpy().astype(np.float64), 32)
    assert np.linalg.norm(out[i:i + 1].cpu().numpy() - ref) < 2e-2 * np.linalg.norm(ref)
    ibem.ibem_cnn_destroy(c)
