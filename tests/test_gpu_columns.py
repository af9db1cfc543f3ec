"""A right-hand side's result does not depend on how many others are applied
with it: columns alone and together, bit for bit, on both sides of every line at
which a launch changes its shape."""
import numpy as np
import pytest

from gpu_common import lib

pytestmark = pytest.mark.gpu


def _handle(p, m, q, kernel, **kw):
    ibem = lib()
    h = ibem.ibem_create(ibem.sphere_patches(), ibem.make_params(p, m, q_cheb=q, eta=1.6, kernel=kernel,
                                                                 kappa=3.0 if kernel else 0.0, **kw))
    ibem.ibem_assemble(h)
    return h


def _vectors(seed, *shape):
    import torch
    return torch.from_numpy(np.random.default_rng(seed).normal(size=shape)).cuda()


def _apply(h, x, precision=0):
    import torch
    y = torch.full_like(x, np.nan)
    lib().ibem_matvec(h, x, y, x.shape[0], precision)
    torch.cuda.synchronize()
    return y


# the larger counts are past the line between groups of lanes and single threads in the restriction
@pytest.mark.parametrize("p,m,q,R", [(0, 3, 3, 200), (1, 3, 4, 170), (2, 4, 4, 24), (3, 3, 5, 40), (4, 3, 4, 24)])
def test_laplace(p, m, q, R):
    import torch
    h = _handle(p, m, q, 0)
    x = _vectors(1800 + p, R, lib().ibem_get_info(h).ndof)
    y = _apply(h, x)
    for r0, n in ((0, 1), (1, 2), (R - 1, 1), (3, 7)):
        assert torch.equal(_apply(h, x[r0:r0 + n].contiguous()), y[r0:r0 + n]), (r0, n)
    lib().ibem_destroy(h)


@pytest.mark.parametrize("kernel", [0, 1])
def test_right_hand_sides(kernel):
    import torch
    ibem = lib()
    h = _handle(2, 4, 4, kernel)
    info = ibem.ibem_get_info(h)
    tail = (2,) if kernel else ()
    g = _vectors(1810 + kernel, 24, info.n_quad_points, *tail)

    def rhs(v):
        b = torch.full((v.shape[0], info.ndof) + tail, np.nan, dtype=torch.float64, device="cuda")
        ibem.ibem_rhs(h, v, v.shape[0], b)
        torch.cuda.synchronize()
        return b

    b = rhs(g)
    for r0, n in ((0, 1), (5, 3), (23, 1)):
        assert torch.equal(rhs(g[r0:r0 + n].contiguous()), b[r0:r0 + n]), (r0, n)
    ibem.ibem_destroy(h)


# passes of the stored Helmholtz coupling: one pass of all, pairs with one left over, and a
# launch too small for that; fewer than four columns take another near product
@pytest.mark.parametrize("p,m,q,R", [(1, 2, 4, 63), (0, 3, 6, 15)])
def test_helmholtz_stored_far_field(p, m, q, R):
    import torch
    h = _handle(p, m, q, 1)
    x = _vectors(1820 + R, R, lib().ibem_get_info(h).ndof, 2)
    for n in (3, 2):
        y = _apply(h, x[:n].contiguous())
        for r in range(n):
            assert torch.equal(_apply(h, x[r:r + 1].contiguous())[0], y[r]), (n, r)
    y = _apply(h, x)
    assert torch.equal(_apply(h, x), y)
    assert float((_apply(h, x[:3].contiguous()) - y[:3]).abs().max()) < 1e-12 * float(y.abs().max())
    lib().ibem_destroy(h)


# FP32 operator of 16 and more columns: 16 to 64 per group of the near product, one to four groups
@pytest.mark.parametrize("kernel,p,m,q", [(0, 2, 3, 4), (0, 3, 2, 6), (1, 2, 3, 4), (1, 3, 2, 8), (1, 1, 3, 4)])
def test_fp32_many(kernel, p, m, q):
    import torch
    h = _handle(p, m, q, kernel)
    x = _vectors(1830 + p, 200, lib().ibem_get_info(h).ndof, *((2,) if kernel else ()))
    y = _apply(h, x, 1)
    for r0, n in ((0, 16), (3, 17), (100, 40), (136, 64), (60, 65), (72, 128)):
        assert torch.equal(_apply(h, x[r0:r0 + n].contiguous(), 1), y[r0:r0 + n]), (r0, n)
    lib().ibem_destroy(h)


# FP64 Helmholtz of four and more columns: one to eight pairs (row, column) per thread, slices side by
# side and (from some 64 columns at p = 3, 113 at p = 2) in turn
@pytest.mark.parametrize("p,m,q,R", [(0, 3, 0, 300), (1, 3, 4, 70), (2, 3, 4, 120), (3, 2, 4, 100), (4, 2, 4, 40)])
def test_helmholtz(p, m, q, R):
    import torch
    h = _handle(p, m, q, 1)
    x = _vectors(1840 + p, R, lib().ibem_get_info(h).ndof, 2)
    y = _apply(h, x)
    for r0, n in ((0, 4), (1, 5), (2, 9), (0, 16), (R - 33, 33)):
        assert torch.equal(_apply(h, x[r0:r0 + n].contiguous()), y[r0:r0 + n]), (r0, n)
    lib().ibem_destroy(h)
