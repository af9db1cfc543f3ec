"""Interaction lists by one walk per point (many points) and by one per point and
patch (few): the same lists in the same order, so the same bits."""
import numpy as np
import pytest

from gpu_common import lib, rel_err

pytestmark = pytest.mark.gpu
N = 8192 + 37      # one walk per point beyond 8192


@pytest.mark.parametrize("kernel", [0, 1])
def test_many_points_equal_few(kernel):
    import torch
    ibem = lib()
    h = ibem.ibem_create(ibem.sphere_patches(), ibem.make_params(1, 3, q_cheb=4, eta=1.6, kernel=kernel,
                                                                 kappa=2.0 if kernel else 0.0))
    rng = np.random.default_rng(2000 + kernel)
    tail = (2,) if kernel else ()
    w = torch.from_numpy(rng.normal(size=(2, ibem.ibem_get_info(h).ndof) + tail)).cuda()
    P = rng.normal(size=(N, 3))
    P *= (rng.uniform(1.02, 4.0, size=N) / np.linalg.norm(P, axis=1))[:, None]
    pts = torch.from_numpy(P).cuda()

    def potential(points):
        u = torch.full((2, points.shape[0]) + tail, np.nan, dtype=torch.float64, device="cuda")
        counts = ibem.ibem_potential_fmm(h, w, 2, points, u)
        torch.cuda.synchronize()
        return u, counts

    u, counts = potential(pts)
    parts = [potential(pts[a:b].contiguous()) for a, b in ((0, 4000), (4000, N))]
    assert torch.equal(u, torch.cat([p[0] for p in parts], dim=1))
    assert counts == tuple(sum(p[1][k] for p in parts) for k in (0, 1))
    # the point sources of the adjoint: lists by the same walks, sums over all sources
    c = torch.from_numpy(rng.normal(size=(2, N) + tail)).cuda()

    def rhs(a, b):
        out = torch.full_like(w, np.nan)
        n = ibem.ibem_rhs_sources(h, pts[a:b].contiguous(), c[:, a:b].contiguous(), 2, out)
        torch.cuda.synchronize()
        return out.cpu().numpy(), n

    b0, n0 = rhs(0, N)
    b1, n1 = rhs(0, 4000)
    b2, n2 = rhs(4000, N)
    assert n0 == tuple(p + q for p, q in zip(n1, n2)) == counts
    assert rel_err(b1 + b2, b0) < 1e-12
    ibem.ibem_destroy(h)
