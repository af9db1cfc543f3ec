"""Cubes whose block lists hang on the last bit of a distance: near blocks
formed once for two mirrored pairs and symmetric stored couplings, at 1e-12
against the FP64 oracle on the library's own lists and classes."""
import numpy as np
import pytest

import shapes
from gpu_common import lib, rel_err

pytestmark = pytest.mark.gpu
TOL64 = 1e-12
CLASSES = ("identical", "edge", "vertex", "nearsing", "regular")


def _oracle(ibem, specs, pats, prm, p, m, q, eta, kern):
    from oracle import fmm, galerkin, geometry, tree
    disc = galerkin.Discretisation([geometry.NurbsPatch(*s) for s in specs], p, m, kern, n_regular=4, n_singular=4)
    near, far = ibem.ibem_block_tree(pats, prm)
    op = fmm.FMMOperator(disc, q, eta)
    cell = lambda r: (r[0], m, r[1], r[2])  # noqa: E731
    op.near = [(cell(r[:3]), cell(r[3:6])) for r in near.tolist()]
    op.near_elements = [(tree.element_index(s, m), tree.element_index(t, m)) for s, t in op.near]
    cls = {e: (CLASSES[r[6]], r[7] // 8, r[7] % 8) for e, r in zip(op.near_elements, near.tolist())}
    disc.pair_class = lambda a, b: cls[a, b]
    op.far = [(tuple(r[:4]), tuple(r[4:])) for r in far.tolist()]
    op.far_by_target.clear()
    for s, t in op.far:
        op.far_by_target[s].append(t)
    return op


@pytest.mark.parametrize("cube,eta,p,m", [((1.7, (0.1, 0.2, 0.3), 0.0), 1.5, 1, 1), ((1.7, (0.1, 0.2, 0.3), 0.0), 0.5, 0, 2),
                                          ((2.0 / np.sqrt(3.0), (0.0, 0.0, 0.0), 0.0), 0.5, 1, 2),
                                          ((1.3, (0.4, -0.7, 0.2), 0.7), 0.5, 1, 2),
                                          ((1.0, (0.0, 0.0, 0.0), 0.3), 1.5, 1, 2)])
@pytest.mark.parametrize("kernel", [0, 1])
def test_cubes_against_oracle(kernel, cube, eta, p, m):
    import torch
    from oracle import galerkin
    ibem = lib()
    specs, q = shapes.cube(*cube), 4
    pats = ibem.nurbs_patches(specs)
    prm = ibem.make_params(p, m, q_cheb=q, eta=eta, kernel=kernel, kappa=2.0 if kernel else 0.0,
                           gauss_regular=4, gauss_singular=4)
    op = _oracle(ibem, specs, pats, prm, p, m, q, eta,
                 galerkin.HelmholtzKernel(2.0) if kernel else galerkin.LaplaceKernel())
    h = ibem.ibem_create(pats, prm)
    ibem.ibem_assemble(h)
    rng = np.random.default_rng(1400 + m)
    x = rng.normal(size=op.mesh.n_dofs) + (1j * rng.normal(size=op.mesh.n_dofs) if kernel else 0.0)
    xd = torch.from_numpy(np.stack([x.real, x.imag], -1) if kernel else x).cuda()
    yd = torch.full_like(xd, np.nan)
    ibem.ibem_matvec(h, xd, yd, 1)
    y = yd.cpu().numpy()
    assert rel_err(y[..., 0] + 1j * y[..., 1] if kernel else y, op.matvec(x)) < TOL64
    ibem.ibem_destroy(h)
