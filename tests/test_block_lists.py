"""The near and far lists are symmetric, classes and Gauss orders included: one
of two mirrored blocks is formed and stored for both.  Cubes at several sizes,
places and angles, where rounding decides ties of distance against diameter; the
library's host tree and the oracle's."""
import numpy as np
import pytest

import shapes

CUBES = [(1.7, (0.1, 0.2, 0.3), 0.0), (2.0 / np.sqrt(3.0), (0.0, 0.0, 0.0), 0.0), (1.0, (0.0, 0.0, 0.0), 0.3),
         (1.3, (0.4, -0.7, 0.2), 0.7)]


@pytest.fixture(scope="module")
def ibem():
    from paper_1708_09162_gb300 import build
    build.build()
    from paper_1708_09162_gb300 import ibem as mod
    return mod


@pytest.mark.parametrize("m", [1, 2, 3])
@pytest.mark.parametrize("eta", [0.5, 1.0, 1.5])
def test_lists_are_symmetric(ibem, eta, m):
    for cube in CUBES:
        pats = ibem.nurbs_patches(shapes.cube(*cube))
        prm = ibem.make_params(1, m, q_cheb=4, eta=eta, gauss_regular=4, gauss_grading=2)
        near, far = ibem.ibem_block_tree(pats, prm)
        pairs = {tuple(r[:6]): (r[6], o) for r, o in zip(near.tolist(), ibem.ibem_near_orders(pats, prm).tolist())}
        assert all(pairs.get(k[3:] + k[:3]) == v for k, v in pairs.items()), cube
        blocks = set(map(tuple, far.tolist()))
        assert all(k[4:] + k[:4] in blocks for k in blocks), cube


@pytest.mark.parametrize("eta", [0.5, 1.0, 1.5])
def test_oracle_lists_are_symmetric(eta):
    from oracle import galerkin, geometry, tree
    for cube in CUBES:
        patches = [geometry.NurbsPatch(*s) for s in shapes.cube(*cube)]
        for blocks in tree.block_cluster_tree(patches, 2, eta):
            assert set(blocks) == {(t, s) for s, t in blocks}, cube
        disc = galerkin.Discretisation(patches, 1, 1, galerkin.LaplaceKernel(), n_regular=4, grading=2)
        for a in range(disc.mesh.n_elements):
            for b in range(a):
                assert disc.pair_class(a, b)[0] == disc.pair_class(b, a)[0], (cube, a, b)
                assert disc.pair_order(a, b) == disc.pair_order(b, a), (cube, a, b)
