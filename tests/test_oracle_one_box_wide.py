"""The oracle's corner field on meshes one root box wide in a periodic direction, whose unrefined
leaves meet themselves across the wrap: it equals the field of the same mesh twice side by side."""
import numpy as np
import pytest

import oracle as O
from paper_1604_07713_gb300 import workloads as W

P, D, N = W.BC_PERIODIC, W.BC_DIRICHLET, W.BC_NEUMANN


@pytest.fixture(scope="module", autouse=True)
def _built():
    O.build()


@pytest.mark.parametrize("nx,ny,bc", [(1, 5, (P, D)), (1, 4, (P, P)), (5, 1, (N, P)), (3, 1, (P, P)), (1, 1, (P, P)), (1, 1, (P, D))])
@pytest.mark.parametrize("lmax", [0, 1, 2, 3])
def test_equals_the_mesh_twice(nx, ny, bc, lmax):
    rng = np.random.default_rng(nx + 10 * ny + lmax)
    r, lv, m = W.random_tree(nx, ny, lmax, 0.35, 3 + lmax, bc[0] == P, bc[1] == P)
    one = O.Mesh(nx, ny, 0.5, lmax, bc[0], bc[1], r, lv, m)
    cx, cy = 1 + (bc[0] == P), 1 + (bc[1] == P)
    copies = [(a, b) for b in range(cy) for a in range(cx)]
    root = np.concatenate([(r % nx + a * nx) + (r // nx + b * ny) * (nx * cx) for a, b in copies])
    two = O.Mesh(nx * cx, ny * cy, 0.5, lmax, bc[0], bc[1], root, np.tile(lv, len(copies)), np.tile(m, len(copies)))
    phi = rng.standard_normal(one.nleaf)
    walls = (0.3, -0.2, 0.1, 0.7)
    x, y = two.centres()
    src = one.locate(np.mod(x, nx * 0.5), np.mod(y, ny * 0.5))
    e1, e2 = one.node_e(phi, walls).reshape(-1, 8), two.node_e(phi[src], walls).reshape(-1, 8)
    assert np.array_equal(e1[src], e2)
