"""Particles that leave their leaf on a mesh of root boxes only, where the new leaf follows from the
lattice cell, against the same boxes in a mesh that may refine, where it is looked up: bit for
bit, for displacements up to several periods, offsets that land on faces, and every wall."""
import numpy as np
import pytest

import paper_1604_07713_gb300 as G
from paper_1604_07713_gb300 import workloads as W

pytestmark = pytest.mark.gpu

P, D, N = W.BC_PERIODIC, W.BC_DIRICHLET, W.BC_NEUMANN


@pytest.mark.parametrize("precision", [W.FP32, W.FP64])
@pytest.mark.parametrize("bc", [(P, P), (D, P), (P, N), (D, N)])
def test_new_leaf_from_the_lattice_cell(bc, precision):
    G.build()
    nx, ny, h, n = 18, 10, 2.0 ** -5, 6000
    rng = np.random.default_rng(11)
    reach = np.exp(rng.uniform(np.log(1e-6), np.log(50.0), n)) * h  # per step, dt = 1
    phi = rng.random(n) * 2.0 * np.pi
    x, y = rng.random(n) * nx * h, rng.random(n) * ny * h
    vx, vy = reach * np.cos(phi), reach * np.sin(phi)
    # on a face, moving whole cells (never zero: an offset of 0 would show the fields' last bits)
    x[:500], vx[:500] = rng.integers(0, nx, 500) * h, (2 * rng.integers(-20, 20, 500) + 1) * h
    y[500:1000], vy[500:1000] = rng.integers(0, ny, 500) * h, (2 * rng.integers(-20, 20, 500) + 1) * h
    root = rng.permutation(nx * ny).astype(np.uint32)
    z = np.zeros(nx * ny, np.uint32)
    out = []
    for lmax in (0, 1):
        # (no field: the charge is far below what moves a velocity)
        cfg = W.base_config(precision=precision, n_species=1, q=[1e-30], m=[1.0], dt=1.0, bc_x=bc[0], bc_y=bc[1],
                            max_level=lmax)
        with G.Context(cfg) as ctx:
            ctx.set_mesh(nx0=nx, ny0=ny, h0=h, root=root, morton=z, level=z.astype(np.uint8))
            ctx.load(0, x, y, vx, vy, np.ones(n), np.ones(n))
            for _ in range(4):
                ctx.step(1, allow_notconv=True)
            out.append(ctx.particles(0))
    assert out[0]["id"].size == out[1]["id"].size > 0
    for k in out[0]:
        assert np.array_equal(out[0][k], out[1][k]), k
