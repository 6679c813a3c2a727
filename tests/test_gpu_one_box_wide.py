"""Meshes one root box wide in a periodic direction, whose unrefined leaves meet themselves across
the wrap, against the FP64 oracle: potential, corner field and |E|, then steps whose particles
cross the whole width, in list order."""
import numpy as np
import pytest

import oracle as O
import paper_1604_07713_gb300 as G
from paper_1604_07713_gb300 import workloads as W

pytestmark = pytest.mark.gpu

P, D, N = W.BC_PERIODIC, W.BC_DIRICHLET, W.BC_NEUMANN


@pytest.fixture(scope="module", autouse=True)
def _built():
    G.build()
    O.build()


@pytest.mark.parametrize("precision", [W.FP64, W.FP32])
@pytest.mark.parametrize("lmax", [0, 1, 3])
@pytest.mark.parametrize("nx,ny,bc", [(1, 7, (P, D)), (1, 6, (P, P)), (9, 1, (D, P)), (1, 1, (P, P)), (1, 2, (P, D))])
def test_fields_and_steps_match_the_oracle(nx, ny, bc, lmax, precision):
    rng, h, n = np.random.default_rng(nx + ny + lmax), 0.5, 400
    r, lv, m = W.random_tree(nx, ny, lmax, 0.35, 3 + lmax, bc[0] == P, bc[1] == P)
    tol = 1e-12 if precision == W.FP64 else 1e-8
    cfg = W.base_config(precision=precision, n_species=1, q=[-1.0], m=[1.0], dt=0.05, bc_x=bc[0], bc_y=bc[1],
                        max_level=lmax, rho_background=1.0, phi_left_dc=0.2 if bc[0] == D else 0.0, mg_rel_tol=tol)
    v = rng.standard_normal((3, n)) * 6.0  # up to several widths a step
    parts = dict(x=rng.random(n) * nx * h, y=rng.random(n) * ny * h, vx=v[0], vy=v[1], vz=v[2],
                 w=np.full(n, nx * ny * h * h / n))
    sim = O.Sim(cfg, O.Mesh(nx, ny, h, lmax, bc[0], bc[1], r, lv, m))
    sim.load(0, **parts)
    with G.Context(cfg) as ctx:
        ctx.set_mesh(nx0=nx, ny0=ny, h0=h, root=r, level=lv, morton=m)
        ctx.load(0, **parts)
        ctx.compute_fields()
        phi, e, emag = (ctx.fields(f) for f in (G.PIC_FIELD_PHI, G.PIC_FIELD_NODE_E, G.PIC_FIELD_EMAG))
        sim.fields()
        # solves to tol of ||b||: the smallest eigenvalue of these meshes is above 0.05 / 4^lmax; the
        # field from differences of phi over the finest side, in the state's precision
        scale = max(np.abs(sim.phi).max(), 1e-3)
        bar = (tol * 200.0 + 1e-13) * 4.0 ** lmax * scale
        assert np.abs(phi - sim.phi).max() <= bar
        E = sim.last_node_e.reshape(e.shape)
        rnd = 1e-13 if precision == W.FP64 else 1e-6
        hf = h / 2 ** lmax
        assert np.abs(e - E).max() <= 4.0 * (bar + rnd * scale) / hf
        assert np.abs(emag - sim.mesh.cell_emag(sim.phi, sim.walls())).max() <= 4.0 * (bar + 1e-13 * scale) / hf
        for _ in range(3):
            ctx.step(1)
            sim.step(1)
        g = ctx.particles(0)
    sp = sim.species[0]
    if precision == W.FP64:
        assert np.array_equal(g["id"], sp.id) and np.array_equal(g["leaf"].astype(np.int64), sp.leaf)
        for k in ("x", "y", "vx", "vy"):
            assert np.abs(g[k] - getattr(sp, k)).max() <= 1e-6, k
    else:
        common, a, b = np.intersect1d(g["id"], sp.id, return_indices=True)
        assert common.size >= 0.99 * max(sp.n, g["id"].size)
        for k, L in (("x", nx * h), ("y", ny * h)):
            d = np.abs(g[k][a] - getattr(sp, k)[b])
            assert np.quantile(np.minimum(d, L - d), 0.99) <= 1e-4
