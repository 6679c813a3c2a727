"""The scans' second forms: a lattice of more than 2048 tiles (mesh construction) and a mesh of more
than 2048 tiles of leaves (list ranks and spawn offsets of a step)."""
import numpy as np
import pytest

import oracle as O
import paper_1604_07713_gb300 as G
from paper_1604_07713_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    G.build()
    O.build()


def test_mesh_of_a_lattice_of_many_tiles():
    nx, ny, lmax, h = 64, 40, 6, 0.5  # 1.05e7 lattice cells
    r, lv, m = W.region_tree(nx, ny, lmax, lambda l, x, y, s: abs(x - 31.3) < s and abs(y - 17.6) < s)
    assert lv.max() == lmax
    p = np.random.default_rng(1).permutation(r.size)
    cfg = W.base_config(precision=W.FP64, n_species=1, q=[-1.0], m=[1.0], bc_x=W.BC_DIRICHLET, bc_y=W.BC_NEUMANN, max_level=lmax)
    M = O.Mesh(nx, ny, h, lmax, W.BC_DIRICHLET, W.BC_NEUMANN, r, lv, m)
    rng = np.random.default_rng(2)
    x, y = rng.random(5000) * M.lx, rng.random(5000) * M.ly
    x[:2000], y[:2000] = 31.3 * h + rng.normal(0, 0.2, 2000), 17.6 * h + rng.normal(0, 0.2, 2000)
    z = np.zeros(x.size)
    with G.Context(cfg) as ctx:
        ctx.set_mesh(nx0=nx, ny0=ny, h0=h, root=r[p], morton=m[p], level=lv[p])
        a, b, c = ctx.mesh()
        assert np.array_equal(a, M.root) and np.array_equal(b, M.morton) and np.array_equal(c, M.level)
        ctx.load(0, x, y, z, z, z, np.ones(x.size))
        assert np.array_equal(np.bincount(M.locate(x, y), minlength=M.nleaf), ctx.fields(G.PIC_FIELD_COUNT_E))


def test_ranks_and_spawn_ids_of_many_leaves():
    """Every electron ionizes in the step (certain collision, no elastic part): pair ids follow the
    parents' list ranks over 2.16e6 leaves."""
    nx, ny, h, n = 1536, 1408, 2.0 ** -10, 300_000
    rng = np.random.default_rng(3)
    cfg = W.base_config(precision=W.FP64, dt=1e-12, eps0=W.EPS0, q=[0.0, 0.0], m=[W.ME, 4 * W.AMU], qe=W.QE, mcc=1,
                        bc_x=W.BC_PERIODIC, bc_y=W.BC_PERIODIC, gas_density=1e33, neutral_mass=4 * W.AMU, sigma_el=0.0,
                        sigma_iz0=1e-20, eps_th_ev=1e-3, mg_rel_tol=1e-6)
    v = rng.standard_normal((3, n)) * 1e6
    p = dict(x=rng.random(n) * nx * h, y=rng.random(n) * ny * h, vx=v[0], vy=v[1], vz=v[2], w=np.ones(n))
    leaf = np.floor(p["x"] / h).astype(int) + nx * np.floor(p["y"] / h).astype(int)
    with G.Context(cfg) as ctx:
        ctx.set_mesh(nx0=nx, ny0=ny, h0=h)
        for s in (0, 1):
            ctx.load(s, **p)
        before = ctx.particles(0)
        ctx.step(1, allow_notconv=True)
        e, i = ctx.particles(0), ctx.particles(1)
    assert np.array_equal(before["id"], np.argsort(leaf, kind="stable"))
    assert e["id"].size == 2 * n and i["id"].size == 2 * n
    # the parent of list rank r has pair ids 2 n + 2 r (electron), + 1 (ion), at the parent's position
    xy = [dict(zip(("id", "x", "y"), (q["id"][o], q["x"][o], q["y"][o]))) for q in (e, i) for o in [np.argsort(q["id"])]]
    parent = np.searchsorted(xy[0]["id"], before["id"])
    pairs = np.searchsorted(xy[0]["id"], 2 * n + 2 * np.arange(n)), np.searchsorted(xy[1]["id"], 2 * n + 2 * np.arange(n) + 1)
    assert np.array_equal(xy[0]["id"][pairs[0]], 2 * n + 2 * np.arange(n))
    assert np.array_equal(xy[1]["id"][pairs[1]], 2 * n + 2 * np.arange(n) + 1)
    for k in ("x", "y"):
        assert np.array_equal(xy[0][k][pairs[0]], xy[0][k][parent]) and np.array_equal(xy[1][k][pairs[1]], xy[0][k][parent])
