"""List repairs: a run whose lists are laid out again, in steps where some leaves still found
room at the tail and others did not, equals the run that never needs it, bit for bit; and the
step's scans at the edges of their tiles."""
import numpy as np
import pytest

import paper_1604_07713_gb300 as G
from paper_1604_07713_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    G.build()


def _run(cfg, mesh, parts, steps):
    with G.Context(cfg) as ctx:
        ctx.set_mesh_dict(mesh)
        for s in sorted(parts):
            ctx.load(s, **parts[s])
        ctx.step(steps)
        return ([ctx.particles(s) for s in sorted(parts)], [G.pic_get_list_stats(ctx.ctx, 0, s) for s in sorted(parts)])


@pytest.mark.parametrize("precision", [W.FP32, W.FP64])
@pytest.mark.parametrize("room", [1.02, 1.2])
def test_relayout_with_leaves_that_moved_in_the_same_step(precision, room):
    cfg, mesh, parts = W.ccp(nx=128, ny=16, ppc=60, seed=4, precision=precision, te=6.0, volt=400.0)
    cfg["sigma_iz0"] = 0.0
    n = parts[0]["x"].size
    cfg["particle_capacity"] = int(room * n)
    tight, stats = _run(cfg, mesh, parts, 40)
    assert stats[0][0] >= 1 and stats[0][1] > stats[0][0]
    cfg["particle_capacity"] = 20 * n
    loose, stats = _run(cfg, mesh, parts, 40)
    assert stats[0][0] == 0
    for a, b in zip(tight, loose):
        for k in a:
            assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("nx,ny", [(2, 2), (31, 33), (32, 32), (41, 25), (64, 64), (2050, 2)])
def test_list_ranks_and_spawn_ids_at_tile_edges(nx, ny):
    """Every electron ionizes in the step (certain collision, elastic section 0): pair ids follow
    the parents' list ranks, which the scans over leaves give."""
    rng = np.random.default_rng(nx * 7 + ny)
    h, n = 2.0 ** -10, 3 * nx * ny + 1
    cfg = W.base_config(precision=W.FP64, dt=1e-12, eps0=W.EPS0, q=[-W.QE, W.QE], m=[W.ME, 4 * W.AMU], qe=W.QE, mcc=1,
                        bc_x=W.BC_PERIODIC, bc_y=W.BC_PERIODIC, gas_density=1e33, neutral_mass=4 * W.AMU, sigma_el=0.0,
                        sigma_iz0=1e-20, eps_th_ev=1e-3, mg_rel_tol=1e-6)
    v = rng.standard_normal((3, n)) * 1e6
    p = dict(x=rng.random(n) * nx * h, y=rng.random(n) * ny * h, vx=v[0], vy=v[1], vz=v[2], w=np.ones(n))
    with G.Context(cfg) as ctx:
        ctx.set_mesh(nx0=nx, ny0=ny, h0=h)
        for s in (0, 1):
            ctx.load(s, **p)
        before = ctx.particles(0)
        ctx.step(1, allow_notconv=True)
        e, i = ctx.particles(0), ctx.particles(1)
    assert e["id"].size == 2 * n and i["id"].size == 2 * n
    # the parent of list rank r has pair ids 2 n + 2 r (electron), + 1 (ion), at the parent's position
    pos = {int(a): (x, y) for a, x, y in zip(e["id"], e["x"], e["y"])}
    ions = {int(a): (x, y) for a, x, y in zip(i["id"], i["x"], i["y"])}
    for r, parent in enumerate(before["id"]):
        assert pos[2 * n + 2 * r] == ions[2 * n + 2 * r + 1] == pos[int(parent)]
