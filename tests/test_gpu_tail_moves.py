"""Leaves that run out of free slots, from one to more than the repair's blocks in a step (a block
for each, then a warp for each), with lists longer than a block: the run equals the one whose
lists had room, bit for bit, alone and in an ensemble's captured step."""
import numpy as np
import pytest

import paper_1604_07713_gb300 as G
from paper_1604_07713_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    G.build()


def _run(nx, ny, dest, per, batch, precision):
    """`per` records per leaf and as many from each leaf's left neighbour for the leaves `dest`:
    (particles by id, leaves moved to the tail)."""
    h = 2.0 ** -5
    cfg = W.base_config(precision=precision, n_species=1, q=[1e-30], m=[1.0], dt=1.0, bc_x=W.BC_PERIODIC,
                        bc_y=W.BC_PERIODIC, max_level=0)
    rng = np.random.default_rng(len(dest))
    leaf = np.repeat(np.arange(nx * ny), per)
    u, v = 0.1 + 0.8 * rng.random(leaf.size), 0.1 + 0.8 * rng.random(leaf.size)
    src = (dest - 1) % nx + (dest // nx) * nx
    vx = np.where(np.isin(leaf, src), h, 0.0)
    z = np.zeros(leaf.size)
    p = dict(x=(leaf % nx + u) * h, y=(leaf // nx + v) * h, vx=vx, vy=z, vz=z, w=np.ones(leaf.size))
    n = 2 if batch else 1
    with G.Context([cfg] * n) as ctx:
        for i in range(n):
            ctx.set_mesh(nx0=nx, ny0=ny, h0=h, inst=i)
            ctx.load(0, **p, inst=i)
        for _ in range(n):  # (an ensemble's second step is a replay; the flying records overflow further leaves)
            ctx.step(1, allow_notconv=True)
        q = ctx.particles(0, inst=n - 1)
        stats = G.pic_get_list_stats(ctx.ctx, n - 1, 0)
    x = np.mod((leaf % nx + u) * h + n * vx, nx * h)
    o = np.argsort(q["id"], kind="stable")
    return x, p, {k: q[k][o] for k in q}, stats


@pytest.mark.parametrize("precision", [W.FP32, W.FP64])
@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("moved", [1, 32, 33, 152, 153, 700])
def test_moves_by_block_and_by_warp(moved, batch, precision):
    nx, ny, per = 64, 32, 300
    dest = np.sort(np.random.default_rng(moved).permutation(nx * ny // 2)[:moved] * 2)  # no two neighbours
    x, p, q, stats = _run(nx, ny, dest, per, batch, precision)
    assert stats[1] >= moved  # each takes 300 records and has 91 free slots
    # every record is there once, where it flew (offsets are in the state's precision)
    assert q["id"].size == x.size and np.all(np.diff(q["id"].astype(np.int64)) == 1)
    tol = 2.0 ** -5 * (2.0 ** -21 if precision == W.FP32 else 2.0 ** -40)
    d = np.abs(q["x"] - x)
    assert np.all(np.minimum(d, nx * 2.0 ** -5 - d) <= tol)
    assert np.all(np.abs(q["y"] - p["y"]) <= tol)
    assert np.array_equal(q["w"], p["w"])
