"""Leaves that move to the tail of the buffer, by blocks and by warps: the lists afterwards, record by
record and in order (staying records in their order, then entering ones in that of the old lists),
with every word of the records, alone and in an ensemble's captured step."""
import numpy as np
import pytest

import paper_1604_07713_gb300 as G
from paper_1604_07713_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [W.FP32, W.FP64])
@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("moved", [1, 31, 152, 153, 700])
def test_lists_after_tail_moves(moved, batch, precision):
    G.build()
    nx, ny, per, h = 64, 32, 300, 2.0 ** -5
    rng = np.random.default_rng(moved)
    dest = np.sort(rng.permutation(nx * ny // 2)[:moved] * 2)  # no two neighbours: each takes 300 records, 91 free slots
    leaf = rng.permutation(np.repeat(np.arange(nx * ny), per))  # (load order mixes the leaves)
    n = leaf.size
    f32 = lambda a: a.astype(np.float32).astype(np.float64)
    u, v = rng.integers(100, 900, (2, n)) / 1024.0  # exact in either precision, also after a cell's move
    vx = np.where(np.isin(leaf, (dest - 1) % nx + dest // nx * nx), h, 0.0)
    p = dict(x=(leaf % nx + u) * h, y=(leaf // nx + v) * h, vx=vx, vy=np.zeros(n), vz=f32(rng.standard_normal(n)),
             w=f32(0.5 + rng.random(n)))
    cfg = W.base_config(precision=precision, n_species=1, q=[0.0], m=[1.0], dt=1.0, max_level=0)
    copies = 2 if batch else 1
    with G.Context([dict(cfg, instance=k) for k in range(copies)]) as ctx:
        for k in range(copies):
            ctx.set_mesh(nx0=nx, ny0=ny, h0=h, inst=k)
            ctx.load(0, **p, inst=k)
        for _ in range(copies):  # (an ensemble's second step is a replay)
            ctx.step(1, allow_notconv=True)
        got = ctx.particles(0, inst=copies - 1)
        assert G.pic_get_list_stats(ctx.ctx, copies - 1, 0)[1] >= moved
    order = np.argsort(leaf, kind="stable")  # the loaded lists
    for _ in range(copies):
        old = leaf
        leaf = np.where(vx > 0, (old % nx + 1) % nx + old // nx * nx, old)
        order = order[np.lexsort((np.arange(n), (leaf != old)[order], leaf[order]))]
    assert np.array_equal(got["id"], order) and np.array_equal(got["leaf"], leaf[order])
    x = np.mod(p["x"] + copies * vx, nx * h)
    for k, want in (("x", x), ("y", p["y"]), ("vx", vx), ("vy", p["vy"]), ("vz", p["vz"]), ("w", p["w"])):
        assert np.array_equal(got[k], want[order]), k
