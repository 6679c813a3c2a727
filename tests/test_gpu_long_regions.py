"""Entering regions of more than 512 records, which whole blocks sort, in the lists of either or both
species, in more leaves than there are blocks and in fewer: list order against the oracle."""
import numpy as np
import pytest

import oracle as O
import paper_1604_07713_gb300 as G
from paper_1604_07713_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [W.FP32, W.FP64])
@pytest.mark.parametrize("nx,ny,long", [(20, 16, (0,)), (20, 16, (1,)), (20, 16, (0, 1)), (6, 4, (0, 1)), (6, 4, ())])
def test_list_order(nx, ny, long, precision):
    G.build()
    O.build()
    h, rng = 2.0 ** -4, np.random.default_rng(nx + sum(long))
    cfg = W.base_config(precision=precision, n_species=2, q=[0.0, 0.0], m=[1.0, 4.0], dt=1.0)
    sim = O.Sim(cfg, O.Mesh(nx, ny, h, 0, W.BC_PERIODIC, W.BC_PERIODIC))
    with G.Context(cfg) as ctx:
        ctx.set_mesh(nx0=nx, ny0=ny, h0=h)
        for s in (0, 1):
            n = nx * ny * (900 if s in long else 40)
            # exact in either precision: offsets in 1/1024, whole cells a step (a few stay)
            x, y = rng.integers(0, nx * 1024, n) * h / 1024, rng.integers(0, ny * 1024, n) * h / 1024
            v = rng.integers(-2, 3, (2, n)) * h
            p = dict(x=x, y=y, vx=v[0], vy=v[1], vz=np.zeros(n), w=np.ones(n))
            sim.load(s, **p)
            ctx.load(s, **p)
        for _ in range(2):
            ctx.step(1)
            sim.step(1)
        for s in (0, 1):
            g, sp = ctx.particles(s), sim.species[s]
            if s in long:  # regions as long as the test is about
                assert np.median(sim.counts(s)) > 850
            assert np.array_equal(g["id"], sp.id) and np.array_equal(g["leaf"].astype(np.int64), sp.leaf)
            for k in ("x", "y", "vx", "vy"):
                assert np.array_equal(g[k], getattr(sp, k)), (s, k)
