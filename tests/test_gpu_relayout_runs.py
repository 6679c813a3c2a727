"""The re-layout's runs of leaves at their edges (one run, ragged and empty last runs, exact fits), with
and without room for a further step's inflow, alone and in the captured step of an ensemble: runs
that are laid out again equal, bit for bit, the runs whose buffers have room."""
import numpy as np
import pytest

import paper_1604_07713_gb300 as G
from paper_1604_07713_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    G.build()


def _run(nx, ny, precision, shape, room, instances, steps=20):
    """A periodic box of 24 records a leaf (22 free slots), most of which change leaf in every step."""
    rng, n, h = np.random.default_rng(nx), 24 * nx * ny, 2.0 ** -5
    cfg = W.base_config(precision=precision, n_species=1, q=[1e-30], m=[1.0], dt=1.0, shape=shape,
                        particle_capacity=int(room * n))
    p = dict(x=rng.random(n) * nx * h, y=rng.random(n) * ny * h, vz=np.ones(n), w=np.ones(n))
    p["vx"], p["vy"] = rng.standard_normal((2, n)) * 2.0 * h
    with G.Context([dict(cfg, instance=k) for k in range(instances)]) as ctx:
        for k in range(instances):
            ctx.set_mesh(nx0=nx, ny0=ny, h0=h, inst=k)
            ctx.load(0, **p, inst=k)
        for _ in range(steps):
            ctx.step(1, allow_notconv=True)
        return ([ctx.particles(0, inst=k) for k in range(instances)],
                [G.pic_get_list_stats(ctx.ctx, k, 0)[0] for k in range(instances)])


# 8 leaves (one run), 80 (ten of 8), 610 (the last of 2), 4864 (608 of 8 exactly), 4900 (runs of 9,
# the last ones empty)
@pytest.mark.parametrize("nx,ny", [(4, 2), (16, 5), (61, 10), (304, 16), (70, 70)])
@pytest.mark.parametrize("precision", [W.FP32, W.FP64])
@pytest.mark.parametrize("room", [1.02, 2.0])
def test_relayout(nx, ny, precision, room):
    tight, n = _run(nx, ny, precision, G.PIC_SHAPE_NGP, room, 1)
    assert n[0] >= 1
    loose, n = _run(nx, ny, precision, G.PIC_SHAPE_NGP, 60.0, 1)
    assert n[0] == 0
    _same(tight, loose)


def test_relayout_in_a_captured_step_on_branches():
    tight, n = _run(16, 5, W.FP32, G.PIC_SHAPE_CIC_EC, 1.02, 3)
    assert min(n) >= 1
    loose, n = _run(16, 5, W.FP32, G.PIC_SHAPE_CIC_EC, 60.0, 3)
    assert max(n) == 0
    _same(tight, loose)


def _same(a, b):
    for p, q in zip(a, b):
        for k in p:
            assert np.array_equal(p[k], q[k]), k
