"""A population that doubles every step, so that the buffers' bound needs each step's counts: one
call of several steps equals as many calls of one, bit for bit, while the buffers grow."""
import numpy as np
import pytest

import paper_1604_07713_gb300 as G
from paper_1604_07713_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    G.build()


def _cfg(precision, shape, **kw):
    # every electron ionizes in every step: a certain collision, no elastic part
    return W.base_config(**(dict(precision=precision, shape=shape, dt=1e-12, eps0=W.EPS0, q=[-W.QE, W.QE],
                                 m=[W.ME, 4 * W.AMU], qe=W.QE, mcc=1, bc_x=W.BC_PERIODIC, bc_y=W.BC_PERIODIC,
                                 gas_density=1e33, neutral_mass=4 * W.AMU, sigma_el=0.0, sigma_iz0=1e-20, eps_th_ev=1e-3,
                                 mg_rel_tol=1e-6) | kw))


def _run(cfgs, n, calls):
    nx, ny, h = 24, 16, 2.0 ** -10
    out = []
    with G.Context(cfgs) as ctx:
        for i in range(len(cfgs)):
            rng = np.random.default_rng(i)
            v = rng.standard_normal((3, n)) * 3e6
            p = dict(x=rng.random(n) * nx * h, y=rng.random(n) * ny * h, vx=v[0], vy=v[1], vz=v[2], w=np.full(n, 1e-3))
            ctx.set_mesh(nx0=nx, ny0=ny, h0=h, inst=i)
            for s in (0, 1):
                ctx.load(s, **p, inst=i)
        for k in calls:
            ctx.step(k, allow_notconv=True)
        for i in range(len(cfgs)):
            out += [ctx.particles(s, inst=i) for s in (0, 1)]
    return out


@pytest.mark.parametrize("instances,shape", [(1, 0), (3, 0), (2, 1)])
@pytest.mark.parametrize("precision", [W.FP32, W.FP64])
def test_one_call_equals_single_steps(precision, instances, shape):
    cfgs = [_cfg(precision, shape) for _ in range(instances)]
    if instances > 2:
        cfgs[1]["sigma_iz0"] = 0.0  # an instance that never grows among those that do
    n = 40_000
    a, b = _run(cfgs, n, [6]), _run(cfgs, n, [1] * 6)
    assert a[0]["id"].size > 32 * n  # (a few fall below the threshold)
    for p, q in zip(a, b):
        for k in p:
            assert np.array_equal(p[k], q[k]), k


def test_a_fixed_capacity_is_enforced_within_a_call():
    cfg = _cfg(W.FP32, 0, particle_capacity=300_000)
    assert 120_000 < _run([cfg], 40_000, [2])[0]["id"].size <= 160_000
    for calls in ([4], [2, 2]):
        with pytest.raises(G.PicError) as e:
            _run([cfg], 40_000, calls)
        assert "PIC_ECAPACITY" in str(e.value)
