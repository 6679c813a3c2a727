"""The FP64 push's collision bound, formed in FP32: whatever the units, every collision of the exact
test happens (against the oracle), also where speeds, their squares or energies leave FP32's range
and where the bound cannot be formed and every particle takes the exact test."""
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


# speed scale, electron mass (energy m v^2 / 2 at qe = 1), threshold, elastic and ionization sections,
# collisions per step at the speed scale
CASES = {
    "ordinary": (1.0, 2.0, 0.3, 1.0, 1.0, 0.5),
    "rare": (1.0, 2.0, 0.3, 1.0, 1.0, 1e-3),
    "squares below FP32's range": (1e-22, 2.0, 1e-20, 1.0, 1.0, 0.5),
    "energies below FP32's range, no threshold": (1e-5, 2e-29, 0.0, 0.0, 1.0, 0.5),
    "squares above FP32's range": (1e25, 2.0, 0.3, 1.0, 1.0, 0.5),
    "speeds above FP32's range": (1e45, 2.0, 0.3, 1.0, 1.0, 0.5),
    "sections of very different size": (1.0, 2.0, 0.3, 1e-9, 1.0, 0.5),
    "mass below FP32's range": (1.0, 2e-40, 1e-41, 1.0, 1.0, 0.5),
    "no threshold": (1.0, 2.0, 0.0, 1.0, 1.0, 0.5),
}


@pytest.mark.parametrize("name", CASES)
def test_every_collision_happens(name):
    V, m, th, el, iz, rate = CASES[name]
    rng, n, nx, ny, h = np.random.default_rng(5), 20_000, 12, 9, V
    dt = 0.3
    cfg = W.base_config(precision=W.FP64, n_species=2, q=[0.0, 0.0], m=[m, 4.0 * m], dt=dt, qe=1.0, mcc=1, neutral_mass=4.0 * m,
                        bc_x=W.BC_DIRICHLET, bc_y=W.BC_PERIODIC, gas_density=rate / (V * dt * max(el, iz)),
                        gas_temperature_ev=0.0, sigma_el=el, sigma_iz0=iz, eps_th_ev=th)
    sim = O.Sim(cfg, O.Mesh(nx, ny, h, 0, W.BC_DIRICHLET, W.BC_PERIODIC))
    with G.Context(cfg) as ctx:
        ctx.set_mesh(nx0=nx, ny0=ny, h0=h)
        for s in (0, 1):
            v = rng.standard_normal((3, n)) * V
            # at rest, far below and far above every other speed
            v[:, :200], v[:, 200:400], v[2, 400:600] = 0.0, v[:, 200:400] * 1e-60, V * 1e50
            p = dict(x=rng.random(n) * nx * h, y=rng.random(n) * ny * h, vx=v[0], vy=v[1], vz=v[2], w=np.ones(n))
            sim.load(s, **p)
            ctx.load(s, **p)
        ctx.step(1)
        sim.step(1)
        g = [ctx.particles(s) for s in (0, 1)]
    for s in (0, 1):
        sp = sim.species[s]
        assert np.array_equal(g[s]["id"], sp.id)
        speed = np.sqrt(sp.vx ** 2 + sp.vy ** 2 + sp.vz ** 2)
        for k in ("vx", "vy", "vz"):
            assert np.all(np.abs(g[s][k] - getattr(sp, k)) <= 1e-9 * speed), (s, k)
    d = sim.last_decisions[0][1]
    assert rate * n / 10 < np.count_nonzero(d[:, 0] < d[:, 1]) < n  # the oracle's collisions
