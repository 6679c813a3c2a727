"""Meshes that do not coarsen and are too large for the one-launch solve: their only level is both
the finest and the coarsest, so the conjugate gradients' result is the cycle's correction.  The
potential against the FP64 oracle, explicit and implicit."""
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


@pytest.mark.parametrize("implicit", [0, 1])
@pytest.mark.parametrize("bc", [(D, P), (P, P), (D, N)])
@pytest.mark.parametrize("nx,ny", [(91, 91), (129, 65), (231, 37), (64, 131)])
def test_potential_matches_the_oracle(nx, ny, bc, implicit):
    n, h = nx * ny, 2.0 ** -6
    rng = np.random.default_rng(nx + ny)
    # neutral on average, so that the potential stays within the residual's FP64 floor
    cfg = W.base_config(precision=W.FP64, n_species=1, q=[-1.0], m=[1.0], dt=0.5, bc_x=bc[0], bc_y=bc[1],
                        implicit=implicit, rho_background=1.0, phi_left_dc=0.0 if bc[0] != D else 0.02, mg_rel_tol=1e-10,
                        mg_max_cycles=60)
    z = np.zeros(n)
    parts = dict(x=rng.random(n) * nx * h, y=rng.random(n) * ny * h, vx=z, vy=z, vz=z, w=np.full(n, h * h))
    with G.Context(cfg) as ctx:
        ctx.set_mesh(nx0=nx, ny0=ny, h0=h)
        ctx.load(0, **parts)
        ctx.compute_fields()
        a = ctx.fields(G.PIC_FIELD_PHI)
        ctx.compute_fields()  # the warm start: the solution already
        b = ctx.fields(G.PIC_FIELD_PHI)
    sim = O.Sim(cfg, O.Mesh(nx, ny, h, 0, bc[0], bc[1]))
    sim.load(0, **parts)
    sim.fields()
    # ||e|| <= tol ||b|| / lambda_min, ||b|| <= 8 kappa_max ||phi||; lambda_min of half a wave across
    # the mesh (kappa >= 1), kappa = 1 + dt^2 (density)
    lam = 2.0 - 2.0 * np.cos(np.pi / max(nx, ny))
    kmax = 1.0 + implicit * 0.25 * sim.counts(0).max()
    bar = (1e-10 * 8.0 + 1e-13) * kmax / lam
    for p in (a, b):
        assert np.linalg.norm(p - sim.phi) <= bar * np.linalg.norm(sim.phi)
