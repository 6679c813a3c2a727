"""The one-launch Poisson solve at the sizes where its level storage, thread counts, coarsest
solver and cluster split change, against the FP64 oracle."""
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


# (nx, ny): a single level (direct; CG), coarsest levels of 1 and 2 cells width, direct solves up
# to 128 cells and CG beyond, 1, 2 and 4 cells of a colour per thread, a ragged last warp, the
# largest mesh of the solver
@pytest.mark.parametrize("bc", [(D, P), (P, P), (P, D), (D, N)])
@pytest.mark.parametrize("nx,ny", [(4, 4), (11, 11), (33, 9), (2, 16), (16, 2), (6, 4), (32, 4), (40, 20), (60, 44),
                                   (208, 24), (34, 66), (96, 32), (384, 16), (64, 64), (512, 16)])
def test_solve_matches_the_oracle(nx, ny, bc):
    n = nx * ny * 3
    rng = np.random.default_rng(nx + 1000 * ny)
    h = 2.0 ** -6
    cfg = W.base_config(precision=W.FP64, n_species=1, q=[-1.0], m=[1.0], bc_x=bc[0], bc_y=bc[1], rho_background=0.7,
                        phi_left_dc=0.0 if bc[0] != D else 0.02, phi_right=0.0 if bc[0] != D else -0.01,
                        mg_rel_tol=1e-12, mg_max_cycles=200)
    mesh = dict(nx0=nx, ny0=ny, h0=h, lmax=0)
    z = np.zeros(n)
    parts = dict(x=rng.random(n) * nx * h, y=rng.random(n) * ny * h, vx=z, vy=z, vz=z, w=np.full(n, h * h / 3))
    with G.Context(cfg) as ctx:
        ctx.set_mesh_dict(mesh)
        ctx.load(0, **parts)
        ctx.compute_fields()
        phi = ctx.fields(G.PIC_FIELD_PHI)
        ctx.compute_fields()  # from the solution: the warm start and the singular projection again
        phi2 = ctx.fields(G.PIC_FIELD_PHI)
    sim = O.Sim(cfg, O.Mesh(nx, ny, h, 0, bc[0], bc[1]))
    sim.load(0, **parts)
    sim.fields()
    # ||e|| <= ||r|| / lambda_min <= tol ||b|| / lambda_min, ||b|| <= 8 ||phi||; lambda_min of the
    # smoother direction (periodic: a whole wave, walls: at least half a wave across the mesh)
    lam = 2.0 - 2.0 * np.cos(np.pi / max(nx, ny, 2))
    bar = 1e-12 * 8.0 / lam + 1e-13 / lam
    for p in (phi, phi2):
        assert np.linalg.norm(p - sim.phi) <= bar * np.linalg.norm(sim.phi)


def test_clusters_of_every_size_give_the_same_bits():
    """41 instances (clusters of 2 CTAs; alone: 8 and 1) and 3 (8): each equals itself alone."""
    def sim(i, nx):
        cfg, mesh, parts = W.ccp(nx=nx, ny=16, ppc=2, seed=50 + i)
        cfg["instance"] = i
        return cfg, mesh, parts

    sims = [sim(i, 512 if i == 0 else 16 + 16 * (i % 5)) for i in range(41)]
    alone = []
    for cfg, mesh, parts in sims[:3]:
        with G.Context(cfg) as ctx:
            ctx.set_mesh_dict(mesh)
            for s in parts:
                ctx.load(s, **parts[s])
            ctx.step(3)
            alone.append(ctx.fields(G.PIC_FIELD_PHI))
    for count in (3, 41):
        with G.Context([s[0] for s in sims[:count]]) as ctx:
            for i, (cfg, mesh, parts) in enumerate(sims[:count]):
                ctx.set_mesh_dict(mesh, inst=i)
                for s in parts:
                    ctx.load(s, **parts[s], inst=i)
            ctx.step(3)
            for i in range(3):
                assert np.array_equal(ctx.fields(G.PIC_FIELD_PHI, inst=i), alone[i])


# the implicit scheme's operator: a coarsest inverse formed by the launch (up to 128 cells), CG
# beyond, a mesh two cells wide in a periodic direction, one level only, ragged strips
@pytest.mark.parametrize("bc", [(D, P), (P, P), (D, N)])
@pytest.mark.parametrize("nx,ny", [(4, 4), (11, 11), (33, 9), (2, 32), (40, 20), (60, 44), (208, 24), (34, 66), (64, 64)])
def test_implicit_solve_matches_the_oracle(nx, ny, bc):
    n = nx * ny * 3
    rng = np.random.default_rng(nx + 1000 * ny)
    h, dt = 2.0 ** -6, 3.0
    cfg = W.base_config(precision=W.FP64, n_species=1, q=[-1.0], m=[1.0], dt=dt, bc_x=bc[0], bc_y=bc[1], implicit=1,
                        rho_background=1.0, phi_left_dc=0.0 if bc[0] != D else 0.02, mg_rel_tol=1e-11, mg_max_cycles=200)
    mesh = dict(nx0=nx, ny0=ny, h0=h, lmax=0)
    z = np.zeros(n)
    parts = dict(x=rng.random(n) * nx * h, y=rng.random(n) * ny * h, vx=z, vy=z, vz=z, w=np.full(n, h * h / 3))
    with G.Context(cfg) as ctx:
        ctx.set_mesh_dict(mesh)
        ctx.load(0, **parts)
        ctx.compute_fields()
        phi = ctx.fields(G.PIC_FIELD_PHI)
    sim = O.Sim(cfg, O.Mesh(nx, ny, h, 0, bc[0], bc[1]))
    sim.load(0, **parts)
    sim.fields()
    # as above, the eigenvalues scaled by kappa = 1 + dt^2 n: at least 1, at most its largest
    kmax = 1.0 + dt * dt * sim.counts(0).max() / 3.0
    lam = 2.0 - 2.0 * np.cos(np.pi / max(nx, ny, 2))
    bar = (1e-11 * 8.0 + 1e-13) * kmax / lam
    assert np.linalg.norm(phi - sim.phi) <= bar * np.linalg.norm(sim.phi)
