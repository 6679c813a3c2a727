"""The implicit scheme on meshes of many blocks whose coarsest level is solved by an inverse formed once
per solve (1 to 128 cells) or by the conjugate gradients (beyond): the potential against the FP64
oracle, again after a step has changed every cell's susceptibility."""
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


# coarsest levels of 15, 77, 121, 117, 154 cells, and of 35 below a refined mesh
@pytest.mark.parametrize("bc", [(D, P), (P, P), (D, N)])
@pytest.mark.parametrize("nx,ny,lmax", [(160, 96, 0), (176, 112, 0), (176, 176, 0), (208, 144, 0), (352, 112, 0), (56, 80, 2)])
def test_potential_matches_the_oracle(nx, ny, lmax, bc):
    h, rng = 2.0 ** -6, np.random.default_rng(nx + ny)
    mesh = dict(nx0=nx, ny0=ny, h0=h, lmax=lmax)
    if lmax:
        mesh["root"], mesh["level"], mesh["morton"] = W.random_tree(nx, ny, lmax, 0.3, 5, bc[0] == P, bc[1] == P)
    n, tol = 3 * nx * ny, 1e-10
    cfg = W.base_config(precision=W.FP64, n_species=1, q=[-1.0], m=[1.0], dt=3.0, bc_x=bc[0], bc_y=bc[1], implicit=1,
                        max_level=lmax, rho_background=1.0, phi_left_dc=0.0 if bc[0] != D else 0.02, mg_rel_tol=tol,
                        mg_max_cycles=100)
    v = rng.standard_normal((3, n)) * 0.3 * h  # dt v: a cell a step
    parts = dict(x=rng.random(n) * nx * h, y=rng.random(n) * ny * h, vx=v[0], vy=v[1], vz=v[2], w=np.full(n, h * h / 3))
    sim = O.Sim(cfg, O.Mesh(nx, ny, h, lmax, bc[0], bc[1], mesh.get("root"), mesh.get("level"), mesh.get("morton")))
    sim.load(0, **parts)
    with G.Context(cfg) as ctx:
        ctx.set_mesh_dict(mesh)
        ctx.load(0, **parts)
        for again in (False, True):
            if again:
                ctx.step(1)
                g = ctx.particles(0)  # the oracle's next solve is that of the same particles
                sim.load(0, **{k: g[k] for k in ("x", "y", "vx", "vy", "vz", "w")})
            ctx.compute_fields()
            phi = ctx.fields(G.PIC_FIELD_PHI)
            sim.fields()
            # ||e|| <= tol ||b|| / lambda_min, ||b|| <= 8 kappa_max ||phi||, lambda_min of half a wave
            # across the mesh (4^lmax smaller where leaf sides differ), kappa >= 1
            lam = (2.0 - 2.0 * np.cos(np.pi / max(nx, ny))) / 4.0 ** lmax
            bar = (tol * 8.0 + 1e-13) * sim.kappa().max() / lam
            assert np.linalg.norm(phi - sim.phi) <= bar * np.linalg.norm(sim.phi)
