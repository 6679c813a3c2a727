"""The multi-block Poisson cycle's tile kernels for uniform levels, at meshes whose tiles are
ragged, wrap onto themselves or end at walls, against the FP64 oracle; and the operator codes of
an adaptive mesh with every kind of face."""
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


def _phi(mesh, bc, seed):
    nx, ny, h = mesh["nx0"], mesh["ny0"], mesh["h0"]
    n = nx * ny
    rng = np.random.default_rng(seed)
    # neutral on average, so that the potential stays within the residual's FP64 floor
    cfg = W.base_config(precision=W.FP64, n_species=1, q=[-1.0], m=[1.0], bc_x=bc[0], bc_y=bc[1], rho_background=1.0,
                        max_level=mesh["lmax"], phi_left_dc=0.0 if bc[0] != D else 0.02, mg_rel_tol=1e-11, mg_max_cycles=60)
    z = np.zeros(n)
    parts = dict(x=rng.random(n) * nx * h, y=rng.random(n) * ny * h, vx=z, vy=z, vz=z, w=np.full(n, h * h))
    with G.Context(cfg) as ctx:
        ctx.set_mesh_dict(mesh)
        ctx.load(0, **parts)
        ctx.compute_fields()
        a = ctx.fields(G.PIC_FIELD_PHI)
        ctx.compute_fields()
        b = ctx.fields(G.PIC_FIELD_PHI)
    sim = O.Sim(cfg, O.Mesh(nx, ny, h, mesh["lmax"], bc[0], bc[1], mesh.get("root"), mesh.get("level"), mesh.get("morton")))
    sim.load(0, **parts)
    sim.fields()
    # ||e|| <= tol ||b|| / lambda_min, ||b|| <= 8 ||phi||; lambda_min of half a wave across the mesh
    # (leaf sides differ by 2^lmax, so the smallest eigenvalue can be 4^lmax smaller)
    lam = (2.0 - 2.0 * np.cos(np.pi / max(nx, ny))) / 4.0 ** mesh["lmax"]
    for p in (a, b):
        assert np.linalg.norm(p - sim.phi) <= (1e-11 * 8.0 / lam + 1e-13 / lam) * np.linalg.norm(sim.phi)


@pytest.mark.parametrize("bc", [(D, P), (P, P), (P, D), (D, N)])
@pytest.mark.parametrize("nx,ny", [(96, 96), (1024, 16), (16, 1024), (100, 84), (328, 40), (176, 112), (32, 512)])
def test_uniform_levels(nx, ny, bc):
    _phi(dict(nx0=nx, ny0=ny, h0=2.0 ** -6, lmax=0), bc, nx + ny)


@pytest.mark.parametrize("bc", [(D, N), (P, P)])
def test_adaptive_levels(bc):
    px, py = bc[0] == P, bc[1] == P
    r, l, m = W.random_tree(96, 96, 2, 0.3, 5, px, py)
    _phi(dict(nx0=96, ny0=96, h0=2.0 ** -6, lmax=2, root=r, level=l, morton=m), bc, 9)
