"""The implicit scheme between Neumann walls only (and one periodic direction), where the coarsest
operator is singular without being periodic in both directions: the potential up to its constant
against a direct solve of the oracle's operator with the constant fixed."""
import numpy as np
import pytest
from scipy.sparse.linalg import spsolve

import oracle as O
import paper_1604_07713_gb300 as G
from paper_1604_07713_gb300 import workloads as W

pytestmark = pytest.mark.gpu

P, N = W.BC_PERIODIC, W.BC_NEUMANN


@pytest.fixture(scope="module", autouse=True)
def _built():
    G.build()
    O.build()


@pytest.mark.parametrize("bc", [(N, N), (N, P), (P, N)])
@pytest.mark.parametrize("nx,ny,lmax", [(4, 4, 0), (11, 11, 0), (16, 8, 0), (40, 20, 0), (160, 96, 0), (5, 5, 1), (12, 10, 2)])
def test_potential_up_to_its_constant(nx, ny, lmax, bc):
    h, rng = 2.0 ** -6, np.random.default_rng(nx + ny + lmax)
    mesh = dict(nx0=nx, ny0=ny, h0=h, lmax=lmax)
    if lmax:
        r, lv, m = W.random_tree(nx, ny, lmax, 0.3, 5, bc[0] == P, bc[1] == P)
        mesh.update(root=r, level=lv, morton=m)
    # exactly neutral (powers of two), so that the singular problem has a solution
    n = 4 * nx * ny
    cfg = W.base_config(precision=W.FP64, n_species=1, q=[-1.0], m=[1.0], dt=2.0, bc_x=bc[0], bc_y=bc[1], implicit=1,
                        max_level=lmax, rho_background=1.0, mg_rel_tol=1e-9, mg_max_cycles=60)
    z = np.zeros(n)
    parts = dict(x=rng.random(n) * nx * h, y=rng.random(n) * ny * h, vx=z, vy=z, vz=z, w=np.full(n, h * h / 4))
    with G.Context(cfg) as ctx:
        ctx.set_mesh_dict(mesh)
        ctx.load(0, **parts)
        ctx.compute_fields()
        phi = ctx.fields(G.PIC_FIELD_PHI)
    M = O.Mesh(nx, ny, h, lmax, bc[0], bc[1], mesh.get("root"), mesh.get("level"), mesh.get("morton"))
    sim = O.Sim(cfg, M)
    sim.load(0, **parts)
    A = M.operator_kappa(sim.kappa())[0].tocsc()
    b = sim.charge() + M.area()
    assert abs(b.sum()) <= 1e-12 * np.abs(b).sum()
    # the sparse solve with the last cell held at zero (its row is implied by the others)
    want = np.zeros(b.size)
    want[:-1] = spsolve(A[:-1, :-1], b[:-1])
    d = (phi - phi.mean()) - (want - want.mean())
    # ||e|| <= tol ||b|| / lambda_2 (the smallest nonzero eigenvalue, >= half a wave across the mesh,
    # 4^lmax smaller where leaf sides differ); the direct solve within the FP64 floor of the same
    lam = (2.0 - 2.0 * np.cos(np.pi / max(nx, ny))) / 4.0 ** lmax
    assert np.linalg.norm(d) <= 2.0 * (1e-9 + 1e-12) * np.linalg.norm(b) / lam

