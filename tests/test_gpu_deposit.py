"""The charge per leaf formed from the records (after a load), where a warp sums several leaves:
every number of leaves per warp, with a last warp that has fewer."""
import numpy as np
import pytest

import paper_1604_07713_gb300 as G
from paper_1604_07713_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [W.FP32, W.FP64])
@pytest.mark.parametrize("nx,ny", [(3, 2), (128, 120), (176, 128), (480, 480), (512, 512)])  # 1, 2, 3, 31, 32 leaves a warp
def test_charge_from_records(nx, ny, precision):
    G.build()
    h = 2.0 ** -6
    rng = np.random.default_rng(nx)
    cfg = W.base_config(precision=precision, n_species=2, q=[-1.0, 2.0], m=[1.0, 9.0], bc_x=W.BC_DIRICHLET,
                        bc_y=W.BC_NEUMANN, max_level=0)
    want, mag = np.zeros(nx * ny), np.zeros(nx * ny)
    with G.Context(cfg) as ctx:
        ctx.set_mesh_dict(dict(nx0=nx, ny0=ny, h0=h, lmax=0))
        for s, n in enumerate((4 * nx * ny + 1, 3 * nx * ny)):
            # half of the records in the last 40 leaves, so that some lists take several rounds
            leaf = np.where(rng.random(n) < 0.5, rng.integers(0, nx * ny, n), nx * ny - 1 - rng.integers(0, min(40, nx * ny), n))
            w = (0.5 + rng.random(n)).astype(np.float32).astype(np.float64)
            z = np.zeros(n)
            ctx.load(s, (leaf % nx + 0.5) * h, (leaf // nx + 0.5) * h, z, z, z, w)
            c = np.bincount(leaf, w, nx * ny) * cfg["q"][s]
            want += c
            mag += np.abs(c)
        ctx.compute_fields(allow_notconv=True)
        got = ctx.fields(G.PIC_FIELD_RHO) * h * h
    # one rounding of a compensated sum in the state's precision, FP64 beyond (bincount: up to
    # 6e5 FP64 additions in a row)
    eps = 2.0 ** -23 if precision == W.FP32 else 1e-12
    assert np.all(np.abs(got - want) <= (eps + 1e-10) * mag)
