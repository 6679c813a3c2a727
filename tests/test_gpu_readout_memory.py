"""Read-outs that need no device memory of their own: counts, charge density, potential and corner
field come out the same when the device has no room for the arrays they are otherwise formed in."""
import numpy as np
import pytest

import paper_1604_07713_gb300 as G
from paper_1604_07713_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lmax", [0, 2])
@pytest.mark.parametrize("precision", [W.FP32, W.FP64])
def test_fields_without_room(precision, lmax):
    G.build()
    cfg, mesh, parts = W.ccp(nx=32, ny=8, ppc=20, seed=4, precision=precision)
    cfg.update(rho_background=0.3, max_level=lmax)
    mesh["lmax"] = lmax
    if lmax:
        mesh["root"], mesh["level"], mesh["morton"] = W.random_tree(32, 8, lmax, 0.3, 7, False, True)
    with G.Context(cfg) as ctx:
        ctx.set_mesh_dict(mesh)
        for s in parts:
            ctx.load(s, **parts[s])
        ctx.step(2, allow_notconv=True)
        for f in (G.PIC_FIELD_PHI, G.PIC_FIELD_RHO, G.PIC_FIELD_COUNT_E, G.PIC_FIELD_COUNT_I, G.PIC_FIELD_NODE_E):
            G.pic_inject_fault(ctx.ctx, G.PIC_FAULT_NONE)
            want = ctx.fields(f)
            G.pic_inject_fault(ctx.ctx, G.PIC_FAULT_ALLOC, 0)
            assert np.array_equal(ctx.fields(f), want), f
        G.pic_inject_fault(ctx.ctx, G.PIC_FAULT_ALLOC, 0)  # |E| always needed its own array
        with pytest.raises(G.PicError) as e:
            ctx.fields(G.PIC_FIELD_EMAG)
        assert e.value.status == G.PIC_ENOMEM
