"""The cloud-in-cell deposit's sums are FP64 for either precision of the state: the charge of every
cell against an exactly rounded sum of exact products, for weights whose sum leaves FP32's range on
either side, for lists of one, a few and many records, equal and random weights."""
import math

import numpy as np
import pytest

import paper_1604_07713_gb300 as G
from paper_1604_07713_gb300 import workloads as W

pytestmark = pytest.mark.gpu

P, D, N = W.BC_PERIODIC, W.BC_DIRICHLET, W.BC_NEUMANN


@pytest.mark.parametrize("precision", [W.FP32, W.FP64])
@pytest.mark.parametrize("shape", [G.PIC_SHAPE_CIC_EM, G.PIC_SHAPE_CIC_EC])
@pytest.mark.parametrize("scale,total,equal", [(2.0 ** 125, 3000, True), (2.0 ** -130, 3000, False), (2.0 ** -100, 3000, True),
                                               (1.0, 20, False), (1.0, 3000, False), (1.0, 300_000, True)])
def test_charge_against_exact_sums(scale, total, equal, shape, precision):
    G.build()
    nx, ny, h = 7, 5, 2.0 ** -4
    rng = np.random.default_rng(total)
    cfg = W.base_config(precision=precision, shape=shape, n_species=2, q=[-1.0, 2.0], m=[1.0, 9.0], bc_x=D, bc_y=P,
                        eps0=scale * total)
    Q = [[] for _ in range(nx * ny)]
    longest = 0
    with G.Context(cfg) as ctx:
        ctx.set_mesh(nx0=nx, ny0=ny, h0=h)
        for s in (0, 1):
            n = total if s == 0 else total // 3
            # half of the records in one cell
            i, j = np.where(rng.random((2, n)) < 0.7, 2, [rng.integers(0, nx, n), rng.integers(0, ny, n)])
            ku, kv = rng.integers(0, 1024, (2, n))  # offsets in 1/1024: every product is exact
            m = np.full(n, 11184811) if equal else rng.integers(1 << 20, 1 << 24, n)
            w = m * 2.0 ** -24 * scale
            if precision == W.FP32:  # (FP32 weights below its normal range have fewer bits)
                w = w.astype(np.float32).astype(np.float64)
            z = np.zeros(n)
            ctx.load(s, (i + ku / 1024.0) * h, (j + kv / 1024.0) * h, z, z, z, w)
            longest = max(longest, int(np.bincount(i + nx * j).max()))
            qx, qy = ku >= 512, kv >= 512
            fx, fy = ku / 1024.0 + 0.5 - qx, kv / 1024.0 + 0.5 - qy
            for a in (0, 1):
                for b in (0, 1):
                    c = np.clip(i - 1 + qx + a, 0, nx - 1) + nx * ((j - 1 + qy + b) % ny)
                    v = cfg["q"][s] * w * (fx if a else 1.0 - fx) * (fy if b else 1.0 - fy)
                    o = np.argsort(c, kind="stable")
                    for k, part in zip(*_groups(c[o], v[o])):
                        Q[k].append(part)
        ctx.compute_fields(allow_notconv=True)
        got = ctx.fields(G.PIC_FIELD_RHO) * h * h
    want = np.array([math.fsum(x for p in q for x in p) for q in Q])
    mass = sum(float(np.abs(p).sum()) for q in Q for p in q)
    # a lane adds every 32nd record of a list, then ~30 additions and the nine cells' combinations,
    # each rounded once, of terms that are parts of the whole charge
    assert np.all(np.isfinite(got))
    assert np.all(np.abs(got - want) <= (longest / 32 + 64) * 2.0 ** -53 * mass)


def _groups(c, v):
    k, first = np.unique(c, return_index=True)
    return k, np.split(v, first[1:])
