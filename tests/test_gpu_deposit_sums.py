"""The charge formed from the records: the lanes' compensated sums in the state's precision and their
error-free combination, with both words of the result, as the same arithmetic in NumPy gives them."""
import numpy as np
import pytest

import paper_1604_07713_gb300 as G
from paper_1604_07713_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [W.FP32, W.FP64])
@pytest.mark.parametrize("nx,ny", [(3, 2), (128, 120), (176, 128), (512, 512)])  # 1, 2, 3, 32 leaves a warp
def test_charge_of_compensated_sums(nx, ny, precision):
    G.build()
    h, nl = 2.0 ** -6, nx * ny
    rng = np.random.default_rng(nx)
    cfg = W.base_config(precision=precision, n_species=2, q=[-1.0, 2.0], m=[1.0, 9.0], bc_x=W.BC_DIRICHLET,
                        bc_y=W.BC_NEUMANN, max_level=0)
    leaves = np.unique(np.concatenate([rng.integers(0, nl, 64), nl - 1 - np.arange(min(6, nl))]))
    R = np.float32 if precision == W.FP32 else np.float64
    want, mass = np.zeros(leaves.size), np.zeros(leaves.size)
    with G.Context(cfg) as ctx:
        ctx.set_mesh(nx0=nx, ny0=ny, h0=h)
        for s, n in enumerate((nl + 20_000, nl)):
            leaf = np.concatenate([np.arange(nl), nl - 1 - rng.integers(0, min(5, nl), n - nl)])
            w = (0.5 + rng.random(n)).astype(np.float32).astype(np.float64)
            z = np.zeros(n)
            ctx.load(s, (leaf % nx + 0.5) * h, (leaf // nx + 0.5) * h, z, z, z, w)
            o = np.argsort(leaf, kind="stable")
            lists = np.split(w[o], np.cumsum(np.bincount(leaf, minlength=nl))[:-1])
            want += cfg["q"][s] * np.array([_sum(lists[i], R) for i in leaves])
            mass += abs(cfg["q"][s]) * np.array([lists[i].sum() for i in leaves])
        ctx.compute_fields(allow_notconv=True)
        got = ctx.fields(G.PIC_FIELD_RHO)[leaves] * h * h
    # the two words of each species added, scaled and summed in FP64
    assert np.all(np.abs(got - want) <= 4.0 * 2.0 ** -53 * mass)


def _sum(w, R):
    """Lane i adds records i, i + 32, ... in rounds of four (zeros past the end), then the lanes' pairs."""
    hi, c = np.zeros(32, R), np.zeros(32, R)
    for k in range(0, w.size, 32):
        first = 128 * (k // 128)  # a lane takes part in a round if it has the round's first record
        live = first + np.arange(32) < w.size
        x = np.zeros(32, R)
        x[: w[k : k + 32].size] = w[k : k + 32]
        y = x - c
        t = hi + y
        hi, c = np.where(live, t, hi), np.where(live, (t - hi) - y, c)
    # (rounds of zeros past the last record)
    for k in range(32 * -(-w.size // 32), 128 * -(-w.size // 128), 32):
        live = 128 * (k // 128) + np.arange(32) < w.size
        y = -c
        t = hi + y
        hi, c = np.where(live, t, hi), np.where(live, (t - hi) - y, c)
    lo = -c
    for o in (16, 8, 4, 2, 1):
        oh, ol = hi[np.arange(32) ^ o], lo[np.arange(32) ^ o]
        t = hi + oh
        bp = t - hi
        hi, lo = t, lo + ol + ((hi - (t - bp)) + (oh - bp))
    return float(hi[0]) + float(lo[0])
