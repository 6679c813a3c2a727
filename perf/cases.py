"""What a user of this framework has it do, as measurable cases: whole steps of the particle
cycle through the public entry points, the mesh adaptation that goes with them, the batched
ensemble, and the load of a population from host memory.

The physics and the sizes are those of ``paper_1604_07713_gb300/workloads.py``, the tests and
``bench.py``: the cold-plasma oscillation, the capacitively coupled discharge (CCP) and its
uneven ensemble, and the 2D streamer on an adaptive quadtree.  Populations are drawn on the
GPU from the seed (the workloads' distributions) and handed to the library as host arrays,
which is what its load takes.

A pass advances the simulation by ``steps`` steps (one ``pic_step`` call), adapts where the
case does, and reads back what a user reads at an output interval.  The fields of an FP32 run
are kept in FP32.  Passes of up to 4 steps read the potential, the corner field and the
particles of both species per leaf; longer ones read the potential (a rounding that lets one
particle cross a face a step later changes a count, and hardly the potential)."""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1604_07713_gb300 as G

QE, ME, AMU, EPS0 = 1.602176634e-19, 9.1093837015e-31, 1.66053906660e-27, 8.8541878128e-12
PERIODIC, DIRICHLET, NEUMANN = 0, 1, 2
NGP, CIC_EM, CIC_EC = 0, 1, 2
H_CCP = 0.067 / 512  # the discharge's cell side [m]
BINS, EV_MAX = 200, 60.0  # the electron energy distribution's bins and range [eV]


def listed():
    return [
        # A cold-plasma oscillation, 64 x 64 cells, 16 electrons per cell, FP64, one step and its
        # fields: the smallest call, and the periodic (singular) solve.
        dict(name="plasma_64_f64", kind="plasma", nx=64, ny=64, ppc=16.0, fp64=True, steps=1),
        # The same on a mesh whose fine multigrid levels span many blocks, several steps a call.
        dict(name="plasma_256_f32", kind="plasma", nx=256, ny=256, ppc=32.0, fp64=False, steps=4),
        # A small discharge with collisions, its fields and its whole particle state read every few
        # steps (RF-phase resolved output): launches and latency count.
        dict(name="ccp_128x16_f32", kind="ccp", nx=128, ny=16, ppc=20.3, fp64=False, steps=4, particles_out=True),
        # The benchmark's discharge, 512 x 16 cells, 2 x 819,200 particles: many steps between
        # outputs, the ordinary production run.
        dict(name="ccp_512x16_f32", kind="ccp", nx=512, ny=16, ppc=100.0, fp64=False, steps=20),
        # The same in FP64, the mode for verification runs.
        dict(name="ccp_512x16_f64", kind="ccp", nx=512, ny=16, ppc=100.0, fp64=True, steps=4),
        # The same with the direct implicit scheme (two push passes, the operator assembled with
        # the susceptibility on every step).
        dict(name="ccp_512x16_implicit", kind="ccp", nx=512, ny=16, ppc=100.0, fp64=False, steps=4, implicit=1),
        # The same with the energy-conserving cloud-in-cell shape.
        dict(name="ccp_512x16_cic", kind="ccp", nx=512, ny=16, ppc=100.0, fp64=False, steps=4, shape=CIC_EC),
        # A discharge of ragged size with its time averages and energy distribution taken.
        dict(name="ccp_208x24_diag", kind="ccp", nx=208, ny=24, ppc=77.7, fp64=False, steps=4, diag=True),
        # The early streamer: a seed of electrons and ions, adapted every 10 steps.
        dict(name="streamer_2e5_f32", kind="streamer", nx=128, lmax=4, particles=200_000, fp64=False, steps=10),
        # The grown streamer, the benchmark's headline size: state far larger than L2.
        dict(name="streamer_5e7_f32", kind="streamer", nx=128, lmax=4, particles=50_000_000, fp64=False, steps=10),
        # A parameter study: uneven discharges advanced together in one context.
        dict(name="ensemble_32_f32", kind="ensemble", instances=32, nx=512, ppc=200.0, fp64=False, steps=5),
        # End to end from host memory: both species of a streamer loaded onto its adapted mesh,
        # one step, the fields read back (a coupled code that hands over its particles).
        dict(name="reload_2e6_f32", kind="reload", nx=128, lmax=4, particles=2_000_000, fp64=False, steps=1),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["plasma", "ccp", "ccp", "ccp", "streamer", "streamer", "ensemble", "reload"])
    fp64 = rng.random() < 0.25
    if kind == "plasma":
        n = rng.choice([2, 3, 4, 5, 7]) << rng.randint(3, 6)  # 16 .. 448 per side
        m = max(16, n // rng.choice([1, 2]))
        return dict(kind=kind, nx=n, ny=m, ppc=round(_log(rng, 3.0, 40.0), 2), fp64=fp64, steps=rng.choice([1, 4]))
    if kind == "ccp":
        c = dict(kind=kind, nx=16 * rng.randint(2, 32), ny=8 * rng.randint(1, 4), ppc=round(_log(rng, 8.0, 300.0), 2),
                 fp64=fp64, steps=rng.choice([1, 4, 20]))
        if rng.random() < 0.15:  # a mesh that does not coarsen
            c.update(nx=2 * rng.randint(8, 24) + 1, ny=2 * rng.randint(3, 6) + 1)
        variant = rng.random()
        if variant < 0.2:
            c["implicit"] = 1
        elif variant < 0.4:
            c["shape"] = rng.choice([CIC_EM, CIC_EC])
        elif variant < 0.5:
            c["diag"] = True
        if c["fp64"] or len(c) > 6:
            c["steps"] = min(c["steps"], 4)
        if c["steps"] <= 4 and c["nx"] * c["ny"] * c["ppc"] < 60_000:
            c["particles_out"] = True
        return c
    if kind == "streamer":
        return dict(kind=kind, nx=rng.choice([48, 64, 96, 128]), lmax=rng.randint(2, 4),
                    particles=int(_log(rng, 5e4, 4e6 if fp64 else 3e7)) | 1, fp64=fp64, steps=10)
    if kind == "ensemble":
        return dict(kind=kind, instances=rng.randint(2, 32), nx=16 * rng.randint(4, 32), ppc=round(_log(rng, 20.0, 200.0), 1),
                    fp64=False, steps=rng.choice([1, 5]))
    return dict(kind=kind, nx=rng.choice([64, 96, 128]), lmax=rng.randint(2, 4), particles=int(_log(rng, 1e5, 6e6)) | 1,
                fp64=fp64, steps=1)


# ---------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


class _Rng:
    def __init__(self, seed):
        self.dev = _device()
        self.g = torch.Generator(device=self.dev)
        self.g.manual_seed(int(seed) * 2654435761 % (1 << 62) + 1)

    def rand(self, *n):
        return torch.rand(*n, generator=self.g, dtype=torch.float64, device=self.dev)

    def randn(self, *n):
        return torch.randn(*n, generator=self.g, dtype=torch.float64, device=self.dev)


def _config(case, **kw):
    c = dict(precision=1 if case["fp64"] else 0, n_species=2, seed=160407713, dt=1e-3, eps0=EPS0, q=[-QE, QE],
             m=[ME, 4.0 * AMU], qe=QE, mcc=1, bc_x=DIRICHLET, bc_y=PERIODIC, max_level=0, gas_density=0.0,
             gas_temperature_ev=0.026, neutral_mass=4.0 * AMU, sigma_el=6e-20, sigma_iz0=1e-20, eps_th_ev=24.6,
             phi_left_dc=0.0, phi_left_amp=0.0, phi_left_freq=0.0, phi_right=0.0, rho_background=0.0, ppc_target=32,
             ppc_min=8, ppc_max=128, adapt_every=0, e_ref=1.0, refine_field=1.5, coarsen_field=1.2, refine_count=128,
             coarsen_count=32, mg_rel_tol=1e-11 if case["fp64"] else 1e-8, mg_max_cycles=40, particle_capacity=0,
             instance=0, shape=case.get("shape", NGP), implicit=case.get("implicit", 0))
    c.update(kw)
    return c


def _plasma(case, rng):
    nx, ny = case["nx"], case["ny"]
    h, n = 1.0 / nx, int(nx * ny * case["ppc"])
    x0, y = rng.rand(n), rng.rand(n) * (ny * h)
    x = torch.remainder(x0 - 0.01 / (2 * math.pi) * torch.sin(2 * math.pi * x0), 1.0)
    x = torch.where(x >= 1.0, torch.zeros_like(x), x)
    z = torch.zeros_like(x)
    # omega_p = 1 in units eps0 = m_e = n0 = 1
    cfg = _config(case, n_species=1, dt=0.05, eps0=1.0, q=[-1.0, 1.0], m=[1.0, 1836.0], qe=1.0, mcc=0, bc_x=PERIODIC,
                  rho_background=1.0, neutral_mass=1.0, mg_rel_tol=1e-12 if case["fp64"] else 1e-10)
    return cfg, dict(nx0=nx, ny0=ny, h0=h), [[x, y, z, z, z, torch.full_like(x, ny * h / n)]]


def _ccp(case, rng, volt=200.0, ng=9.6e20, instance=0, nx=None, ppc=None):
    nx, ny, ppc = nx or case["nx"], case.get("ny", 16), ppc or case["ppc"]
    h, n = H_CCP, int(nx * ny * ppc)
    freq = 13.56e6
    parts = []
    for m, t in ((ME, 2.5), (4.0 * AMU, 0.026)):
        x, y = rng.rand(n) * (nx * h), rng.rand(n) * (ny * h)
        v = rng.randn(3, n) * math.sqrt(t * QE / m)
        parts.append([x, y, v[0], v[1], v[2], torch.full_like(x, 1e15 * h * h / ppc)])
    cfg = _config(case, dt=1.0 / (400.0 * freq), gas_density=ng, phi_left_amp=volt, phi_left_freq=freq, instance=instance)
    return cfg, dict(nx0=nx, ny0=ny, h0=h), parts


def _streamer(case, rng, box=0.01, e0=3e6):
    """A seed (below a million particles: a neutral Gaussian at the centre) or a grown channel."""
    n, nx, seedling = case["particles"] // 2, case["nx"], case["particles"] < 1_000_000
    parts = []
    for m, t in ((ME, 5.0), (4.0 * AMU, 0.026)):
        if seedling:
            x = 0.5 * box + rng.randn(n) * (8e-4)
            y = 0.5 * box + rng.randn(n) * (2e-4)
            w = 1e13 / n
        else:
            x = 0.25 * box + 0.5 * box * rng.rand(n)
            tail = rng.rand(n) < 0.1
            x = torch.where(tail, 0.5 * box + 0.3 * box * rng.randn(n), x)
            y = 0.5 * box + 0.05 * box * rng.randn(n)
            w = 1e19 * 0.5 * box * 2.5 * 0.05 * box / n
        x, y = x.clamp(1e-4 * box, box * (1 - 1e-4)), y.clamp(1e-4 * box, box * (1 - 1e-4))
        v = rng.randn(3, n) * math.sqrt(t * QE / m)
        parts.append([x, y, v[0], v[1], v[2], torch.full_like(x, w)])
    cfg = _config(case, dt=1e-13, bc_y=NEUMANN, max_level=case["lmax"], gas_density=3.2e24, phi_right=e0 * box, e_ref=e0,
                  adapt_every=10)
    return cfg, dict(nx0=nx, ny0=nx, h0=box / nx), parts


def _ensemble(case, seed):
    """Uneven discharges: x-cells a multiple of 16 up to nx, 20 .. ppc per cell and species,
    amplitude 100-400 V, gas density log-uniform; the sizes fixed by the case, the rest by the seed."""
    shape = np.random.default_rng([case["instances"], case["nx"]])
    out = []
    for i in range(case["instances"]):
        nx = 16 * int(shape.integers(4, case["nx"] // 16 + 1)) if i else case["nx"]
        ppc = float(shape.uniform(20.0, max(21.0, case["ppc"])))
        volt, ng = float(shape.uniform(100.0, 400.0)), float(np.exp(shape.uniform(np.log(3e20), np.log(3e21))))
        out.append(_ccp(case, _Rng(seed * 1009 + i), volt, ng, i, nx, ppc))
    return out


def _inputs(case, seed):
    if case["kind"] == "ensemble":
        return _ensemble(case, seed)
    make = {"plasma": _plasma, "ccp": _ccp, "streamer": _streamer, "reload": _streamer}[case["kind"]]
    return [make(case, _Rng(seed))]


def _host(arrays, pinned=False):
    out = []
    for a in arrays:
        t = torch.empty(a.shape, dtype=torch.float64, pin_memory=pinned)
        t.copy_(a)
        out.append(t.numpy())
    return out


def prepare(case, seed):
    sims = _inputs(case, seed)
    ctx = G.Context([s[0] for s in sims])
    for i, (_, mesh, parts) in enumerate(sims):
        ctx.set_mesh_dict(mesh, inst=i)
        for s, p in enumerate(parts):
            ctx.load(s, *_host(p), inst=i)
    state = dict(ctx=ctx, case=case, instances=len(sims), species=len(sims[0][2]))
    if case["kind"] in ("streamer", "reload"):  # refine the root grid onto the particles, then manage them
        for _ in range(case["lmax"] + 1):
            ctx.compute_fields(allow_notconv=True)
            ctx.adapt(G.PIC_ADAPT_MESH)
        ctx.compute_fields(allow_notconv=True)
        ctx.adapt()
    if case["kind"] == "reload":
        state["parts"] = [_host(p, pinned=torch.cuda.is_available()) for p in sims[0][2]]
    if case.get("diag"):
        ctx.diag_enable(BINS, EV_MAX)
    return state


# ---------------------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------------------
def _leaves_at_most(case):
    return case["nx"] ** 2 + case["particles"] // 64 + 60_000


def _kept(case, a, kind):
    """A field in the run's precision; an adaptive mesh's in an array of the run's fixed leaf capacity."""
    if case["kind"] not in ("streamer", "reload"):
        return a.astype(kind)
    return _padded(a, _leaves_at_most(case), kind)


def _loaded(case):
    return int(case["nx"] * case["ny"] * case["ppc"])


def _padded(a, n, kind):
    out = np.zeros((max(n, a.shape[0]),) + a.shape[1:], kind)
    out[: a.shape[0]] = a
    return out


def run(state):
    ctx, case = state["ctx"], state["case"]
    kind = np.float64 if case["fp64"] else np.float32
    if case["kind"] == "reload":
        for s, p in enumerate(state["parts"]):
            ctx.load(s, *p)
    ctx.step(case["steps"])
    if case["kind"] == "ensemble":
        return {"phi": [ctx.fields(G.PIC_FIELD_PHI, i).astype(kind) for i in range(state["instances"])]}
    out = {"phi": _kept(case, ctx.fields(G.PIC_FIELD_PHI), kind)}
    if case["steps"] <= 4:
        out["e"] = _kept(case, ctx.fields(G.PIC_FIELD_NODE_E), kind)
        out["n"] = [_kept(case, ctx.fields(f), np.float64)
                    for f in (G.PIC_FIELD_COUNT_E, G.PIC_FIELD_COUNT_I)[: state["species"]]]
    if case.get("particles_out"):
        for s in range(state["species"]):
            p = ctx.particles(s)
            types = dict.fromkeys(("x", "y", "vx", "vy", "vz", "w"), kind) | dict(id=np.int64, leaf=np.int64)
            out["particles%d" % s] = [_padded(p[k], _loaded(case), t) for k, t in types.items()]
    if case.get("diag"):
        out["avg_phi"] = ctx.fields(G.PIC_FIELD_AVG_PHI).astype(kind)
        out["avg_n"] = [ctx.fields(f).astype(kind) for f in (G.PIC_FIELD_AVG_NE, G.PIC_FIELD_AVG_NI)]
        out["avg_te"] = ctx.fields(G.PIC_FIELD_AVG_TE).astype(kind)
        out["eedf"] = ctx.eedf()[0].astype(kind)
    if case["kind"] == "streamer":
        ctx.adapt()
    return out


def work(case):
    """Per step and particle the record read (6 words and the id) and its 5 changed words
    written, per leaf the corner field and the deposit; ~90 flops per particle (gather, push,
    the collision test) and ~400 per leaf (solve).  A load reads its 48 bytes per particle."""
    if case["kind"] == "ensemble":
        shape = np.random.default_rng([case["instances"], case["nx"]])
        n = leaves = 0
        for i in range(case["instances"]):
            nx = 16 * int(shape.integers(4, case["nx"] // 16 + 1)) if i else case["nx"]
            ppc = float(shape.uniform(20.0, max(21.0, case["ppc"])))
            shape.uniform(), shape.uniform()
            n, leaves = n + 2 * int(nx * 16 * ppc), leaves + nx * 16
    elif case["kind"] in ("streamer", "reload"):
        n = case["particles"]
        leaves = case["nx"] ** 2 + n // 128
    else:
        leaves = case["nx"] * case["ny"]
        n = _loaded(case) * (1 if case["kind"] == "plasma" else 2)
    r = 8 if case["fp64"] else 4
    passes = 2 if case.get("implicit") else 1
    b = case["steps"] * (passes * n * (11 * r + 4) + leaves * (16 * r + 24))
    f = case["steps"] * (passes * n * 90 + leaves * 400)
    if case["kind"] == "reload":
        b += n * (48 + 6 * r + 4)
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------------------------------
# What a pass returns, in 64 bits by plain torch (uniform meshes)
# ---------------------------------------------------------------------------------------
_M32 = 0xFFFFFFFF


def _mulhilo(a, m):
    t = (a & 0xFFFF) * m
    s = (a >> 16) * m + (t >> 16)
    return s >> 16, ((s & 0xFFFF) << 16) | (t & 0xFFFF)


def _philox2(c0, c1, key):
    """First word of Philox2x32-10 (Salmon, Moraes, Dror & Shaw, SC'11)."""
    for _ in range(10):
        hi, lo = _mulhilo(c0, 0xD256D193)
        c0, c1 = hi ^ c1 ^ key, lo
        key = (key + 0x9E3779B9) & _M32
    return c0


def _philox4(c0, c1, c2, c3, seed):
    """Philox4x32-10 (same paper)."""
    k0, k1 = seed & _M32, seed >> 32
    c1, c2, c3 = (torch.full_like(c0, v) for v in (c1, c2, c3))
    for _ in range(10):
        h0, l0 = _mulhilo(c0, 0xD2511F53)
        h1, l1 = _mulhilo(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _u24(r):
    return (r >> 8).double() / 16777216.0


def _direction(uc, up):
    ct = 1 - 2 * uc
    st = (1 - ct * ct).clamp(min=0).sqrt()
    return torch.stack([st * torch.cos(2 * math.pi * up), st * torch.sin(2 * math.pi * up), ct])


def _normals(r):
    u = [_u24(x) for x in r]
    a, b = (-2 * torch.log(1 - u[0])).sqrt(), (-2 * torch.log(1 - u[2])).sqrt()
    return torch.stack([a * torch.cos(2 * math.pi * u[1]), a * torch.sin(2 * math.pi * u[1]), b * torch.cos(2 * math.pi * u[3])])


class _Reference:
    """The particle cycle on a uniform mesh (periodic in y; x periodic or between plates)."""

    def __init__(self, cfg, mesh, parts):
        self.c, self.nx, self.ny, self.h = cfg, mesh["nx0"], mesh["ny0"], mesh["h0"]
        self.px, self.step_no, self.next_id, self.lists = cfg["bc_x"] == PERIODIC, 0, 0, []
        for p in parts:
            x = torch.stack(p)
            ids = torch.arange(self.next_id, self.next_id + x.shape[1], device=x.device)
            self.next_id += x.shape[1]
            o = torch.sort(self.leaf(x), stable=True).indices
            self.lists.append((x[:, o], ids[o]))
        self.dev = parts[0][0].device
        self._lu = None

    def leaf(self, x):
        return torch.floor(x[0] / self.h).long() + self.nx * torch.floor(x[1] / self.h).long()

    def cloud(self, x, fold):
        """The four centres around each particle: indices (i, j) pairs and bilinear fractions."""
        X, Y = x[0] / self.h - 0.5, x[1] / self.h - 0.5
        i, j = torch.floor(X).long(), torch.floor(Y).long()
        fx, fy = X - i, Y - j
        ii = [(i + a) % self.nx if self.px else ((i + a).clamp(0, self.nx - 1) if fold else i + a) for a in (0, 1)]
        return ii, [(j + b) % self.ny for b in (0, 1)], fx, fy

    def weights(self, x):
        out = torch.zeros(self.nx * self.ny, dtype=torch.float64, device=self.dev)
        if self.c["shape"] == NGP:
            return out.index_add_(0, self.leaf(x), x[5])
        ii, jj, fx, fy = self.cloud(x, True)
        for a in (0, 1):
            for b in (0, 1):
                out.index_add_(0, ii[a] + self.nx * jj[b], x[5] * (fx if a else 1 - fx) * (fy if b else 1 - fy))
        return out

    def faces(self, kappa):
        """Conductances toward the right and upper neighbour (and the left wall), [ny, nx]."""
        k = kappa.reshape(self.ny, self.nx)
        gx, gy = 0.5 * (k + torch.roll(k, -1, 1)), 0.5 * (k + torch.roll(k, -1, 0))
        wl = torch.zeros_like(gx[:, 0])
        if not self.px:
            gx = gx.clone()
            gx[:, -1], wl = 2 * k[:, -1], 2 * k[:, 0]
        return gx, gy, wl

    def apply(self, p, f):
        gx, gy, wl = f
        right = torch.roll(p, -1, 1)
        if not self.px:
            right = torch.cat([p[:, 1:], torch.zeros_like(p[:, :1])], 1)
        d = gx * (p - right)
        e = gy * (p - torch.roll(p, -1, 0))
        out = d + e - torch.roll(e, 1, 0)
        if self.px:
            return out - torch.roll(d, 1, 1)
        out[:, 1:] -= d[:, :-1]
        out[:, 0] += wl * p[:, 0]
        return out

    def solve(self, b, kappa):
        nx, ny = self.nx, self.ny
        f = self.faces(kappa if kappa is not None else torch.ones_like(b))
        b = b.reshape(ny, nx).clone()
        lam_y = 2 - 2 * torch.cos(2 * math.pi * torch.arange(ny // 2 + 1, device=self.dev, dtype=torch.float64) / ny)
        if self.px:
            lam = (2 - 2 * torch.cos(2 * math.pi * torch.arange(ny, device=self.dev, dtype=torch.float64) / ny))[:, None] \
                + (2 - 2 * torch.cos(2 * math.pi * torch.arange(nx, device=self.dev, dtype=torch.float64) / nx))[None, :]
            lam[0, 0] = math.inf
            return torch.fft.ifft2(torch.fft.fft2(b - b.mean()) / lam).real
        if self._lu is None:
            t = torch.zeros(nx, nx, dtype=torch.float64, device=self.dev)
            i = torch.arange(nx, device=self.dev)
            t[i, i] = 2.0
            t[i[:-1], i[1:]] = t[i[1:], i[:-1]] = -1.0
            t[0, 0] = t[-1, -1] = 3.0
            t = t[None] + lam_y[:, None, None] * torch.eye(nx, dtype=torch.float64, device=self.dev)
            self._lu = torch.linalg.inv(t)

        def direct(r):  # the operator with kappa = 1, mode by mode in y
            m = torch.fft.rfft(r, dim=0)
            z = torch.view_as_real(m)
            return torch.fft.irfft(torch.view_as_complex(torch.einsum("kij,kjc->kic", self._lu, z).contiguous()), n=ny, dim=0)
        if kappa is None:
            p = direct(b)
            return p + direct(b - self.apply(p, f))
        # conjugate gradients, preconditioned by the kappa = 1 inverse between scalings
        s = kappa.reshape(ny, nx).sqrt()
        p = direct(b / s) / s
        for _ in range(3):
            r = b - self.apply(p, f)
            z = direct(r / s) / s
            d, rz, r0 = z, (r * z).sum(), r.norm()
            for it in range(400):
                q = self.apply(d, f)
                a = rz / (d * q).sum()
                p, r = p + a * d, r - a * q
                if it % 10 == 9 and float(r.norm()) <= 1e-13 * float(b.norm()):
                    break
                z = direct(r / s) / s
                new = (r * z).sum()
                d, rz = z + (new / rz) * d, new
        return p

    def fields(self):
        c, h = self.c, self.h
        q = sum(c["q"][s] * self.weights(x) for s, (x, _) in enumerate(self.lists))
        kappa = None
        if c["implicit"]:
            kappa = 1 + sum(c["dt"] ** 2 * c["q"][s] ** 2 / (c["m"][s] * c["eps0"]) * self.weights(x)
                            for s, (x, _) in enumerate(self.lists)) / (h * h)
        t = self.step_no * c["dt"]
        self.wall = (c["phi_left_dc"] + c["phi_left_amp"] * math.sin(2 * math.pi * c["phi_left_freq"] * t), c["phi_right"])
        b = ((q + c["rho_background"] * h * h) / c["eps0"]).reshape(self.ny, self.nx)
        if not self.px:
            k = torch.ones_like(b) if kappa is None else kappa.reshape(self.ny, self.nx)
            b = b.clone()
            b[:, 0] += 2 * k[:, 0] * self.wall[0]
            b[:, -1] += 2 * k[:, -1] * self.wall[1]
        self.phi = p = self.solve(b.reshape(-1), kappa)
        # face gradients, then the corner field: the mean of the faces that meet there
        if self.px:
            gx = torch.cat([p - torch.roll(p, 1, 1), (p - torch.roll(p, 1, 1))[:, :1]], 1) / h
        else:
            gx = torch.cat([2 * (p[:, :1] - self.wall[0]), p[:, 1:] - p[:, :-1], 2 * (self.wall[1] - p[:, -1:])], 1) / h
        gy = (p - torch.roll(p, 1, 0)) / h
        ex = -0.5 * (gx + torch.roll(gx, 1, 0))
        if self.px:
            ey = 0.5 * (gy + torch.roll(gy, 1, 1))
            ey = -torch.cat([ey, ey[:, :1]], 1)
        else:
            ey = -torch.cat([gy[:, :1], 0.5 * (gy[:, 1:] + gy[:, :-1]), gy[:, -1:]], 1)
        e = torch.stack([ex, ey], 2)
        up = torch.roll(e, -1, 0)
        self.corner = torch.stack([e[:, :-1], e[:, 1:], up[:, :-1], up[:, 1:]], 2).reshape(-1, 4, 2)

    def gather(self, x):
        if self.c["shape"] == NGP:
            l = self.leaf(x)
            u, v = x[0] / self.h - l % self.nx, x[1] / self.h - l // self.nx
            e = self.corner[l]
            return ((1 - u) * (1 - v) * e[:, 0].T + u * (1 - v) * e[:, 1].T + (1 - u) * v * e[:, 2].T + u * v * e[:, 3].T)
        p = self.phi
        if self.px:
            g = torch.cat([p[:, -1:], p, p[:, :1]], 1)
        else:
            g = torch.cat([2 * self.wall[0] - p[:, :1], p, 2 * self.wall[1] - p[:, -1:]], 1)
        ii, jj, fx, fy = self.cloud(x, self.c["shape"] == CIC_EM)
        if self.c["shape"] == CIC_EC:
            v = [[g[jj[b], ii[a] + 1] for b in (0, 1)] for a in (0, 1)]
            if self.px:
                v = [[p[jj[b], ii[a]] for b in (0, 1)] for a in (0, 1)]
            return -torch.stack([(v[1][0] - v[0][0]) * (1 - fy) + (v[1][1] - v[0][1]) * fy,
                                 (v[0][1] - v[0][0]) * (1 - fx) + (v[1][1] - v[1][0]) * fx]) / self.h
        e = -torch.stack([g[:, 2:] - g[:, :-2], torch.roll(p, -1, 0) - torch.roll(p, 1, 0)]) / (2 * self.h)
        return sum(e[:, jj[b], ii[a]] * (fx if a else 1 - fx) * (fy if b else 1 - fy) for a in (0, 1) for b in (0, 1))

    def move(self, mode):
        """mode 0: leapfrog, 1: the implicit predictor (drift only), 2: its corrector."""
        c, dt = self.c, self.c["dt"]
        born = [[], []]
        moved = []
        for s, (x, ids) in enumerate(self.lists):
            x = x.clone()
            old = self.leaf(x)
            if mode == 1:
                dv = x[2:4]
            else:
                dv = c["q"][s] / c["m"][s] * dt * self.gather(x)
                x[2:4] += dv
                if mode == 0:
                    dv = x[2:4]
            x[:2] += dt * dv
            lx, ly = self.nx * self.h, self.ny * self.h
            alive = torch.ones_like(old, dtype=torch.bool)
            if self.px:
                x[0] = torch.remainder(x[0], lx)
                x[0][x[0] >= lx] = 0.0
            else:
                alive = (x[0] >= 0) & (x[0] < lx)
            x[1] = torch.remainder(x[1], ly)
            x[1][x[1] >= ly] = 0.0
            if mode != 1 and c["mcc"]:
                self.collide(s, x, ids, alive, born)
            moved.append((x, ids, old, alive))
        nid = self.next_id
        for s, (x, ids, old, alive) in enumerate(moved):
            new = torch.where(alive, self.leaf(x), -1)
            stay, enter = (new == old) & alive, (new != old) & alive
            groups = [(x[:, stay], ids[stay]), (x[:, enter], ids[enter])]
            if born[s]:
                b = torch.cat(born[s], 1)
                groups.append((b, nid + 2 * torch.arange(b.shape[1], device=self.dev) + s))
                self.next_id = nid + 2 * b.shape[1]
            x, ids = torch.cat([g[0] for g in groups], 1), torch.cat([g[1] for g in groups])
            o = torch.sort(self.leaf(x), stable=True).indices
            self.lists[s] = (x[:, o], ids[o])

    def collide(self, s, x, ids, alive, born):
        c, st = self.c, self.step_no
        m, mn, ngdt = c["m"][s], c["neutral_mass"], c["gas_density"] * c["dt"]
        vt = math.sqrt(c["gas_temperature_ev"] * c["qe"] / mn)
        word = c["instance"] << 24
        u0 = _u24(_philox2(ids, torch.full_like(ids, st), (c["seed"] & _M32) ^ (c["seed"] >> 32) ^ word))
        if s == 0:
            v2 = (x[2:5] ** 2).sum(0)
            eps = 0.5 * m / c["qe"] * v2
            siz = torch.where(eps > c["eps_th_ev"], c["sigma_iz0"] * (1 - c["eps_th_ev"] / eps), torch.zeros_like(eps))
            sig = c["sigma_el"] + siz
            hit = torch.nonzero(alive & (u0 < -torch.expm1(-ngdt * sig * v2.sqrt()))).flatten()
            r = _philox4(ids[hit], word, st, 0, c["seed"])
            v, e, u2 = x[2:5, hit], eps[hit], _u24(r[2])
            ion = _u24(r[1]) * sig[hit] < siz[hit]
            d = _direction(u2, _u24(r[3]))
            cchi = (v * d).sum(0) / v2[hit].sqrt()
            out = (2 * c["qe"] / m * e * (1 - 2 * m / mn * (1 - cchi))).sqrt() * d
            if bool(ion.any()):
                i, rest, ui = hit[ion], e[ion] - c["eps_th_ev"], u2[ion]
                r1 = _philox4(ids[i], word, st, 1, c["seed"])
                w = [_u24(t) for t in r1]
                out[:, ion] = (2 * c["qe"] / m * ui * rest).sqrt() * _direction(w[0], w[1])
                ve = (2 * c["qe"] / m * (1 - ui) * rest).sqrt() * _direction(w[2], w[3])
                vi = vt * _normals(_philox4(ids[i], word, st, 2, c["seed"]))
                born[0].append(torch.cat([x[:2, i], ve, x[5:, i]]))
                born[1].append(torch.cat([x[:2, i], vi, x[5:, i]]))
            x[2:5, hit] = out
            return
        vn = vt * _normals(_philox4(ids, word, st, 2, c["seed"]))
        g = ((x[2:5] - vn) ** 2).sum(0).sqrt()
        hit = torch.nonzero(alive & (u0 < -torch.expm1(-ngdt * c["sigma_el"] * g))).flatten()
        r = _philox4(ids[hit], word, st, 0, c["seed"])
        cm = (m * x[2:5, hit] + mn * vn[:, hit]) / (m + mn)
        x[2:5, hit] = cm + mn / (m + mn) * g[hit] * _direction(_u24(r[2]), _u24(r[3]))

    def step(self):
        if self.c["implicit"]:
            self.move(1)
        self.fields()
        self.sample()
        self.move(2 if self.c["implicit"] else 0)
        self.step_no += 1

    def sample(self):
        """Sums over steps: the weights, the electrons' energy, the potential, the histogram."""
        x = self.lists[0][0]
        eps = 0.5 * self.c["m"][0] / self.c["qe"] * (x[2:5] ** 2).sum(0)
        cell = torch.zeros(self.nx * self.ny, dtype=torch.float64, device=self.dev)
        now = [torch.zeros_like(cell).index_add_(0, self.leaf(y), y[5]) for y, _ in self.lists]
        now += [cell.index_add_(0, self.leaf(x), x[5] * eps), self.phi.reshape(-1)]
        b = torch.floor(eps * (BINS / EV_MAX)).long()
        now.append(torch.zeros(BINS, dtype=torch.float64, device=self.dev).index_add_(0, b[b < BINS], x[5][b < BINS]))
        self.sums = [a + n for a, n in zip(self.sums, now)] if self.step_no else now

    def averages(self):
        n = self.step_no
        we, wi, ee, phi, hist = (a.cpu().numpy() for a in self.sums)
        te = np.where(we > 0, 2.0 / 3.0 * ee / np.where(we > 0, we, 1.0), 0.0)
        return dict(avg_phi=phi / n, avg_n=[we / n / self.h ** 2, wi / n / self.h ** 2], avg_te=te,
                    eedf=hist / (hist.sum() * (EV_MAX / BINS)))

    def counts(self):
        return [torch.bincount(self.leaf(x), minlength=self.nx * self.ny).double().cpu().numpy() for x, _ in self.lists]


def exact(case, seed):
    """Uniform meshes.  On an adaptive mesh (streamer, reload) a pass has no plain 64-bit
    counterpart within the time: its refinement, splitting and merging decide by thresholds."""
    if case["kind"] in ("streamer", "reload"):
        return None
    refs = [_Reference(*s) for s in _inputs(case, seed)]
    for r in refs:
        for _ in range(case["steps"]):
            r.step()
    if case["kind"] == "ensemble":
        return {"phi": [r.phi.reshape(-1).cpu().numpy() for r in refs]}
    r = refs[0]
    out = {"phi": r.phi.reshape(-1).cpu().numpy()}
    if case["steps"] <= 4:
        out["e"] = r.corner.cpu().numpy()
        out["n"] = r.counts()
    if case.get("particles_out"):
        for s in range(len(r.lists)):
            # (in FP32 a rounding can move a particle, and so the order of all that follow)
            x = r.lists[s][0]
            out["particles%d" % s] = ([_padded(a.cpu().numpy(), _loaded(case), np.float64) for a in x] if case["fp64"]
                                      else [None] * 6) + [None, None]
    if case.get("diag"):
        out.update(r.averages())
    return out
