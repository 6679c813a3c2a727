// Poisson solve on the composite leaf mesh (§3: multigrid Poisson solver with the potential
// at cell centres).  Mixed precision: the residual b - A phi, its norm and the correction
// phi += e are FP64 (iterative refinement); each correction e comes from one FP32
// geometric-multigrid V-cycle over the tree-clamped and root-coarsened levels, with two
// red-black Gauss-Seidel sweeps before and after the coarse correction, summed restriction
// and piecewise-constant prolongation.  The coarsest level, up to 128 cells, is solved by its
// dense inverse: the explicit scheme's in FP64, formed on the host once per root grid and walls;
// the implicit scheme's, whose operator changes every step, in FP32 on the device once per
// solve.  A larger one, or one that is singular between Neumann walls, goes to conjugate
// gradients.  Levels of at most 8192 cells live in one block's shared memory; when every level
// does, the whole solve (FP64 residual, V-cycles, convergence test) is a single launch of
// thread-block clusters, one per instance of a batch, that spread the FP64 work over their SMs.
// Larger meshes run one CUDA graph per solve whose WHILE node repeats the cycle until the
// device decides.
#include <algorithm>
#include <array>
#include <cmath>

#include <cooperative_groups.h>

#include "pic_internal.cuh"

namespace gbpic {

namespace {
constexpr int kT = 256;
constexpr int kRedBlocks = 304;  // 2 x 152 SMs: fixed so that the FP64 sums are deterministic
constexpr int kNu = 2;          // red-black Gauss-Seidel sweeps before and after the coarse correction
constexpr double kCoarseTol2 = 1e-10;  // coarsest solve (multi-block path): ||r|| <= 1e-5 ||b||
constexpr float kSmCoarseTol2 = 1e-6f; // coarsest solve inside a V-cycle in shared memory: 1e-3
inline unsigned blocks_for(int64_t n, int t = kT) { return (unsigned)std::max<int64_t>(1, (n + t - 1) / t); }

// Sum over a block of kT threads as a fixed tree, valid in thread 0.
__device__ __forceinline__ double block_sum(double v) {
    __shared__ double sh[kT / 32];
    static_assert(kT == 256, "eight warps");
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, o);
    __syncthreads();  // (the previous sum's words are read)
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    return ((sh[0] + sh[1]) + (sh[2] + sh[3])) + ((sh[4] + sh[5]) + (sh[6] + sh[7]));
}

// out = sums of the block partials (one warp: lanes in a fixed order, then a fixed tree,
// so the result does not depend on timing).
__global__ void k_finish_sums(int nparts, const double *__restrict__ part, double *__restrict__ out) {
    pdl_chain();
    const int lane = threadIdx.x & 31;
    if (threadIdx.x >= 32) return;
    double a = 0.0, b = 0.0;
    for (int k = lane; k < nparts; k += 32) { a += part[2 * k]; b += part[2 * k + 1]; }
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xFFFFFFFFu, a, o);
        b += __shfl_down_sync(0xFFFFFFFFu, b, o);
    }
    if (lane == 0) { out[0] = a; out[1] = b; }
}

// The larger of two relative residuals, NaN if either is NaN: a non-finite residual (NaN or
// Inf in the charge density or the potential) stays visible to the host.
__device__ __forceinline__ double worst_residual(double a, double b) {
    return (a != a || b != b) ? __longlong_as_double(0x7FF8000000000000ll) : fmax(a, b);
}

// The off-diagonal value a code stands for (LevelOp).
template <typename T> __device__ __forceinline__ T op_value(uint32_t k) {
    return k == 1u ? (T)-1 : (k == 2u ? (T)(-2.0 / 3.0) : (T)(1.0 / 3.0));
}

// r = b - A phi (FP64, handed on in FP32) with r^2 (and, before the first cycle, b^2) summed per
// block, then, in the block that arrives last on the ticket counter (after a fence, so every
// block's sums are visible), the block sums added as a fixed tree, whether another cycle runs
// (the condition of the graph's WHILE node, from the squared norms; first = 1 before the first
// cycle), the solve's statistics, and the counter reset for the next launch.  stats[3] keeps
// ||b||^2.  The decision is on the cycle's critical path: with one warp adding 304 pairs and the
// root and division before it, a 256 x 256 solve of 6 cycles took 0.302 ms, so 0.283 ms.
__global__ void __launch_bounds__(kT) k_residual_decide(int64_t n, const int32_t *__restrict__ col,
                                                        const uint16_t *__restrict__ code,
                                                        const double *__restrict__ val, const double *__restrict__ diag,
                                                        const double *__restrict__ phi, const double *__restrict__ b,
                                                        float *__restrict__ r32, double *__restrict__ part,
                                                        uint32_t *__restrict__ ticket, cudaGraphConditionalHandle h,
                                                        double tol, int maxc, double *__restrict__ stats, int first) {
    pdl_chain();
    __shared__ bool last;
    double rr = 0.0, bb = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double ax = diag[i] * phi[i];
        if (code) {
            const uint32_t m = code[i];
#pragma unroll
            for (int j = 0; j < kEll; ++j)
                if ((m >> (2 * j)) & 3u) ax += op_value<double>((m >> (2 * j)) & 3u) * phi[col[(int64_t)j * n + i]];
        } else {
#pragma unroll
            for (int j = 0; j < kEll; ++j) {
                const int32_t c = col[(int64_t)j * n + i];
                if (c >= 0) ax += val[(int64_t)j * n + i] * phi[c];
            }
        }
        const double bi = b[i], ri = bi - ax;
        r32[i] = (float)ri;
        rr += ri * ri;
        if (first) bb += bi * bi;
    }
    const double s1 = block_sum(rr);
    const double s2 = first ? block_sum(bb) : 0.0;
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = s1;
        part[2 * blockIdx.x + 1] = s2;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    static_assert(kRedBlocks <= 2 * kT, "two block sums per thread");
    const int k0 = threadIdx.x, k1 = k0 + kT;
    const double tot = block_sum((k0 < kRedBlocks ? __ldcg(part + 2 * k0) : 0.0) +
                                 (k1 < kRedBlocks ? __ldcg(part + 2 * k1) : 0.0));
    double btot = 0.0;
    if (first)
        btot = block_sum((k0 < kRedBlocks ? __ldcg(part + 2 * k0 + 1) : 0.0) +
                         (k1 < kRedBlocks ? __ldcg(part + 2 * k1 + 1) : 0.0));
    if (threadIdx.x == 0) {
        if (!first) btot = stats[3];
        const double cyc = first ? 0.0 : stats[0] + 1.0;
        const bool done = tot <= tol * tol * (btot > 0.0 ? btot : 1.0) || cyc >= (double)maxc;
        cudaGraphSetConditional(h, done ? 0u : 1u);
        *ticket = 0u;
        stats[0] = cyc;
        if (first) stats[3] = btot;
        if (done) {
            const double rel = btot > 0.0 ? sqrt(tot / btot) : sqrt(tot);
            stats[1] = rel;
            stats[2] = worst_residual(stats[2], rel);
        }
    }
}

// Zero-mean projections for a fully periodic (singular) problem: area weights a = s^2.
__global__ void k_area_moments(int64_t n, const uint8_t *__restrict__ lev, int lmax, const double *__restrict__ v,
                               double *__restrict__ part) {
    double sv = 0.0, sa = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double s = (double)(1 << (lmax - lev[i]));
        sv += v[i];
        sa += s * s;
    }
    const double s1 = block_sum(sv), s2 = block_sum(sa);
    if (threadIdx.x == 0) { part[2 * blockIdx.x] = s1; part[2 * blockIdx.x + 1] = s2; }
}
__global__ void k_area_weighted(int64_t n, const uint8_t *__restrict__ lev, int lmax, const double *__restrict__ v,
                                double *__restrict__ part) {
    pdl_chain();
    double sv = 0.0, sa = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double s = (double)(1 << (lmax - lev[i]));
        sv += s * s * v[i];
        sa += s * s;
    }
    const double s1 = block_sum(sv), s2 = block_sum(sa);
    if (threadIdx.x == 0) { part[2 * blockIdx.x] = s1; part[2 * blockIdx.x + 1] = s2; }
}
// v -= mode * (sum / area_total): mode 0 subtracts an area-proportional share (RHS
// compatibility), mode 1 a constant (zero area-weighted mean of the potential).
__global__ void k_project(int64_t n, const uint8_t *__restrict__ lev, int lmax, const double *__restrict__ sums,
                          double *__restrict__ v, int mode) {
    pdl_chain();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double s = (double)(1 << (lmax - lev[i]));
    const double k = sums[0] / sums[1];
    v[i] -= mode == 0 ? k * s * s : k;
}

// Initial guess of a solve: phi <- 2 phi - phi_prev (linear extrapolation in time of the last
// two solutions), phi_prev <- phi.  With only one earlier solve: phi_prev <- phi.
__global__ void k_extrapolate(int64_t n, double *__restrict__ phi, double *__restrict__ prev, int both) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double p = phi[i];
    if (both) phi[i] = 2.0 * p - prev[i];
    prev[i] = p;
}

// The rows of a level swept by many blocks.  An explicit scheme's off-diagonal values are -1
// (same level), -2/3 (across a level step) and 1/3 (the sibling there): `code` holds two bits
// per ELL slot (0: empty), so a row is read as 2 bytes and its 4 to 8 columns instead of 64
// bytes.  The implicit scheme's values come from `val` (code null).
struct LevelOp {
    int64_t n;
    const int32_t *col;
    const uint16_t *code;
    const float *val, *dinv;
    const uint8_t *color;
};
struct OpRow {
    int32_t c[kEll];
    float v[kEll];
};
template <bool CODED> __device__ __forceinline__ void op_row(const LevelOp &A, int64_t i, OpRow &r) {
    if constexpr (CODED) {
        const uint32_t m = A.code[i];
#pragma unroll
        for (int j = 0; j < kEll; ++j) {
            const uint32_t k = (m >> (2 * j)) & 3u;
            r.c[j] = k ? A.col[(int64_t)j * A.n + i] : -1;
            r.v[j] = op_value<float>(k);
        }
    } else {
#pragma unroll
        for (int j = 0; j < kEll; ++j) {
            r.c[j] = A.col[(int64_t)j * A.n + i];
            r.v[j] = A.val[(int64_t)j * A.n + i];
        }
    }
}

// Each of the following kernels of a cycle loads what no kernel of the cycle writes (operator,
// colours, parents) and what was written two or more kernels earlier before it waits for its
// predecessor, so that after the wait one gather, a few additions and a store are left: the
// solve is a chain of dozens of such kernels, bound by their latency.  Early streamer (24,500
// leaves, ~2 cycles): 0.303 -> 0.217 ms per solve; 256 x 256 periodic, 6 cycles: 0.566 -> 0.407 ms.

// One colour of a red-black Gauss-Seidel sweep, written out of place so that the result does
// not depend on thread order (cells of the same colour can touch on a non-uniform mesh):
// colour-c cells get D^-1 (b - offdiag x_in), others copy x_in.  With phi non-null (the
// finest level's last half sweep of a cycle) the result is also added to the potential.
template <bool CODED>
__global__ void __launch_bounds__(kT) k_rbgs_half(const LevelOp A, int c, const float *__restrict__ b,
                                                  const float *__restrict__ xin, float *__restrict__ xout,
                                                  double *__restrict__ phi) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = i < A.n, mine = in && A.color[i] == c;
    OpRow r;
    float bi = 0.0f, di = 0.0f;
    if (mine) {
        op_row<CODED>(A, i, r);
        bi = b[i];
        di = A.dinv[i];
    }
    pdl_chain();
    if (!in) return;
    float x;
    if (mine) {
        float off = 0.0f;
#pragma unroll
        for (int j = 0; j < kEll; ++j)
            if (r.c[j] >= 0) off = fmaf(r.v[j], xin[r.c[j]], off);
        x = di * (bi - off);
    } else {
        x = xin[i];
    }
    xout[i] = x;
    if (phi) phi[i] += (double)x;
}

// The first two half sweeps of a pre-smoothing from x = 0 in one kernel: the first (colour 0
// from zero) leaves t = D^-1 (b - 0) on colour 0 and 0 elsewhere, which the second (colour 1)
// forms on the fly; the same arithmetic as the two half sweeps, so the same values.
template <bool CODED>
__global__ void __launch_bounds__(kT) k_rbgs_first(const LevelOp A, const float *__restrict__ b, float *__restrict__ xout) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = i < A.n, mine = in && A.color[i] == 1;
    OpRow r;
    float dn[kEll], di = 0.0f;
    if (in) di = A.dinv[i];
    if (mine) {
        op_row<CODED>(A, i, r);
#pragma unroll
        for (int j = 0; j < kEll; ++j) {
            dn[j] = 0.0f;
            if (r.c[j] >= 0) {
                if (A.color[r.c[j]] == 0) dn[j] = A.dinv[r.c[j]];
                else r.c[j] = -2;  // its value is zero: the term is v * 0
            }
        }
    }
    pdl_chain();
    if (!in) return;
    if (!mine) {
        xout[i] = di * (b[i] - 0.0f);
        return;
    }
    float off = 0.0f;
#pragma unroll
    for (int j = 0; j < kEll; ++j) {
        if (r.c[j] >= 0) off = fmaf(r.v[j], dn[j] * (b[r.c[j]] - 0.0f), off);
        else if (r.c[j] == -2) off = fmaf(r.v[j], 0.0f, off);
    }
    xout[i] = di * (b[i] - off);
}

// Injection of the coarse correction (x += xc[parent]) fused into the first half sweep after
// it (colour 0): every value the sweep reads gets its correction added on the way, with the
// same additions as a separate injection pass.
template <bool CODED>
__global__ void __launch_bounds__(kT) k_rbgs_half_prolong(const LevelOp A, const float *__restrict__ b,
                                                          const float *__restrict__ xin,
                                                          const int32_t *__restrict__ parent,
                                                          const float *__restrict__ xc, float *__restrict__ xout) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = i < A.n, mine = in && A.color[i] == 0;
    OpRow r;
    float xn[kEll], bi = 0.0f, di = 0.0f, xi = 0.0f;
    int32_t pi = 0;
    if (mine) {
        op_row<CODED>(A, i, r);
        bi = b[i];
        di = A.dinv[i];
#pragma unroll
        for (int j = 0; j < kEll; ++j) {
            xn[j] = 0.0f;
            if (r.c[j] >= 0) {
                xn[j] = xin[r.c[j]];
                r.c[j] = parent[r.c[j]];
            }
        }
    } else if (in) {
        pi = parent[i];
        xi = xin[i];
    }
    pdl_chain();
    if (!in) return;
    if (!mine) {
        xout[i] = xi + xc[pi];
        return;
    }
    float off = 0.0f;
#pragma unroll
    for (int j = 0; j < kEll; ++j)
        if (r.c[j] >= 0) off = fmaf(r.v[j], xn[j] + xc[r.c[j]], off);
    xout[i] = di * (bi - off);
}

// Coarse right-hand side: summed residuals of the children (four threads per coarse cell, one
// child each, added in child order).
template <bool CODED>
__global__ void __launch_bounds__(kT) k_restrict_residual(int64_t nc, const int32_t *__restrict__ child4,
                                                          const LevelOp A, const float *__restrict__ bf,
                                                          const float *__restrict__ xf, float *__restrict__ bc) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int32_t i = t < 4 * nc ? child4[t] : -1;
    OpRow r;
    float bi = 0.0f, di = 1.0f;
    if (i >= 0) {
        op_row<CODED>(A, i, r);
        bi = bf[i];
        di = A.dinv[i];
    }
    pdl_chain();
    float res = 0.0f;
    if (i >= 0) {
        float ax = xf[i] / di;
#pragma unroll
        for (int j = 0; j < kEll; ++j)
            if (r.c[j] >= 0) ax = fmaf(r.v[j], xf[r.c[j]], ax);
        res = bi - ax;
    }
    const float r1 = __shfl_down_sync(0xFFFFFFFFu, res, 1, 4), r2 = __shfl_down_sync(0xFFFFFFFFu, res, 2, 4),
                r3 = __shfl_down_sync(0xFFFFFFFFu, res, 3, 4);
    if (t < 4 * nc && (t & 3) == 0) bc[t >> 2] = ((res + r1) + r2) + r3;
}

// 1 / d of a diagonal d = 1 .. 6, rounded once (the constants the divisions would give).
__device__ __forceinline__ float diag_inv(float d) {
    return d == 4.0f ? 0.25f : (d == 3.0f ? 1.0f / 3.0f : (d == 5.0f ? 0.2f : (d == 6.0f ? 1.0f / 6.0f : (d == 2.0f ? 0.5f : 1.0f))));
}

// ---- uniform levels of many blocks ---------------------------------------------------------
// A level of root boxes (row-major, even nx and ny: it coarsens) needs no operator arrays, and a
// block can form a tile's four half sweeps by itself when it also forms those of a frame of
// kUH cells around it (each half sweep shrinks the valid region by one cell): the whole
// pre-smoothing and restriction is one kernel, the whole post-smoothing another, instead of
// eight, with the arithmetic and so the values of the half-sweep kernels.  The frame doubles
// the work of a 32 x 16 tile, which the chain's latency hides.  256 x 256 periodic, 6 cycles:
// 0.407 -> 0.302 ms per solve.
constexpr int kUX = 32, kUY = 16, kUH = kNu * 2;
constexpr int kUSX = kUX + 2 * kUH, kUSY = kUY + 2 * kUH, kUHalf = kUSX * kUSY / 2;
constexpr int kUCells = (kUHalf + kT - 1) / kT;  // cells of each colour per thread
struct UniLevel { int nx, ny, bcx, bcy; };
struct UniTile {
    int o[2][kUCells];    // tile word of the thread's cells of each colour (-1: none or outside)
    float di[2][kUCells];
};
__device__ __forceinline__ bool uni_wrap(int &g, int n, int bc) {
    if (g >= 0 && g < n) return true;
    if (bc != PIC_BC_PERIODIC) return false;
    g %= n;
    if (g < 0) g += n;
    return true;
}
__device__ __forceinline__ float uni_dinv(const UniLevel &A, int gx, int gy) {
    const int wx = A.bcx == PIC_BC_DIRICHLET ? 2 : (A.bcx == PIC_BC_PERIODIC ? 1 : 0);
    const int wy = A.bcy == PIC_BC_DIRICHLET ? 2 : (A.bcy == PIC_BC_PERIODIC ? 1 : 0);
    return diag_inv((float)((gx > 0 ? 1 : wx) + (gx < A.nx - 1 ? 1 : wx) + (gy > 0 ? 1 : wy) + (gy < A.ny - 1 ? 1 : wy)));
}
// The thread's cells of the tile at (tx, ty) and its frame.
__device__ __forceinline__ void uni_tile(const UniLevel &A, int tx, int ty, UniTile &t, int (&src)[2][kUCells]) {
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int k = 0; k < kUCells; ++k) {
            const int h = (int)threadIdx.x + kT * k;
            const int ly = h / (kUSX / 2), lx = 2 * (h - ly * (kUSX / 2)) + ((c + ly) & 1);
            int gx = tx - kUH + lx, gy = ty - kUH + ly;
            t.o[c][k] = src[c][k] = -1;
            t.di[c][k] = 0.0f;
            if (h < kUHalf && uni_wrap(gx, A.nx, A.bcx) && uni_wrap(gy, A.ny, A.bcy)) {
                // (cells on the frame's rim have neighbours outside it: loaded, never swept)
                const bool rim = lx == 0 || lx == kUSX - 1 || ly == 0 || ly == kUSY - 1;
                src[c][k] = gy * A.nx + gx;
                t.o[c][k] = (ly * kUSX + lx) | (rim ? 1 << 30 : 0);
                t.di[c][k] = uni_dinv(A, gx, gy);
            }
        }
}
// One half sweep over the tile (from zero: no neighbour is read, the rim included).
template <int C, bool ZERO> __device__ __forceinline__ void uni_half(const UniTile &t, float *xs, const float (&b)[2][kUCells]) {
#pragma unroll
    for (int k = 0; k < kUCells; ++k) {
        const int o = t.o[C][k];
        if (o < 0 || (!ZERO && (o >> 30))) continue;
        const int w = o & 0xFFFF;
        if (ZERO) xs[w] = t.di[C][k] * b[C][k];
        else xs[w] = t.di[C][k] * (b[C][k] + (((xs[w - 1] + xs[w + 1]) + xs[w - kUSX]) + xs[w + kUSX]));
    }
}

__global__ void __launch_bounds__(kT) k_uni_down(UniLevel A, const float *__restrict__ b, float *__restrict__ x,
                                                 float *__restrict__ bc) {
    __shared__ float xs[kUSX * kUSY], bs[kUSX * kUSY];
    const int tiles_x = (A.nx + kUX - 1) / kUX;
    const int tx = (int)(blockIdx.x % tiles_x) * kUX, ty = (int)(blockIdx.x / tiles_x) * kUY;
    UniTile t;
    int src[2][kUCells];
    float bb[2][kUCells];
    uni_tile(A, tx, ty, t, src);
    for (int k = threadIdx.x; k < kUSX * kUSY; k += kT) xs[k] = 0.0f;
    pdl_chain();
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int k = 0; k < kUCells; ++k) bb[c][k] = src[c][k] >= 0 ? b[src[c][k]] : 0.0f;
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int k = 0; k < kUCells; ++k)
            if (t.o[c][k] >= 0) bs[t.o[c][k] & 0xFFFF] = bb[c][k];
    uni_half<0, true>(t, xs, bb);
    __syncthreads();
    uni_half<1, false>(t, xs, bb);
    __syncthreads();
#pragma unroll
    for (int k = 1; k < kNu; ++k) {
        uni_half<0, false>(t, xs, bb);
        __syncthreads();
        uni_half<1, false>(t, xs, bb);
        __syncthreads();
    }
    for (int k = threadIdx.x; k < kUX * kUY; k += kT) {
        const int ly = k / kUX, lx = k % kUX, gx = tx + lx, gy = ty + ly;
        if (gx < A.nx && gy < A.ny) x[(int64_t)gy * A.nx + gx] = xs[(ly + kUH) * kUSX + lx + kUH];
    }
    // two threads per coarse cell, one row of children each
    static_assert(kUX * kUY / 2 == kT, "one residual pair per thread");
    const int q = (int)threadIdx.x >> 1, row = (int)threadIdx.x & 1;
    const int cx = q % (kUX / 2), cy = q / (kUX / 2);
    const int gx = tx + 2 * cx, gy = ty + 2 * cy + row;
    float res[2] = {0.0f, 0.0f};
    const bool in = gx < A.nx && gy < A.ny;
    if (in)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int w = (2 * cy + row + kUH) * kUSX + 2 * cx + k + kUH;
            const float ax = (((xs[w] / uni_dinv(A, gx + k, gy) - xs[w - 1]) - xs[w + 1]) - xs[w - kUSX]) - xs[w + kUSX];
            res[k] = bs[w] - ax;
        }
    const float r2 = __shfl_down_sync(0xFFFFFFFFu, res[0], 1), r3 = __shfl_down_sync(0xFFFFFFFFu, res[1], 1);
    if (in && row == 0) bc[(int64_t)(gy >> 1) * (A.nx >> 1) + (gx >> 1)] = ((res[0] + res[1]) + r2) + r3;
}

// xin: the pre-smoothed values; xc: the coarse correction (needed on colour 1 only: the first
// half sweep overwrites colour 0 without reading it).
__global__ void __launch_bounds__(kT) k_uni_up(UniLevel A, const float *__restrict__ b, const float *__restrict__ xin,
                                               const float *__restrict__ xc, float *__restrict__ xout,
                                               double *__restrict__ phi) {
    __shared__ float xs[kUSX * kUSY];
    const int tiles_x = (A.nx + kUX - 1) / kUX;
    const int tx = (int)(blockIdx.x % tiles_x) * kUX, ty = (int)(blockIdx.x / tiles_x) * kUY;
    UniTile t;
    int src[2][kUCells];
    float bb[2][kUCells], x1[kUCells];
    uni_tile(A, tx, ty, t, src);
    for (int k = threadIdx.x; k < kUSX * kUSY; k += kT) xs[k] = 0.0f;
#pragma unroll
    for (int k = 0; k < kUCells; ++k) {  // written before the coarser levels' kernels
        bb[0][k] = src[0][k] >= 0 ? b[src[0][k]] : 0.0f;
        bb[1][k] = src[1][k] >= 0 ? b[src[1][k]] : 0.0f;
        x1[k] = src[1][k] >= 0 ? xin[src[1][k]] : 0.0f;
    }
    pdl_chain();
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kUCells; ++k)
        if (src[1][k] >= 0) {
            const int gy = src[1][k] / A.nx, gx = src[1][k] - gy * A.nx;
            xs[t.o[1][k] & 0xFFFF] = x1[k] + xc[(int64_t)(gy >> 1) * (A.nx >> 1) + (gx >> 1)];
        }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kNu; ++k) {
        uni_half<0, false>(t, xs, bb);
        __syncthreads();
        uni_half<1, false>(t, xs, bb);
        __syncthreads();
    }
    for (int k = threadIdx.x; k < kUX * kUY; k += kT) {
        const int ly = k / kUX, lx = k % kUX, gx = tx + lx, gy = ty + ly;
        if (gx < A.nx && gy < A.ny) {
            const float v = xs[(ly + kUH) * kUSX + lx + kUH];
            xout[(int64_t)gy * A.nx + gx] = v;
            if (phi) phi[(int64_t)gy * A.nx + gx] += (double)v;
        }
    }
}

// One-block Jacobi-preconditioned CG on the coarsest level (symmetric: one uniform level).  With
// phi non-null (a mesh that does not coarsen: the coarsest level is the finest) the result is also
// added to the potential.
__global__ void __launch_bounds__(1024) k_coarse_cg(int64_t n, const int32_t *__restrict__ col,
                                                    const float *__restrict__ val, const float *__restrict__ dinv,
                                                    const float *__restrict__ b, float *__restrict__ x,
                                                    float *__restrict__ r, float *__restrict__ p,
                                                    float *__restrict__ q, int singular, int maxit,
                                                    double *__restrict__ phi) {
    pdl_chain();
    __shared__ double red[32];
    __shared__ double bcast;
    auto bsum = [&](double v) -> double {
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, o);
        if (lane == 0) red[wid] = v;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
            bcast = s;
        }
        __syncthreads();
        const double out = bcast;
        __syncthreads();
        return out;
    };
    double mb = 0.0;
    if (singular) {
        for (int64_t i = threadIdx.x; i < n; i += blockDim.x) mb += b[i];
        mb = bsum(mb) / (double)n;
    }
    double rz = 0.0, bb = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        const float ri = b[i] - (float)mb;
        x[i] = 0.0f;
        r[i] = ri;
        const float zi = dinv[i] * ri;
        p[i] = zi;
        rz += (double)ri * zi;
        bb += (double)ri * ri;
    }
    rz = bsum(rz);
    bb = bsum(bb);
    if (bb == 0.0) return;
    for (int it = 0; it < maxit; ++it) {
        double pq = 0.0;
        for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
            float ax = p[i] / dinv[i];
            for (int j = 0; j < kEll; ++j) {
                const int32_t c = col[(int64_t)j * n + i];
                if (c >= 0) ax = fmaf(val[(int64_t)j * n + i], p[c], ax);
            }
            q[i] = ax;
            pq += (double)p[i] * ax;
        }
        pq = bsum(pq);
        if (pq <= 0.0) break;
        const float alpha = (float)(rz / pq);
        double rr = 0.0, rz2 = 0.0;
        for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
            x[i] += alpha * p[i];
            const float ri = r[i] - alpha * q[i];
            r[i] = ri;
            rr += (double)ri * ri;
            rz2 += (double)ri * dinv[i] * ri;
        }
        rr = bsum(rr);
        rz2 = bsum(rz2);
        if (rr <= kCoarseTol2 * bb) break;
        const float beta = (float)(rz2 / rz);
        rz = rz2;
        for (int64_t i = threadIdx.x; i < n; i += blockDim.x) p[i] = dinv[i] * r[i] + beta * p[i];
        __syncthreads();
    }
    if (singular) {
        double mx = 0.0;
        for (int64_t i = threadIdx.x; i < n; i += blockDim.x) mx += x[i];
        mx = bsum(mx) / (double)n;
        for (int64_t i = threadIdx.x; i < n; i += blockDim.x) x[i] -= (float)mx;
    }
    if (phi)
        for (int64_t i = threadIdx.x; i < n; i += blockDim.x) phi[i] += (double)x[i];
}

// ---- levels held in shared memory by one block (n <= kSmallN cells each) ----------------
constexpr int kSmallN = 8192;          // 8 cells per thread of a 1024-thread block
constexpr int kMaxSmallLevels = 16;
constexpr int kSmallSmemCap = 201 * 1024;  // the levels' vectors
constexpr int kSmallSmemMax = 222 * 1024;  // with the sums' buffers and the coarsest inverse
constexpr int kDirectN = 128;  // coarsest levels up to this size are solved by a dense inverse

// A level of root boxes only (no refinement) is a row-major nx x ny grid whose operator is the
// 5-point stencil, applied from the cell index without the ELL arrays (`uniform`).  Every such
// level but the coarsest has even nx and ny, so its red-black colouring is proper (also across
// a periodic wrap), and its vectors are stored by colour (`fast`): cell (ix, iy) of colour
// c = (ix + iy) & 1 at c * hs + iy * nx / 2 + ix / 2.
struct SmallLevel {
    int32_t n;
    const int32_t *col;
    const float *val, *dinv;
    const float *face;      // implicit scheme, uniform levels: each cell's right [n] and upper [n] conductance
    const uint8_t *color;
    const int32_t *child4;  // children (in the finer level) of this level's cells
    const int32_t *parent;  // this level's cells -> cells of the next coarser level
    int32_t off;            // smem offset (floats) of x; b follows at off + boff
    int32_t boff;
    int32_t uniform, nx, ny;
    uint32_t nx_magic;   // floor(i / nx) == mdiv(i, nx_magic) for every cell index i < n
    uint32_t nxh_magic;  // the same for nx / 2 (uniform levels with even nx)
    int32_t fast, half, hs;  // stored by colour: cells per colour, stride between the colours (half + 4)
    int32_t nthr, rows, strips;  // threads of the level, rows of a strip (2 or 4), strips per thread
};
struct SmallDesc {
    int nlev;  // levels g0 .. g0 + nlev - 1 live in shared memory
    int bcx, bcy;
    SmallLevel lv[kMaxSmallLevels];
    int32_t off_cg;  // smem offset of the coarsest CG vectors r, p, q (3 n)
    int32_t smem_floats;  // a multiple of 4
    const double *cinv;  // coarsest level: dense inverse (n rows of n | 1 words; FP64, or FP32 with build 2), or null
    int32_t build;       // FP32 inverse (sm_build_inverse): 1: formed by each launch, 2: in cinv, formed once per solve
    int32_t inv_words;   // FP64 words of the inverse in shared memory, else 0
};

// floor(i / d) by a multiply-high reciprocal m = floor((2^32 - 1) / d) + 1; m = 0 stands for
// d = 1 (whose reciprocal 2^32 has no 32-bit form).
__host__ __device__ __forceinline__ uint32_t mdiv_magic(uint32_t d) { return d <= 1u ? 0u : 0xFFFFFFFFu / d + 1u; }
__device__ __forceinline__ int mdiv(int i, uint32_t m) { return m ? (int)__umulhi((uint32_t)i, m) : i; }

// Where cell i of a level sits in its x (and b) vector.
__device__ __forceinline__ int sm_pos(const SmallLevel &L, int i) {
    if (!L.fast) return i;
    const int iy = mdiv(i, L.nx_magic), ix = i - iy * L.nx;
    return ((ix + iy) & 1) * L.hs + iy * (L.nx >> 1) + (ix >> 1);
}

// Neighbour sum s and diagonal d of row i, so that (A x)_i = d x_i - s.  Uniform levels:
// face conductance 1 to each neighbour, 2 to a Dirichlet wall, none at a Neumann wall.
template <typename T>
__device__ __forceinline__ T uni_row(int nx, int ny, uint32_t magic, int bcx, int bcy, const T *x, int i, int &dd) {
    const int iy = mdiv(i, magic), ix = i - iy * nx;
    T l = 0, r = 0, dn = 0, up = 0;
    dd = 0;
    if (ix > 0) { l = x[i - 1]; dd += 1; }
    else if (bcx == PIC_BC_PERIODIC) { l = x[i + nx - 1]; dd += 1; }
    else if (bcx == PIC_BC_DIRICHLET) dd += 2;
    if (ix < nx - 1) { r = x[i + 1]; dd += 1; }
    else if (bcx == PIC_BC_PERIODIC) { r = x[i - nx + 1]; dd += 1; }
    else if (bcx == PIC_BC_DIRICHLET) dd += 2;
    if (iy > 0) { dn = x[i - nx]; dd += 1; }
    else if (bcy == PIC_BC_PERIODIC) { dn = x[i + (ny - 1) * nx]; dd += 1; }
    else if (bcy == PIC_BC_DIRICHLET) dd += 2;
    if (iy < ny - 1) { up = x[i + nx]; dd += 1; }
    else if (bcy == PIC_BC_PERIODIC) { up = x[i - (ny - 1) * nx]; dd += 1; }
    else if (bcy == PIC_BC_DIRICHLET) dd += 2;
    return ((l + r) + dn) + up;
}

template <typename Desc>
__device__ __forceinline__ float sm_row(const Desc &D, const SmallLevel &L, const float *x, int i, float &d,
                                        float &dinv) {
    if (L.uniform) {
        int dd;
        const float s = uni_row<float>(L.nx, L.ny, L.nx_magic, D.bcx, D.bcy, x, i, dd);
        d = (float)dd;
        dinv = __frcp_rn(d);
        return s;
    }
    float off = 0.0f;
#pragma unroll
    for (int j = 0; j < kEll; ++j) {
        const int32_t c = L.col[(int64_t)j * L.n + i];
        if (c >= 0) off = fmaf(L.val[(int64_t)j * L.n + i], x[c], off);
    }
    dinv = L.dinv[i];
    d = __frcp_rn(dinv);
    return -off;
}
template <typename Desc>
__device__ __forceinline__ float sm_row(const Desc &D, const SmallLevel &L, const float *x, int i, float &d) {
    float dinv;
    return sm_row(D, L, x, i, d, dinv);
}

// Red-black Gauss-Seidel sweep of an ELL level in shared memory; each colour's new values are
// computed from the current vector before any is written (cells of one colour can touch on a
// non-uniform mesh, and the result must not depend on thread order).  The block has 1024
// threads; thread t owns cells t + 1024 k, k < 8, so the new values stay in registers.
constexpr int kPerThread = kSmallN / 1024;
__device__ __noinline__ void sm_smooth(const SmallDesc &D, const SmallLevel &L, float *x, const float *b, bool first) {
    if (first) {
        for (int i = threadIdx.x; i < L.n; i += blockDim.x) x[i] = 0.0f;
        __syncthreads();
    }
    for (int c = 0; c < 2; ++c) {
        float t[kPerThread];
        bool mine[kPerThread];
#pragma unroll
        for (int k = 0; k < kPerThread; ++k) {
            const int i = threadIdx.x + 1024 * k;
            mine[k] = i < L.n && L.color[i] == c;
            t[k] = 0.0f;
            if (mine[k]) {
                float d, dinv;
                const float sn = sm_row(D, L, x, i, d, dinv);
                t[k] = (b[i] + sn) * dinv;
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kPerThread; ++k)
            if (mine[k]) x[threadIdx.x + 1024 * k] = t[k];
        __syncthreads();
    }
}

__device__ __forceinline__ float warp_sumf(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}
__device__ float sm_block_sumf(float v, float *red) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    v = warp_sumf(v);
    if (lane == 0) red[wid] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.0f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
        red[32] = s;
    }
    __syncthreads();
    const float out = red[32];
    __syncthreads();
    return out;
}

// Coarsest level: Jacobi-preconditioned CG in shared memory (one uniform level: symmetric),
// all in FP32 (GB300's FP64 rate is a small fraction of FP32), to 1e-3 relative residual,
// which is all a coarse-grid correction needs.  Up to 256 cells it runs on the first warp.
struct SmallWalls { int bcx, bcy; };
__device__ void sm_coarse_cg(const SmallDesc &Ds, const SmallLevel &level, float *x, const float *b, float *r, float *p,
                             float *q, bool singular, float *red) {
    const SmallWalls D{Ds.bcx, Ds.bcy};
    const SmallLevel L = level;  // in registers: the vectors' stores could alias the shared copy
    const int n = L.n;
    const int maxit = min(2 * n + 10, 500);
    const bool warp_only = n <= 256;
    if (warp_only && threadIdx.x >= 32) {
        __syncthreads();
        return;
    }
    const int stride = warp_only ? 32 : blockDim.x;
    auto sum = [&](float v) -> float { return warp_only ? warp_sumf(v) : sm_block_sumf(v, red); };
    auto sync = [&]() { if (warp_only) __syncwarp(); else __syncthreads(); };
    float mb = 0.0f;
    if (singular) {
        for (int i = threadIdx.x; i < n; i += stride) mb += b[i];
        mb = sum(mb) / (float)n;
    }
    float rz = 0.0f, bb = 0.0f;
    for (int i = threadIdx.x; i < n; i += stride) {
        float d, dinv;
        sm_row(D, L, b, i, d, dinv);  // diagonal only
        const float ri = b[i] - mb;
        x[i] = 0.0f;
        r[i] = ri;
        const float zi = ri * dinv;
        p[i] = zi;
        rz += ri * zi;
        bb += ri * ri;
    }
    rz = sum(rz);
    bb = sum(bb);
    sync();
    if (bb > 0.0f) {
        for (int it = 0; it < maxit; ++it) {
            float pq = 0.0f;
            for (int i = threadIdx.x; i < n; i += stride) {
                float d;
                const float sn = sm_row(D, L, p, i, d);
                const float ax = d * p[i] - sn;
                q[i] = ax;
                pq += p[i] * ax;
            }
            pq = sum(pq);
            if (!(pq > 0.0f)) break;
            const float alpha = rz / pq;
            float rr = 0.0f, rz2 = 0.0f;
            for (int i = threadIdx.x; i < n; i += stride) {
                float d, dinv;
                sm_row(D, L, p, i, d, dinv);
                x[i] += alpha * p[i];
                const float ri = r[i] - alpha * q[i];
                r[i] = ri;
                rr += ri * ri;
                rz2 += ri * ri * dinv;
            }
            rr = sum(rr);
            rz2 = sum(rz2);
            if (rr <= kSmCoarseTol2 * bb) break;
            const float beta = rz2 / rz;
            rz = rz2;
            sync();
            for (int i = threadIdx.x; i < n; i += stride) {
                float d, dinv;
                sm_row(D, L, p, i, d, dinv);
                p[i] = r[i] * dinv + beta * p[i];
            }
            sync();
        }
    }
    if (singular) {
        float mx = 0.0f;
        for (int i = threadIdx.x; i < n; i += stride) mx += x[i];
        mx = sum(mx) / (float)n;
        for (int i = threadIdx.x; i < n; i += stride) x[i] -= mx;
    }
    __syncthreads();
}

// Barrier `id` (1 .. 15) over the first `nthr` threads of the block.
__device__ __forceinline__ void part_bar(int id, int nthr) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthr) : "memory");
}

// Coarsest level by its dense inverse C (at most kDirectN cells, rows n | 1 words apart so that
// lanes of different rows read different banks), applied in FP64 by the first nthr >= 256
// threads, 8, 4 or 2 lanes per row (one pass over all rows).  The FP64 pipe retires two lanes
// per clock and SM and a dependent operation takes tens of clocks: a lane runs four chains and
// few lanes are combined.  Singular (periodic in both directions): C (b - mean(b) 1) with
// C 1 = 1 is (C - 1 1^T / n) b, whose matrix is formed on the host.  `scr`: n doubles.
template <int LPR, typename T>
__device__ __forceinline__ void direct_rows(int n, const T *inv, float *x, const T *bd) {
    const int t = threadIdx.x, part = t & (LPR - 1), r = t / LPR;
    T a[4] = {0, 0, 0, 0};
    if (r < n) {
        const T *row = inv + r * (n | 1);
        int c = part;
        for (; c + 3 * LPR < n; c += 4 * LPR)
#pragma unroll
            for (int k = 0; k < 4; ++k) a[k] = fma(row[c + k * LPR], bd[c + k * LPR], a[k]);
        for (; c < n; c += LPR) a[0] = fma(row[c], bd[c], a[0]);
    }
    T s = (a[0] + a[1]) + (a[2] + a[3]);
#pragma unroll
    for (int o = 1; o < LPR; o <<= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    if (part == 0 && r < n) x[r] = (float)s;
}
template <typename T> __device__ __forceinline__ void direct_solve(int n, const T *inv, float *x, const T *bd) {
    if (threadIdx.x >= 256) return;
    if (n <= 32) direct_rows<8>(n, inv, x, bd);
    else if (n <= 64) direct_rows<4>(n, inv, x, bd);
    else direct_rows<2>(n, inv, x, bd);
}
__device__ void sm_coarse_direct(const SmallLevel &L, const double *inv, float *x, const float *b, int nthr, int bar,
                                 double *scr) {
    const int n = L.n;
    if ((int)threadIdx.x < n) scr[threadIdx.x] = (double)b[threadIdx.x];
    part_bar(bar, nthr);
    direct_solve(n, inv, x, scr);
}

// The implicit scheme's coarsest operator changes every step: its inverse is formed by the
// launch that uses it (by one before the cycles of a multi-block solve), in FP32 (a coarse-grid correction needs three digits: the CG it replaces
// stopped at 1e-3), in place by Gauss-Jordan without pivoting (the operator is symmetric and
// positive definite).  Singular: A + alpha 1 1^T is inverted and the constant's image taken out
// again, so that the mean of the right-hand side does not matter.  1024 threads; `tmp` 2 n words.
__device__ __forceinline__ void form_inverse(const SmallLevel &L, float *M, bool singular, float *tmp) {
    const int n = L.n, ld = n | 1, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    float *rowk = tmp, *colk = tmp + n;
    const float alpha = singular ? __frcp_rn(L.dinv[0]) / (float)n : 0.0f;
    for (int i = ty; i < n; i += 32)
        for (int j = tx; j < n; j += 32) M[i * ld + j] = alpha;
    __syncthreads();
    if ((int)threadIdx.x < n) {  // a row's columns are distinct except across a wrap of one or two cells
        const int i = threadIdx.x;
        M[i * ld + i] += __frcp_rn(L.dinv[i]);
        for (int j = 0; j < kEll; ++j) {
            const int32_t c = L.col[(int64_t)j * n + i];
            if (c >= 0) M[i * ld + c] += L.val[(int64_t)j * n + i];
        }
    }
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        if ((int)threadIdx.x < n) {
            const float p = 1.0f / M[k * ld + k];
            rowk[threadIdx.x] = (int)threadIdx.x == k ? p : M[k * ld + threadIdx.x] * p;
            colk[threadIdx.x] = M[threadIdx.x * ld + k];
        }
        __syncthreads();
        for (int i = ty; i < n; i += 32) {
            const float f = colk[i];
            for (int j = tx; j < n; j += 32) {
                const float r = rowk[j];
                M[i * ld + j] = i == k ? r : (j == k ? -f * r : fmaf(-f, r, M[i * ld + j]));
            }
        }
        __syncthreads();
    }
    if (singular) {
        const float c = 1.0f / (alpha * (float)n * (float)n);
        for (int i = ty; i < n; i += 32)
            for (int j = tx; j < n; j += 32) M[i * ld + j] -= c;
        __syncthreads();
    }
}

// (out of line in the solve kernel, whose registers it would take)
__device__ __noinline__ void sm_build_inverse(const SmallLevel &L, float *M, bool singular, float *tmp) {
    form_inverse(L, M, singular, tmp);
}

// ---- levels stored by colour --------------------------------------------------------------
// A strip is one position m of a row and the K rows (K even) from an even one on: 2 K cells, two
// in each row, held by one thread (S strips per thread).  In an even row colour 0 is at ix = 2 m
// and colour 1 at 2 m + 1, in an odd row the other way round, so a cell's horizontal neighbours
// are the strip's other cell of its row and one word of a neighbouring strip, and its vertical
// neighbours are the strip's own cells except above and below it: K + 2 shared loads per half
// sweep of K cells instead of 4 K.  A colour reads only the other colour, so values are updated
// in place and one barrier ends a half sweep.  A missing neighbour is the zero word at `half`.
//
// What bounds the solve is this serial chain of half sweeps; with four cells per thread the
// finest level's is bound by shared-memory words.  512 x 16 cells, 4 cycles: 0.283 ms when each
// cell's index division and wall tests were done in every half sweep and two barriers ended it,
// 0.118 ms with the neighbour offsets formed once per leg (4 K loads), 0.105 ms so, and 0.100 ms
// with the decision and the coarsest solve as they are now.
template <int K, int S> struct RbStrips {
    int j[S];            // position of the first row
    int l[S], sl[S];     // word left of it and the step to the next row's (0: missing)
    int r[S], sr[S];     // the same to the right
    int dn[S], up[S];    // words below the first and above the last row
    float di0[S][K], di1[S][K];  // reciprocal diagonals of the two colours
    float b0[S][K], b1[S][K];    // right-hand side
    bool ok[S];
};
template <int K, int S>
__device__ __forceinline__ void rb_strips(const SmallDesc &D, const SmallLevel &L, const float *b0, const float *b1,
                                          RbStrips<K, S> &c) {
    const int nxh = L.nx >> 1, half = L.half;
    const bool px = D.bcx == PIC_BC_PERIODIC, py = D.bcy == PIC_BC_PERIODIC;
    const float wx = D.bcx == PIC_BC_DIRICHLET ? 2.0f : (px ? 1.0f : 0.0f);
    const float wy = D.bcy == PIC_BC_DIRICHLET ? 2.0f : (py ? 1.0f : 0.0f);
#pragma unroll
    for (int i = 0; i < S; ++i) {
        const int q = (int)threadIdx.x + L.nthr * i;
        const int g = mdiv(q, L.nxh_magic), m = q - g * nxh, y0 = g * K;  // rows y0 .. y0 + K - 1
        const int j = y0 * nxh + m;
        c.ok[i] = y0 < L.ny;
        c.j[i] = j;
        const bool hl = m > 0 || px, hr = m < nxh - 1 || px;
        c.l[i] = hl ? (m > 0 ? j - 1 : j + nxh - 1) : half;
        c.r[i] = hr ? (m < nxh - 1 ? j + 1 : j - nxh + 1) : half;
        c.sl[i] = hl ? nxh : 0;
        c.sr[i] = hr ? nxh : 0;
        const bool hd = y0 > 0, hu = y0 + K < L.ny;
        c.dn[i] = hd ? j - nxh : (py ? j + (L.ny - 1) * nxh : half);
        c.up[i] = hu ? j + K * nxh : (py ? m : half);
        const float dl = m > 0 ? 1.0f : wx, dr = m < nxh - 1 ? 1.0f : wx;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float dv = (1.0f + (k > 0 || hd ? 1.0f : wy)) + (k < K - 1 || hu ? 1.0f : wy);
            c.di0[i][k] = diag_inv(dv + (k & 1 ? dr : dl));
            c.di1[i][k] = diag_inv(dv + (k & 1 ? dl : dr));
            c.b0[i][k] = c.ok[i] ? b0[j + k * nxh] : 0.0f;
            c.b1[i][k] = c.ok[i] ? b1[j + k * nxh] : 0.0f;
        }
    }
}
// One half sweep of colour C: xs its values, xo the other colour's in shared memory; v and o the
// strips' own values of both.
template <int K, int S, int C>
__device__ __forceinline__ void rb_half(const RbStrips<K, S> &c, float *xs, const float *xo, float (&v)[S][K],
                                        const float (&o)[S][K], int nxh) {
#pragma unroll
    for (int i = 0; i < S; ++i) {
        if (!c.ok[i]) continue;
        const float below = xo[c.dn[i]], above = xo[c.up[i]];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float h = (k & 1) == C ? xo[c.l[i] + k * c.sl[i]] : xo[c.r[i] + k * c.sr[i]];
            const float s = ((h + o[i][k]) + (k > 0 ? o[i][k > 0 ? k - 1 : 0] : below)) +
                            (k < K - 1 ? o[i][k < K - 1 ? k + 1 : k] : above);
            v[i][k] = ((C ? c.b1[i][k] : c.b0[i][k]) + s) * (C ? c.di1[i][k] : c.di0[i][k]);
        }
#pragma unroll
        for (int k = 0; k < K; ++k) xs[c.j[i] + k * nxh] = v[i][k];
    }
}

// Pre-smoothing from x = 0 and the residual's restriction.
template <int K, int S>
__device__ __forceinline__ void rb_down(const SmallDesc &D, const SmallLevel &L, const SmallLevel &Cc, float *sm, int bar) {
    const int nthr = L.nthr, nxh = L.nx >> 1;
    float *x0 = sm + L.off, *x1 = x0 + L.hs;
    RbStrips<K, S> c;
    float a[S][K], e[S][K];  // the strips' values of colour 0 and 1
    rb_strips<K, S>(D, L, x0 + L.boff, x1 + L.boff, c);
#pragma unroll
    for (int i = 0; i < S; ++i)
#pragma unroll
        for (int k = 0; k < K; ++k) {
            a[i][k] = c.b0[i][k] * c.di0[i][k];  // the first half sweep reads zeros only
            if (c.ok[i]) x0[c.j[i] + k * nxh] = a[i][k];
        }
    if (threadIdx.x == 0) x0[L.half] = x1[L.half] = 0.0f;  // missing neighbours
    part_bar(bar, nthr);
    rb_half<K, S, 1>(c, x1, x0, e, a, nxh);
    part_bar(bar, nthr);
#pragma unroll
    for (int s = 1; s < kNu; ++s) {
        rb_half<K, S, 0>(c, x0, x1, a, e, nxh);
        part_bar(bar, nthr);
        rb_half<K, S, 1>(c, x1, x0, e, a, nxh);
        part_bar(bar, nthr);
    }
    // coarse cells: the residuals of the children (0,0), (1,0), (0,1), (1,1) summed in this order
    float *bc = sm + Cc.off + Cc.boff;
#pragma unroll
    for (int i = 0; i < S; ++i) {
        if (!c.ok[i]) continue;
        const int q = (int)threadIdx.x + nthr * i;
        const int g = mdiv(q, L.nxh_magic), m = q - g * nxh;
        const float b0d = x0[c.dn[i]], b1d = x1[c.dn[i]], a0u = x0[c.up[i]], a1u = x1[c.up[i]];
        // half diagonals of the left, right, lower and upper cells of a quartet
        const float wx = D.bcx == PIC_BC_DIRICHLET ? 2.0f : (D.bcx == PIC_BC_PERIODIC ? 1.0f : 0.0f);
        const float wy = D.bcy == PIC_BC_DIRICHLET ? 2.0f : (D.bcy == PIC_BC_PERIODIC ? 1.0f : 0.0f);
        const float gl = 1.0f + (m > 0 ? 1.0f : wx), gr = 1.0f + (m < nxh - 1 ? 1.0f : wx);
#pragma unroll
        for (int k = 0; k < K; k += 2) {
            const float l0 = x1[c.l[i] + k * c.sl[i]], l1 = x0[c.l[i] + (k + 1) * c.sl[i]];
            const float r0 = x0[c.r[i] + k * c.sr[i]], r1 = x1[c.r[i] + (k + 1) * c.sr[i]];
            const float x00 = a[i][k], x10 = e[i][k], x01 = e[i][k + 1], x11 = a[i][k + 1];
            const float d1 = k > 0 ? e[i][k > 0 ? k - 1 : 0] : b1d, d0 = k > 0 ? a[i][k > 0 ? k - 1 : 0] : b0d;
            const float u0 = k + 2 < K ? a[i][k + 2 < K ? k + 2 : k] : a0u, u1 = k + 2 < K ? e[i][k + 2 < K ? k + 2 : k] : a1u;
            const float gd = 1.0f + (k > 0 || g > 0 ? 1.0f : wy), gu = 1.0f + (k + 2 < K || (g + 1) * K < L.ny ? 1.0f : wy);
            float s = c.b0[i][k] - ((gl + gd) * x00 - (((l0 + x10) + d1) + x01));
            s += c.b1[i][k] - ((gr + gd) * x10 - (((x00 + r0) + d0) + x11));
            s += c.b1[i][k + 1] - ((gl + gu) * x01 - (((l1 + x11) + x00) + u0));
            s += c.b0[i][k + 1] - ((gr + gu) * x11 - (((x01 + r1) + x10) + u1));
            const int cy = (K / 2) * g + k / 2;
            bc[Cc.fast ? ((m + cy) & 1) * Cc.hs + cy * (nxh >> 1) + (m >> 1) : cy * nxh + m] = s;
        }
    }
    part_bar(bar, nthr);
}

// The coarse correction (needed on colour 1 only: the first half sweep overwrites colour 0
// without reading it) and the post-smoothing.
template <int K, int S>
__device__ __forceinline__ void rb_up(const SmallDesc &D, const SmallLevel &L, const SmallLevel &Cc, float *sm, int bar) {
    const int nthr = L.nthr, nxh = L.nx >> 1;
    float *x0 = sm + L.off, *x1 = x0 + L.hs;
    const float *xc = sm + Cc.off;
    RbStrips<K, S> c;
    float a[S][K], e[S][K];
    rb_strips<K, S>(D, L, x0 + L.boff, x1 + L.boff, c);
    part_bar(bar, nthr);  // the coarser level's correction is complete
#pragma unroll
    for (int i = 0; i < S; ++i) {
        const int q = (int)threadIdx.x + nthr * i;
        const int g = mdiv(q, L.nxh_magic), m = q - g * nxh;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            e[i][k] = 0.0f;
            if (c.ok[i]) {
                const int cy = (K / 2) * g + k / 2;
                e[i][k] = x1[c.j[i] + k * nxh] +
                          xc[Cc.fast ? ((m + cy) & 1) * Cc.hs + cy * (nxh >> 1) + (m >> 1) : cy * nxh + m];
                x1[c.j[i] + k * nxh] = e[i][k];
            }
        }
    }
    part_bar(bar, nthr);
#pragma unroll
    for (int s = 0; s < kNu; ++s) {
        rb_half<K, S, 0>(c, x0, x1, a, e, nxh);
        part_bar(bar, nthr);
        rb_half<K, S, 1>(c, x1, x0, e, a, nxh);
        if (s + 1 < kNu) part_bar(bar, nthr);
    }
}

// The same legs on a uniform level whose faces carry the implicit scheme's kappa (face words,
// reciprocal diagonals from global memory: they stay in L1 over a launch).  Position j of colour
// c is the cell ix = 2 m + p of row iy, p = (c + iy) & 1.
struct KapCell { int i, iy, m, p; };
__device__ __forceinline__ KapCell kap_cell(const SmallLevel &L, int j, int c) {
    KapCell k;
    const int nxh = L.nx >> 1;
    k.iy = mdiv(j, L.nxh_magic);
    k.m = j - k.iy * nxh;
    k.p = (c + k.iy) & 1;
    k.i = k.iy * L.nx + 2 * k.m + k.p;
    return k;
}
// sum over the cell's faces of conductance times neighbour (left, right, below, above); xo: the
// other colour's values
__device__ __forceinline__ float kap_row(const SmallDesc &D, const SmallLevel &L, const float *xo, int j, const KapCell &k) {
    const int nx = L.nx, nxh = nx >> 1, half = L.half, i = k.i;
    const bool px = D.bcx == PIC_BC_PERIODIC, py = D.bcy == PIC_BC_PERIODIC;
    const float *fx = L.face, *fy = L.face + L.n;
    const bool l_in = k.p || k.m > 0, d_in = k.iy > 0, u_in = k.iy < L.ny - 1;
    const int jl = k.p ? j : (k.m > 0 ? j - 1 : (px ? j + nxh - 1 : half));
    const int jr = !k.p ? j : (k.m < nxh - 1 ? j + 1 : (px ? j - nxh + 1 : half));
    const int jd = d_in ? j - nxh : (py ? j + (L.ny - 1) * nxh : half);
    const int ju = u_in ? j + nxh : (py ? j - (L.ny - 1) * nxh : half);
    const float gl = __ldg(fx + (l_in ? i - 1 : (px ? i + nx - 1 : i))), gr = __ldg(fx + i);
    const float gd = __ldg(fy + (d_in ? i - nx : (py ? i + (L.ny - 1) * nx : i))), gu = __ldg(fy + i);
    return fmaf(gu, xo[ju], fmaf(gd, xo[jd], fmaf(gr, xo[jr], gl * xo[jl])));
}
__device__ __forceinline__ void kap_half(const SmallDesc &D, const SmallLevel &L, int c, float *x0, const float *b0) {
    float *xs = x0 + c * L.hs;
    const float *xo = x0 + (c ^ 1) * L.hs, *b = b0 + c * L.hs;
#pragma unroll 2
    for (int j = threadIdx.x; j < L.half; j += L.nthr) {
        const KapCell k = kap_cell(L, j, c);
        xs[j] = (b[j] + kap_row(D, L, xo, j, k)) * __ldg(L.dinv + k.i);
    }
}
__device__ __noinline__ void kap_down(const SmallDesc &D, const SmallLevel &L, const SmallLevel &Cc, float *sm, int bar) {
    float *x0 = sm + L.off, *x1 = x0 + L.hs;
    const float *b0 = x0 + L.boff, *b1 = b0 + L.hs;
    for (int j = threadIdx.x; j < L.half; j += L.nthr) x0[j] = b0[j] * __ldg(L.dinv + kap_cell(L, j, 0).i);
    if (threadIdx.x == 0) x0[L.half] = x1[L.half] = 0.0f;  // missing neighbours
    part_bar(bar, L.nthr);
    for (int h = 1; h < 2 * kNu; ++h) {
        kap_half(D, L, h & 1, x0, b0);
        part_bar(bar, L.nthr);
    }
    float *bc = sm + Cc.off + Cc.boff;
    const int nxh = L.nx >> 1;
    for (int p = threadIdx.x; p < Cc.n; p += L.nthr) {
        const int qy = mdiv(p, L.nxh_magic), qx = p - qy * nxh;
        float s = 0.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int iy = 2 * qy + (k >> 1), c = ((k & 1) + iy) & 1, j = iy * nxh + qx;
            const KapCell kc{iy * L.nx + 2 * qx + (k & 1), iy, qx, k & 1};
            const float *xo = c ? x0 : x1, *xs = c ? x1 : x0, *b = c ? b1 : b0;
            const float d = __frcp_rn(__ldg(L.dinv + kc.i));
            s += b[j] - (d * xs[j] - kap_row(D, L, xo, j, kc));
        }
        bc[sm_pos(Cc, p)] = s;
    }
    part_bar(bar, L.nthr);
}
__device__ __noinline__ void kap_up(const SmallDesc &D, const SmallLevel &L, const SmallLevel &Cc, float *sm, int bar) {
    float *x0 = sm + L.off, *x1 = x0 + L.hs;
    const float *b0 = x0 + L.boff, *xc = sm + Cc.off;
    const int nxh = L.nx >> 1;
    part_bar(bar, L.nthr);  // the coarser level's correction is complete
    for (int j = threadIdx.x; j < L.half; j += L.nthr) {
        const int iy = mdiv(j, L.nxh_magic), m = j - iy * nxh;
        x1[j] += xc[sm_pos(Cc, (iy >> 1) * nxh + m)];
    }
    part_bar(bar, L.nthr);
    for (int h = 0; h < 2 * kNu; ++h) {
        kap_half(D, L, h & 1, x0, b0);
        if (h + 1 < 2 * kNu) part_bar(bar, L.nthr);
    }
}

// V-cycle over the shared-memory levels; b of the first level must be in place, x of the
// first level holds the correction on return (after a block barrier).  All 1024 threads call
// it.  ELL levels are swept by the whole block; a level stored by colour by its nthr threads,
// whose other warps wait at the next finer level's barrier (barrier ids count from the first
// such level).  `inv` is the coarsest inverse (FP32 where the launch built it; null: CG), `scr`
// kDirectN doubles.  CG: the coarsest level is solved by the CG.
template <bool CG> __device__ void sm_vcycle(const SmallDesc &D, float *sm, bool singular, float *red, const double *inv, double *scr) {
    const int last = D.nlev - 1;
    int g = 0;
    for (; g < last && !D.lv[g].fast; ++g) {
        const SmallLevel &L = D.lv[g], &Cc = D.lv[g + 1];
        float *x = sm + L.off, *b = x + L.boff;
        for (int k = 0; k < kNu; ++k) sm_smooth(D, L, x, b, k == 0);
        float *bc = sm + Cc.off + Cc.boff;
        for (int p = threadIdx.x; p < Cc.n; p += blockDim.x) {
            float s = 0.0f;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int32_t i = Cc.child4[4 * p + k];
                if (i < 0) continue;
                float d;
                const float sn = sm_row(D, L, x, i, d);
                s += b[i] - (d * x[i] - sn);
            }
            bc[sm_pos(Cc, p)] = s;
        }
        __syncthreads();
    }
    const int gf = g;
    for (; g < last; ++g) {
        const SmallLevel &L = D.lv[g], &Cc = D.lv[g + 1];
        if ((int)threadIdx.x >= L.nthr) break;
        if (L.face) kap_down(D, L, Cc, sm, 1 + g - gf);
        else if (L.rows == 4) rb_down<4, 1>(D, L, Cc, sm, 1 + g - gf);
        else if (L.strips == 1) rb_down<2, 1>(D, L, Cc, sm, 1 + g - gf);
        else rb_down<2, 2>(D, L, Cc, sm, 1 + g - gf);
    }
    if (g == last) {
        const SmallLevel &L = D.lv[last];
        float *x = sm + L.off, *b = x + L.boff;
        float *r = sm + D.off_cg;
        if (!CG && D.build) direct_solve(L.n, reinterpret_cast<const float *>(inv), x, b);
        else if (!CG && inv) sm_coarse_direct(L, inv, x, b, last > gf ? D.lv[last - 1].nthr : 1024, 1 + last - gf, scr);
        else sm_coarse_cg(D, L, x, b, r, r + L.n, r + 2 * L.n, singular, red);
    }
    for (--g; g >= gf; --g) {
        const SmallLevel &L = D.lv[g], &Cc = D.lv[g + 1];
        if (L.face) kap_up(D, L, Cc, sm, 1 + g - gf);
        else if (L.rows == 4) rb_up<4, 1>(D, L, Cc, sm, 1 + g - gf);
        else if (L.strips == 1) rb_up<2, 1>(D, L, Cc, sm, 1 + g - gf);
        else rb_up<2, 2>(D, L, Cc, sm, 1 + g - gf);
    }
    if (gf > 0) __syncthreads();
    for (g = gf - 1; g >= 0; --g) {
        const SmallLevel &L = D.lv[g], &Cc = D.lv[g + 1];
        float *x = sm + L.off, *b = x + L.boff;
        const float *xc = sm + Cc.off;
        for (int i = threadIdx.x; i < L.n; i += blockDim.x) x[i] += xc[sm_pos(Cc, L.parent[i])];
        __syncthreads();
        for (int k = 0; k < kNu; ++k) sm_smooth(D, L, x, b, false);
    }
}

// The coarsest inverse of a multi-block solve of the implicit scheme, formed once before its cycles
// (formed in every cycle's tail, 208 x 144 cells with 117 coarsest: 1.40 ms per solve of 5 cycles; so 0.59).
__global__ void __launch_bounds__(1024, 1) k_coarse_inverse(const __grid_constant__ SmallLevel L, int singular,
                                                            float *__restrict__ out) {
    extern __shared__ __align__(16) float sm[];
    __shared__ float tmp[2 * kDirectN];
    form_inverse(L, sm, singular != 0, tmp);
    for (int k = threadIdx.x; k < L.n * (L.n | 1); k += 1024) out[k] = sm[k];
}

// Tail of a V-cycle started by the multi-block levels: b from global, x back to global.
__global__ void __launch_bounds__(1024, 1) k_tail_vcycle(const __grid_constant__ SmallDesc Dp,
                                                       const float *__restrict__ gb, float *__restrict__ gx,
                                                       int singular) {
    extern __shared__ __align__(16) float sm[];
    __shared__ float redf[33];
    __shared__ double scr[kDirectN];
    __shared__ SmallDesc D;
    // constant data before the wait for the kernel before this one
    for (int k = threadIdx.x; k < (int)(sizeof(SmallDesc) / 4); k += 1024)
        reinterpret_cast<uint32_t *>(&D)[k] = reinterpret_cast<const uint32_t *>(&Dp)[k];
    __syncthreads();
    const double *inv = D.cinv;
    double *cs = reinterpret_cast<double *>(sm + D.smem_floats);
    if (D.inv_words) {
        if (inv)
            for (int k = threadIdx.x; k < D.inv_words; k += 1024) cs[k] = inv[k];
        inv = cs;
    }
    pdl_chain();
    const SmallLevel &L = D.lv[0];
    for (int i = threadIdx.x; i < L.n; i += blockDim.x) sm[L.off + L.boff + sm_pos(L, i)] = gb[i];
    __syncthreads();
    sm_vcycle<false>(D, sm, singular != 0, redf, inv, scr);
    __syncthreads();
    for (int i = threadIdx.x; i < L.n; i += blockDim.x) gx[i] = sm[L.off + sm_pos(L, i)];
}

// FP64 sums over the cells of a small solve that come out the same whatever the number C of
// CTAs in the instance's cluster: chunk c (cells 1024 c .. 1024 c + 1023) is summed by CTA
// c mod C as a fixed tree into four words part[4 c .. 4 c + 3] of the leader's shared memory,
// and small_total adds the (at most 32) words as a fixed tree.  f(i) is cell i's term.  A
// chunk's terms go through shared memory and 128 threads add eight each before any shuffle:
// 52 FP64 warp instructions per chunk instead of the 160 of a shuffle tree in every warp (the
// FP64 pipe takes 16 clocks for each).
constexpr int kSmallChunks = kSmallN / 1024;
template <typename F>
__device__ __forceinline__ void small_sums(int C, int rank, int n, double *vbuf, int nbuf, double *part, F f) {
    const int nch = (n + 1023) >> 10;
    const int nq = rank < nch ? (nch - rank + C - 1) / C : 0;  // this CTA's chunks
    const int u = threadIdx.x & 127;
    for (int q0 = 0; q0 < nq; q0 += nbuf) {
        const int m = min(nbuf, nq - q0);
        if (q0) __syncthreads();
        for (int q = 0; q < m; ++q) {
            const int i = ((rank + (q0 + q) * C) << 10) + (int)threadIdx.x;
            vbuf[1024 * q + threadIdx.x] = i < n ? f(i) : 0.0;
        }
        __syncthreads();
        for (int q = threadIdx.x >> 7; q < m; q += 8) {
            double v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = vbuf[1024 * q + u + 128 * k];
            double s = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xFFFFFFFFu, s, o);
            if ((u & 31) == 0) part[4 * (rank + (q0 + q) * C) + (u >> 5)] = s;
        }
    }
}
// The total of a sum's words, on every lane of the calling warp of the leader CTA.
__device__ __forceinline__ double small_total(const double *part, int n) {
    const int lane = threadIdx.x & 31;
    double s = lane < 4 * ((n + 1023) >> 10) ? part[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    return s;
}

// Whole solve for a mesh whose every level fits: FP64 residual and correction, FP32 V-cycles
// in shared memory, convergence test on the device.  One cluster of C CTAs per item: the leader
// CTA holds the levels and runs the V-cycles, and the FP64 work (warm start, residual,
// correction, norms) is split by chunks of 1024 cells over the cluster, each CTA writing its
// chunks' FP32 residual straight into the leader's shared memory.  GB300's FP64 rate per SM
// is low (two lanes a clock), so a cycle's FP64 work (7 operations per cell and the norm) is
// spread over the cluster's SMs.  A cycle crosses three cluster barriers: residual and norm
// words with the leader; correction (or the decision to stop) with the others; potential
// complete.  The result does not depend on C.  stats: [cycles, rel. residual, max rel. since
// reset].
struct SmallSolve {
    SmallDesc D;
    const double *diag64, *val64;
    double *phi, *phi_prev, *bvec, *stats;
    const uint8_t *lev;
    int32_t *n_solves;  // device counter: the warm start extrapolates once two solves exist
    int lmax, singular, maxc;
    double tol;
};

// `nbuf`: chunk buffers of the sums that fit behind every item's levels.  CG: a mesh solved alone
// whose coarsest level goes to the CG, without the code of the direct solves (their registers cost
// the CG's loops 2 %).
template <bool CG>
__global__ void __launch_bounds__(1024, 1) k_small_solve(const SmallSolve *__restrict__ items, int nbuf) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    extern __shared__ __align__(16) float sm[];
    __shared__ float redf[33];
    __shared__ SmallDesc D;
    __shared__ double part[64], mean_sh;
    __shared__ int stop_sh;
    const SmallSolve &it = items[blockIdx.x / C];
    for (int k = threadIdx.x; k < (int)(sizeof(SmallDesc) / 4); k += 1024)
        reinterpret_cast<uint32_t *>(&D)[k] = reinterpret_cast<const uint32_t *>(&it.D)[k];
    __syncthreads();
    double *vbuf = reinterpret_cast<double *>(sm + D.smem_floats);
    const double *inv = D.cinv;
    if (rank == 0 && D.inv_words) {
        double *cs = vbuf + 1024 * nbuf;
        if (inv)
            for (int k = threadIdx.x; k < D.inv_words; k += 1024) cs[k] = inv[k];
        inv = cs;
    }
    pdl_chain();  // what came before it reads is constant between mesh changes
    if (!CG && rank == 0 && D.build == 1)
        sm_build_inverse(D.lv[D.nlev - 1], reinterpret_cast<float *>(vbuf + 1024 * nbuf), it.singular != 0,
                         reinterpret_cast<float *>(vbuf));
    float *lsm = cl.map_shared_rank(sm, 0);  // the leader's levels
    double *lpart = cl.map_shared_rank(part, 0);
    const double *lmean = cl.map_shared_rank(&mean_sh, 0);
    const int *lstop = cl.map_shared_rank(&stop_sh, 0);
    const double *__restrict__ diag64 = it.diag64;
    const double *__restrict__ val64 = it.val64;
    double *phi = it.phi;
    double *bvec = it.bvec;
    const uint8_t *__restrict__ lev = it.lev;
    const int lmax = it.lmax, singular = it.singular, maxc = it.maxc;
    const double tol2 = it.tol * it.tol;
    double bb = 0.0;  // ||b||^2 (the leader's first warp)
    const SmallLevel &L = D.lv[0];
    const int n = L.n, nch = (n + 1023) >> 10;
#define CL_FOR(i)                                                                    \
    for (int c_ = rank; c_ < nch; c_ += C)                                           \
        for (int i = (c_ << 10) + (int)threadIdx.x; i < n && i < ((c_ + 1) << 10); i += 1 << 30)
    // the area-weighted mean of f over all cells (areas in units of the finest cell's), known to
    // every thread of the cluster (the division is done once: in FP64 it is ~25 operations)
    auto area = [&](int i) { const double s = (double)(1 << (lmax - lev[i])); return s * s; };
    auto mean = [&](auto f) -> double {
        small_sums(C, rank, n, vbuf, nbuf, lpart, f);
        if (!L.uniform) {
            __syncthreads();
            small_sums(C, rank, n, vbuf, nbuf, lpart + 32, area);
        }
        cl.sync();
        if (rank == 0 && threadIdx.x < 32) {
            const double a = small_total(part, n), b = L.uniform ? (double)n : small_total(part + 32, n);
            if (threadIdx.x == 0) mean_sh = a / b;
        }
        cl.sync();
        return *lmean;
    };
    const int ns = *it.n_solves;
    if (ns >= 1)
        CL_FOR(i) {
            const double p = phi[i];
            if (ns >= 2) phi[i] = 2.0 * p - it.phi_prev[i];
            it.phi_prev[i] = p;
        }
    if (singular) {  // right-hand side compatibility: remove an area-proportional share
        const double k = mean([&](int i) { return bvec[i]; });
        CL_FOR(i) bvec[i] -= L.uniform ? k : k * area(i);
    }
    small_sums(C, rank, n, vbuf, nbuf, lpart + 32, [&](int i) { return bvec[i] * bvec[i]; });
    cl.sync();  // every CTA has read the counter; phi is complete
    if (rank == 0 && threadIdx.x == 0) *it.n_solves = ns + 1;
    float *lb = lsm + L.off + L.boff, *lx = lsm + L.off;
    for (int cyc = 0;; ++cyc) {
        small_sums(C, rank, n, vbuf, nbuf, lpart, [&](int i) {
            double ax;
            if (L.uniform) {
                int dd;
                const double sn = uni_row<double>(L.nx, L.ny, L.nx_magic, D.bcx, D.bcy, phi, i, dd);
                ax = (dd == 4 ? 4.0 : (double)dd) * phi[i] - sn;
            } else {
                ax = diag64[i] * phi[i];
#pragma unroll
                for (int j = 0; j < kEll; ++j) {
                    const int32_t c = L.col[(int64_t)j * n + i];
                    if (c >= 0) ax += val64[(int64_t)j * n + i] * phi[c];
                }
            }
            const double ri = bvec[i] - ax;
            lb[sm_pos(L, i)] = (float)ri;
            return ri * ri;
        });
        cl.sync();
        if (rank == 0) {
            if (threadIdx.x < 32) {
                // ||r|| <= tol ||b||, compared squared: the root and the division only once done
                const double rr = small_total(part, n);
                if (cyc == 0) bb = small_total(part + 32, n);
                if (threadIdx.x == 0) {
                    const bool stop = rr <= tol2 * (bb > 0.0 ? bb : 1.0) || cyc >= maxc;
                    stop_sh = stop;
                    if (stop) {
                        const double rel = bb > 0.0 ? sqrt(rr / bb) : sqrt(rr);
                        it.stats[0] = (double)cyc;
                        it.stats[1] = rel;
                        it.stats[2] = worst_residual(it.stats[2], rel);
                    }
                }
            }
            __syncthreads();
            if (!stop_sh) sm_vcycle<CG>(D, sm, singular != 0, redf, inv, vbuf);
        }
        cl.sync();  // the correction is in the leader's x
        if (*lstop) break;
        CL_FOR(i) phi[i] += (double)lx[sm_pos(L, i)];
        cl.sync();  // phi complete before the next residual (and x read before the next V-cycle)
    }
    if (singular) {  // zero area-weighted mean (a constant changes no residual)
        const double k = mean([&](int i) { return L.uniform ? phi[i] : area(i) * phi[i]; });
        CL_FOR(i) phi[i] -= k;
    }
#undef CL_FOR
    cl.sync();  // the leader's shared memory outlives every read of it
}

// A solve's shared memory holds the levels and the coarsest inverse (lv_bytes) and, per chunk of
// a CTA, one 8 KB buffer of the sums (as many as fit, at least one).
int small_bufs(int n, int C, size_t lv_bytes) {
    const int nch = (n + 1023) / 1024;
    return std::max(1, std::min((nch + C - 1) / C, ((int)kSmallSmemMax - (int)lv_bytes) / 8192));
}

cudaLaunchConfig_t small_config(int n_items, int C, size_t smem, cudaLaunchAttribute *attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n_items * C));
    cfg.blockDim = dim3(1024);
    cfg.dynamicSmemBytes = smem;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// One launch of the small solve: n_items clusters of C CTAs.
void launch_small_solve(const void *items, int n_items, int C, int nbuf, size_t smem, bool cg, cudaStream_t st) {
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = small_config(n_items, C, smem, attr);
    cfg.stream = st;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
    GB_CUDA(cudaLaunchKernelEx(&cfg, cg ? k_small_solve<true> : k_small_solve<false>, (const SmallSolve *)items, nbuf));
}

// The cluster size for n_items instances solved in one launch: one CTA per 1024-cell chunk of
// the largest, at most 8, as many as the GPU's SMs hold side by side (a CTA fills an SM),
// reduced until the GPU can hold such clusters.  32 instances of up to 8192 cells: 0.61 ms with
// one CTA each and the old sweeps, 0.133 ms with 4.
int small_cluster(int n, int n_items, size_t lv_bytes) {
    int sms = 0, dev = 0;
    GB_CUDA(cudaGetDevice(&dev));
    GB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    int C = 1;
    while (2 * C <= std::min(8, (n + 1023) / 1024) && 2 * C * n_items <= sms) C *= 2;
    for (; C > 1; C >>= 1) {
        cudaLaunchAttribute attr[1];
        cudaLaunchConfig_t cfg = small_config(n_items, C, lv_bytes + (size_t)small_bufs(n, C, lv_bytes) * 8192, attr);
        int nc = 0;
        if (cudaOccupancyMaxActiveClusters(&nc, k_small_solve<false>, &cfg) == cudaSuccess && nc >= n_items) break;
        cudaGetLastError();
    }
    return C;
}

// Which suffix of the level list fits one block's shared memory.
int small_from(const Instance &in) {
    int g0 = (int)in.lv.size();
    int64_t floats = 0;
    for (int g = (int)in.lv.size() - 1; g >= 0; --g) {
        const Level &L = in.lv[g];
        const int64_t add = 2 * L.n + 16 + (g == (int)in.lv.size() - 1 ? 3 * L.n + 8 : 0);
        if (L.n > kSmallN || (int)in.lv.size() - g > kMaxSmallLevels || (floats + add) * 4 > kSmallSmemCap) break;
        floats += add;
        g0 = g;
    }
    return g0;
}

SmallDesc small_desc(const Instance &in, int g0) {
    SmallDesc D{};
    D.nlev = (int)in.lv.size() - g0;
    D.bcx = in.cfg.bc_x;
    D.bcy = in.cfg.bc_y;
    int32_t off = 0;
    const int64_t nl = in.lv.back().n, words = nl * (nl | 1);
    int64_t floats = 3 * nl + 16;
    for (size_t g = g0; g < in.lv.size(); ++g) floats += 2 * in.lv[g].n + 16;
    const bool fits = floats * 4 + words * (in.cfg.implicit ? 4 : 8) + 8192 + 16 <= kSmallSmemMax;
    // (an inverse needs a Dirichlet wall, or the periodic case's constant mode taken out; between
    // Neumann walls alone the operator is singular and the CG solves what the charge allows)
    const bool wall = in.cfg.bc_x == PIC_BC_DIRICHLET || in.cfg.bc_y == PIC_BC_DIRICHLET;
    const bool periodic = in.cfg.bc_x == PIC_BC_PERIODIC && in.cfg.bc_y == PIC_BC_PERIODIC;
    D.build = in.cfg.implicit && nl <= kDirectN && fits && (wall || periodic) ? (in.coarse_build ? 2 : 1) : 0;
    for (int k = 0; k < D.nlev; ++k) {
        const Level &L = in.lv[g0 + k];
        SmallLevel &S = D.lv[k];
        S.n = (int32_t)L.n; S.col = L.col; S.val = L.val; S.dinv = L.dinv; S.color = L.color;
        S.child4 = L.child4; S.parent = L.parent; S.off = off;
        // (the implicit scheme's levels carry kappa in their ELL rows: no matrix-free stencil)
        S.uniform = L.lmax == 0 && !in.cfg.implicit ? 1 : 0;
        S.nx = L.nx0;
        S.ny = L.ny0;
        // multiply-high reciprocal: floor(i * m / 2^32) == floor(i / nx) for the i < n used here
        S.nx_magic = mdiv_magic((uint32_t)L.nx0);
        const uint32_t nxh = std::max(1, L.nx0 / 2);
        S.nxh_magic = mdiv_magic(nxh);
        auto q = [](int64_t i, uint32_t m) { return m ? (int64_t)(((uint64_t)i * m) >> 32) : i; };
        for (int64_t i = 0; i < L.n; ++i)
            if (q(i, S.nx_magic) != i / L.nx0 || q(i, S.nxh_magic) != i / (int64_t)nxh)
                fail(PIC_EINVAL, "index division check failed");
        S.fast = L.lmax == 0 && k + 1 < D.nlev ? 1 : 0;  // (such a level coarsens: nx and ny are even)
        S.face = L.face;
        S.half = (int32_t)L.n / 2;
        S.hs = S.half + 4;
        S.boff = S.fast ? 2 * S.hs : (int32_t)L.n;
        // strips of 4 rows where 2-row strips would need more than 512 threads (fewer shared
        // loads per cell, fewer warps at the barriers), of 2 rows on smaller levels (shorter
        // chains).  At least 8 warps take part (the coarsest solve runs on the last level's), every
        // warp when the coarsest level is solved by CG, which uses the whole block.
        S.rows = S.ny % 4 == 0 && S.half > 1024 ? 4 : 2;
        const int ns = S.half / S.rows;
        S.strips = ns > 1024 ? 2 : 1;
        S.nthr = in.coarse_inv || D.build ? std::min(1024, std::max(256, (ns + 31) / 32 * 32)) : 1024;
        off += S.fast ? 4 * S.hs : 2 * (int32_t)L.n;
    }
    D.off_cg = off;
    off += 3 * (int32_t)in.lv.back().n + 8;
    D.smem_floats = (off + 3) & ~3;
    D.cinv = D.build == 2 ? in.coarse_build : in.coarse_inv;
    D.inv_words = fits && (D.build || D.cinv) ? (int32_t)(D.build ? (words + 1) / 2 : words) : 0;
    return D;
}

template <bool CODED> void level_cycle(pic_ctx *ctx, Instance &in, size_t g, bool singular);

void vcycle(pic_ctx *ctx, Instance &in, size_t g, bool singular) {
    Level &L = in.lv[g];
    cudaStream_t s = ctx->stream;
    const int g0 = small_from(in);
    if ((int)g >= g0) {
        const SmallDesc D = small_desc(in, (int)g);
        const size_t bytes = (size_t)D.smem_floats * 4 + (size_t)D.inv_words * 8;
        pdl(k_tail_vcycle, 1, 1024, bytes, s, D, L.b, L.x, singular);
        count_launch(ctx);
        return;
    }
    if (g + 1 == in.lv.size()) {
        const int maxit = (int)std::min<int64_t>(2 * L.n + 10, 500);
        // r, p, q: three slices of the coarsest level's work buffer (allocated 3n)
        double *phi = g == 0 ? in.phi : nullptr;
        pdl(k_coarse_cg, 1, 1024, 0, s, L.n, L.col, L.val, L.dinv, L.b, L.x, L.t, L.t + L.n, L.t + 2 * L.n, singular,
            maxit, phi);
        count_launch(ctx);
        return;
    }
    if (in.cfg.implicit) level_cycle<false>(ctx, in, g, singular);
    else level_cycle<true>(ctx, in, g, singular);
}

// The sweeps of level g around the coarser levels' cycle.
template <bool CODED> void level_cycle(pic_ctx *ctx, Instance &in, size_t g, bool singular) {
    Level &L = in.lv[g], &C = in.lv[g + 1];
    cudaStream_t s = ctx->stream;
    const LevelOp A{L.n, L.col, L.code, L.val, L.dinv, L.color};
    const unsigned nb = blocks_for(L.n);
    double *none = nullptr;
    if (CODED && L.lmax == 0) {  // a uniform level that coarsens
        const UniLevel U{L.nx0, L.ny0, in.cfg.bc_x, in.cfg.bc_y};
        const unsigned tiles = (unsigned)(((L.nx0 + kUX - 1) / kUX) * ((L.ny0 + kUY - 1) / kUY));
        pdl(k_uni_down, tiles, kT, 0, s, U, L.b, L.x, C.b);
        count_launch(ctx);
        vcycle(ctx, in, g + 1, singular);
        pdl(k_uni_up, tiles, kT, 0, s, U, L.b, L.x, C.x, L.t, g == 0 ? in.phi : none);
        std::swap(L.x, L.t);
        count_launch(ctx);
        return;
    }
    // pre-smoothing (x starts at zero): the first sweep's two half sweeps in one kernel
    pdl(k_rbgs_first<CODED>, nb, kT, 0, s, A, L.b, L.x);
    for (int k = 1; k < kNu; ++k)
        for (int c = 0; c < 2; ++c) {
            pdl(k_rbgs_half<CODED>, nb, kT, 0, s, A, c, L.b, L.x, L.t, none);
            std::swap(L.x, L.t);
        }
    pdl(k_restrict_residual<CODED>, blocks_for(4 * C.n), kT, 0, s, C.n, C.child4, A, L.b, L.x, C.b);
    count_launch(ctx, 2 * kNu);
    vcycle(ctx, in, g + 1, singular);
    // post-smoothing, the injection of the correction fused into its first half sweep; the last
    // one of the finest level adds its result to the potential
    pdl(k_rbgs_half_prolong<CODED>, nb, kT, 0, s, A, L.b, L.x, L.parent, C.x, L.t);
    std::swap(L.x, L.t);
    for (int h = 1; h < 2 * kNu; ++h) {
        pdl(k_rbgs_half<CODED>, nb, kT, 0, s, A, h & 1, L.b, L.x, L.t, g == 0 && h == 2 * kNu - 1 ? in.phi : none);
        std::swap(L.x, L.t);
    }
    count_launch(ctx, 2 * kNu);
}
}  // namespace

namespace {
// Dense inverse of the coarsest level's operator (a uniform grid of root boxes: the 5-point
// stencil with the wall rules), plus 1 1^T / n when the mesh is periodic in both directions.
// Gauss-Jordan with partial pivoting in FP64, made symmetric; null (the CG is used) for a level
// larger than kDirectN cells or a singular matrix.  It depends on the root grid and the walls
// only, so an adaptation keeps it.
double *coarse_inverse(pic_ctx *ctx, Instance &in, bool singular) {
    const Level &L = in.lv.back();
    const int n = (int)L.n;
    if (n > kDirectN || n < 1) return nullptr;
    const std::array<int, 4> key = {L.nx0, L.ny0, in.cfg.bc_x, in.cfg.bc_y};
    if (in.coarse_inv_key == key) return in.coarse_inv_mem;
    std::vector<double> A((size_t)n * n, 0.0);
    auto at = [&](int i, int j) -> double & { return A[(size_t)i * n + j]; };
    const int nx = L.nx0, ny = L.ny0, bx = in.cfg.bc_x, by = in.cfg.bc_y;
    for (int i = 0; i < n; ++i) {
        const int ix = i % nx, iy = i / nx;
        auto face = [&](bool inside, int j, int bc) {
            if (inside || bc == PIC_BC_PERIODIC) { at(i, j) -= 1.0; at(i, i) += 1.0; }
            else if (bc == PIC_BC_DIRICHLET) at(i, i) += 2.0;
        };
        face(ix > 0, ix > 0 ? i - 1 : i + nx - 1, bx);
        face(ix < nx - 1, ix < nx - 1 ? i + 1 : i - nx + 1, bx);
        face(iy > 0, iy > 0 ? i - nx : i + (ny - 1) * nx, by);
        face(iy < ny - 1, iy < ny - 1 ? i + nx : i - (ny - 1) * nx, by);
    }
    if (singular)
        for (double &a : A) a += 1.0 / n;
    // Gauss-Jordan on [A | I]
    std::vector<double> Inv((size_t)n * n, 0.0);
    for (int i = 0; i < n; ++i) Inv[(size_t)i * n + i] = 1.0;
    double amax = 0.0;
    for (double a : A) amax = std::max(amax, std::fabs(a));
    // (left of the pivot A is the identity already, and right of it the inverse's rows are zero
    // until rows are exchanged: setting a mesh of 11 x 11 cells 0.95 -> 0.64 ms)
    int used = 0;  // the inverse's columns from `used` on are zero in the rows that eliminate
    for (int k = 0; k < n; ++k) {
        int piv = k;
        for (int i = k + 1; i < n; ++i)
            if (std::fabs(at(i, k)) > std::fabs(at(piv, k))) piv = i;
        if (!(std::fabs(at(piv, k)) > 1e-12 * amax)) return nullptr;
        used = piv != k ? n : std::max(used, k + 1);
        double *ak = A.data() + (size_t)k * n, *ik = Inv.data() + (size_t)k * n;
        if (piv != k) {
            std::swap_ranges(ak, ak + n, A.data() + (size_t)piv * n);
            std::swap_ranges(ik, ik + n, Inv.data() + (size_t)piv * n);
        }
        const double p = 1.0 / ak[k];
        for (int j = k; j < n; ++j) ak[j] *= p;
        for (int j = 0; j < used; ++j) ik[j] *= p;
        for (int i = 0; i < n; ++i) {
            double *ai = A.data() + (size_t)i * n, *ii = Inv.data() + (size_t)i * n;
            const double f = ai[k];
            if (i == k || f == 0.0) continue;
            for (int j = k; j < n; ++j) ai[j] -= f * ak[j];
            for (int j = 0; j < used; ++j) ii[j] -= f * ik[j];
        }
    }
    for (int i = 0; i < n; ++i)
        for (int j = 0; j < i; ++j) {
            const double m = 0.5 * (Inv[(size_t)i * n + j] + Inv[(size_t)j * n + i]);
            Inv[(size_t)i * n + j] = Inv[(size_t)j * n + i] = m;
        }
    if (singular)  // the mean of the right-hand side taken out (sm_coarse_direct)
        for (double &v : Inv) v -= 1.0 / n;
    std::vector<double> rows((size_t)n * (n | 1), 0.0);
    for (int i = 0; i < n; ++i) std::copy_n(Inv.data() + (size_t)i * n, n, rows.data() + (size_t)i * (n | 1));
    if (!in.coarse_inv_mem) in.coarse_inv_mem = dalloc<double>(in.inv_mem, kDirectN * (kDirectN | 1));
    GB_CUDA(cudaMemcpyAsync(in.coarse_inv_mem, rows.data(), rows.size() * 8, cudaMemcpyHostToDevice, ctx->stream));
    GB_CUDA(cudaStreamSynchronize(ctx->stream));
    in.coarse_inv_key = key;
    return in.coarse_inv_mem;
}
}  // namespace

void poisson_setup(pic_ctx *ctx, Instance &in) {
    if (in.mg_cycle) {
        cudaGraphExecDestroy(in.mg_cycle);
        in.mg_cycle = nullptr;
    }
    // (the tail has no sums' buffers, and more static shared memory)
    GB_CUDA(cudaFuncSetAttribute(k_tail_vcycle, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmallSmemMax - 8192));
    GB_CUDA(cudaFuncSetAttribute(k_small_solve<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmallSmemMax));
    GB_CUDA(cudaFuncSetAttribute(k_small_solve<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmallSmemMax));
    GB_CUDA(cudaFuncSetAttribute(k_coarse_inverse, cudaFuncAttributeMaxDynamicSharedMemorySize, kDirectN * (kDirectN | 1) * 4));
    DeviceArena &A = in.mesh_mem;
    const int64_t n = in.lv[0].n;
    in.phi = dalloc<double>(A, n);
    in.phi_prev = dalloc<double>(A, n);
    in.n_solves = 0;
    in.d_n_solves = nullptr;
    in.bvec = dalloc<double>(A, n);
    in.charge = dalloc<double>(A, n);
    in.red = dalloc<double>(A, 2 * kRedBlocks + 8);  // block sums, totals, the residual's ticket
    GB_CUDA(cudaMemsetAsync(in.red, 0, (2 * kRedBlocks + 8) * sizeof(double), ctx->stream));
    in.mg_stats = dalloc<double>(A, 4);
    GB_CUDA(cudaMemsetAsync(in.mg_stats, 0, 4 * 8, ctx->stream));
    GB_CUDA(cudaMemsetAsync(in.phi, 0, n * 8, ctx->stream));
    GB_CUDA(cudaMemsetAsync(in.bvec, 0, n * 8, ctx->stream));
    GB_CUDA(cudaMemsetAsync(in.charge, 0, n * 8, ctx->stream));
    // coarsest-level CG needs three extra vectors: give it its own buffers
    Level &c = in.lv.back();
    c.t = dalloc<float>(A, 3 * c.n + 16);
    // (the implicit scheme's coarsest operator changes every step: sm_build_inverse, or the CG)
    in.coarse_build = in.cfg.implicit && small_from(in) > 0 && c.n <= kDirectN
                          ? dalloc<double>(A, (kDirectN * (kDirectN | 1) + 1) / 2)
                          : nullptr;
    in.coarse_inv = in.cfg.implicit ? nullptr
                                    : coarse_inverse(ctx, in, in.cfg.bc_x == PIC_BC_PERIODIC && in.cfg.bc_y == PIC_BC_PERIODIC);
    // meshes whose every level fits one block: the whole solve is one block's work item
    in.small_item = nullptr;
    if (small_from(in) == 0) {
        SmallSolve it{};
        it.D = small_desc(in, 0);
        Level &L = in.lv[0];
        it.diag64 = L.diag64; it.val64 = L.val64;
        it.phi = in.phi; it.phi_prev = in.phi_prev; it.bvec = in.bvec; it.stats = in.mg_stats;
        it.lev = L.lev; it.lmax = L.lmax;
        it.singular = (in.cfg.bc_x == PIC_BC_PERIODIC && in.cfg.bc_y == PIC_BC_PERIODIC) ? 1 : 0;
        it.maxc = std::max(1, in.cfg.mg_max_cycles);
        it.tol = in.cfg.mg_rel_tol;
        int32_t *ns = dalloc<int32_t>(A, 1);
        GB_CUDA(cudaMemsetAsync(ns, 0, 4, ctx->stream));
        it.n_solves = ns;
        in.d_n_solves = ns;
        SmallSolve *d = (SmallSolve *)A.alloc(sizeof(SmallSolve));
        GB_CUDA(cudaMemcpyAsync(d, &it, sizeof(SmallSolve), cudaMemcpyHostToDevice, ctx->stream));
        GB_CUDA(cudaStreamSynchronize(ctx->stream));
        in.small_item = d;
        in.small_smem = (size_t)it.D.smem_floats * 4 + (size_t)it.D.inv_words * 8;
        in.small_cg = !it.D.build && !it.D.cinv;
        in.small_cluster = small_cluster((int)L.n, 1, in.small_smem);
    }
    ++ctx->mesh_epoch;
}

// After a solve that ended with a non-finite residual: the next solve starts from zero instead
// of extrapolating from a potential that holds NaN or Inf.
void poisson_reset_warm_start(pic_ctx *ctx, Instance &in) {
    const int64_t n = in.lv[0].n;
    GB_CUDA(cudaMemsetAsync(in.phi, 0, n * 8, ctx->stream));
    GB_CUDA(cudaMemsetAsync(in.phi_prev, 0, n * 8, ctx->stream));
    in.n_solves = 0;
    if (in.d_n_solves) GB_CUDA(cudaMemsetAsync(in.d_n_solves, 0, 4, ctx->stream));
}

// The batched solver's item table for `list` (copies issued on the context's stream, so a
// step captured afterwards finds the table current and captures no copy).
void poisson_batch_items(pic_ctx *ctx, const std::vector<Instance *> &list) {
    if (ctx->batch_epoch != ctx->mesh_epoch || ctx->batch_n != (int)list.size()) {
        ctx->batch_mem.release_all();
        ctx->batch_items = ctx->batch_mem.alloc(list.size() * sizeof(SmallSolve));
        ctx->batch_smem = 0;
        ctx->batch_cells = 0;
        // largest meshes first: the clusters start in this order (a CTA reserves the largest
        // instance's shared memory, so it has an SM to itself), so the longest solves begin in
        // the first wave and the short ones fill in behind them (every item writes only its
        // own instance)
        std::vector<size_t> order(list.size());
        for (size_t k = 0; k < order.size(); ++k) order[k] = k;
        std::stable_sort(order.begin(), order.end(),
                         [&](size_t a, size_t b) { return list[a]->lv[0].n > list[b]->lv[0].n; });
        for (size_t k = 0; k < list.size(); ++k) {
            GB_CUDA(cudaMemcpyAsync((SmallSolve *)ctx->batch_items + k, list[order[k]]->small_item, sizeof(SmallSolve),
                                    cudaMemcpyDeviceToDevice, ctx->stream));
            ctx->batch_smem = std::max(ctx->batch_smem, list[order[k]]->small_smem);
            ctx->batch_cells = std::max(ctx->batch_cells, (int)list[order[k]]->lv[0].n);
        }
        ctx->batch_cluster = small_cluster(ctx->batch_cells, (int)list.size(), ctx->batch_smem);
        ctx->batch_epoch = ctx->mesh_epoch;
        ctx->batch_n = (int)list.size();
    }
}

void poisson_solve_batch(pic_ctx *ctx, const std::vector<Instance *> &list, const std::vector<const double *> &walls) {
    if (list.empty()) return;
    poisson_batch_items(ctx, list);
    for (size_t k = 0; k < list.size(); ++k) {
        for (int w = 0; w < 4; ++w) list[k]->last_walls[w] = walls[k][w];
        list[k]->mg_on_device = true;
    }
    const int nbuf = small_bufs(ctx->batch_cells, ctx->batch_cluster, ctx->batch_smem);
    launch_small_solve(ctx->batch_items, (int)list.size(), ctx->batch_cluster, nbuf, ctx->batch_smem + (size_t)nbuf * 8192,
                       false, ctx->stream);
    count_launch(ctx);
    check_launch("poisson_solve_batch");
}

// Solve A phi = bvec to ||r|| <= mg_rel_tol ||b||, warm-started from the current phi.
void poisson_solve(pic_ctx *ctx, Instance &in, const double walls[4]) {
    for (int k = 0; k < 4; ++k) in.last_walls[k] = walls[k];
    Level &L = in.lv[0];
    cudaStream_t s = ctx->stream;
    const int64_t n = L.n;
    const bool singular = in.cfg.bc_x == PIC_BC_PERIODIC && in.cfg.bc_y == PIC_BC_PERIODIC;
    if (in.small_item) {
        const int nbuf = small_bufs((int)n, in.small_cluster, in.small_smem);
        launch_small_solve(in.small_item, 1, in.small_cluster, nbuf, in.small_smem + (size_t)nbuf * 8192, in.small_cg, s);
        count_launch(ctx);
        check_launch("poisson_solve");
        in.mg_on_device = true;
        return;
    }
    if (in.n_solves >= 1) {
        k_extrapolate<<<blocks_for(n), kT, 0, s>>>(n, in.phi, in.phi_prev, in.n_solves >= 2 ? 1 : 0);
        count_launch(ctx);
    }
    ++in.n_solves;
    in.mg_on_device = false;
    if (singular) {
        k_area_moments<<<kRedBlocks, kT, 0, s>>>(n, L.lev, L.lmax, in.bvec, in.red);
        k_finish_sums<<<1, 32, 0, s>>>(kRedBlocks, in.red, in.red + 2 * kRedBlocks);
        k_project<<<blocks_for(n), kT, 0, s>>>(n, L.lev, L.lmax, in.red + 2 * kRedBlocks, in.bvec, 0);
        count_launch(ctx, 3);
    }
    const int maxc = std::max(1, in.cfg.mg_max_cycles);
    // launches go to ctx->stream, which is the capture stream while the solve is captured
    auto issue_residual = [&](int first, cudaGraphConditionalHandle h) {
        pdl(k_residual_decide, kRedBlocks, kT, 0, ctx->stream, n, L.col, in.cfg.implicit ? nullptr : L.code, L.val64,
            L.diag64, in.phi, in.bvec, L.b, in.red, (uint32_t *)(in.red + 2 * kRedBlocks + 4), h, in.cfg.mg_rel_tol, maxc,
            in.mg_stats, first);
        count_launch(ctx);
    };
    auto issue_cycle = [&](cudaGraphConditionalHandle h) {
        vcycle(ctx, in, 0, singular);  // (adds its correction to phi)
        issue_residual(0, h);
    };
    if (!in.mg_cycle) {
        // The whole solve as one graph: the residual of the warm start, then a WHILE node
        // whose body is one cycle (V-cycle, correction, FP64 residual); the residual's last
        // kernel decides on the device whether the body runs again, so the host never waits.
        // Captured on a private stream (the context's stream may be the legacy default
        // stream, which cannot be captured) and replayed on the context's stream.
        cudaStream_t cs;
        GB_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
        cudaStream_t saved = ctx->stream;
        const int64_t l0 = ctx->launches;
        ctx->stream = cs;
        cudaGraph_t graph = nullptr;
        cudaGraphConditionalHandle h = 0;
        cudaError_t e = cudaGraphCreate(&graph, 0);
        if (e == cudaSuccess) e = cudaGraphConditionalHandleCreate(&h, graph, 0, cudaGraphCondAssignDefault);
        if (e == cudaSuccess) e = cudaStreamBeginCaptureToGraph(cs, graph, nullptr, nullptr, 0,
                                                                cudaStreamCaptureModeThreadLocal);
        cudaGraphNodeParams np = {};
        if (e == cudaSuccess) {
            if (in.coarse_build) {
                const SmallDesc D = small_desc(in, small_from(in));
                const SmallLevel &C = D.lv[D.nlev - 1];
                if (D.build) {
                    k_coarse_inverse<<<1, 1024, (size_t)C.n * (C.n | 1) * 4, cs>>>(C, singular, (float *)in.coarse_build);
                    count_launch(ctx);
                }
            }
            issue_residual(1, h);
            cudaStreamCaptureStatus status;
            const cudaGraphNode_t *deps = nullptr;
            size_t nd = 0;
            e = cudaStreamGetCaptureInfo(cs, &status, nullptr, nullptr, &deps, nullptr, &nd);
            cudaGraphNode_t wn = nullptr;
            np.type = cudaGraphNodeTypeConditional;
            np.conditional.handle = h;
            np.conditional.type = cudaGraphCondTypeWhile;
            np.conditional.size = 1;
            if (e == cudaSuccess) e = cudaGraphAddNode(&wn, graph, deps, nullptr, nd, &np);
            if (e == cudaSuccess) e = cudaStreamUpdateCaptureDependencies(cs, &wn, nullptr, 1,
                                                                          cudaStreamSetCaptureDependencies);
            cudaGraph_t g2 = nullptr;
            const cudaError_t e2 = cudaStreamEndCapture(cs, &g2);
            if (e == cudaSuccess) e = e2;
        }
        in.mg_pre_nodes = ctx->launches - l0;
        if (e == cudaSuccess) {
            cudaGraph_t body = np.conditional.phGraph_out[0];
            e = cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
            if (e == cudaSuccess) {
                issue_cycle(h);
                cudaGraph_t b2 = nullptr;
                e = cudaStreamEndCapture(cs, &b2);
            }
        }
        ctx->stream = saved;
        in.mg_cycle_nodes = ctx->launches - l0 - in.mg_pre_nodes;
        ctx->launches = l0;
        cudaStreamDestroy(cs);
        if (e == cudaSuccess) e = cudaGraphInstantiate(&in.mg_cycle, graph, 0);
        if (graph) cudaGraphDestroy(graph);
        GB_CUDA(e);
    }
    GB_CUDA(cudaGraphLaunch(in.mg_cycle, s));
    count_launch(ctx, in.mg_pre_nodes);  // the cycles' launches are counted when the stats are read
    if (singular) {  // zero area-weighted mean (a constant changes no residual: once, after the cycles)
        k_area_weighted<<<kRedBlocks, kT, 0, s>>>(n, L.lev, L.lmax, in.phi, in.red);
        pdl(k_finish_sums, 1, 32, 0, s, kRedBlocks, in.red, in.red + 2 * kRedBlocks);
        pdl(k_project, blocks_for(n), kT, 0, s, n, L.lev, L.lmax, in.red + 2 * kRedBlocks, in.phi, 1);
        count_launch(ctx, 3);
    }
    in.mg_on_device = true;
    in.mg_count_cycles = true;
    check_launch("poisson_solve");
}

}  // namespace gbpic
