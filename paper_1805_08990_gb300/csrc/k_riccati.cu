// T3, the exact flow of dP/dt = -P B R^{-1} B^T P (Eq. nonlinear):
//     T3(t) P = (I + t P B R^{-1} B^T)^{-1} P.
// With Bt = B L_R^{-T} (B R^{-1} B^T = Bt Bt^T) and Z = P Bt (n x m), the
// Sherman-Morrison-Woodbury identity gives the m x m form
//     T3(t) P = P - t Z (I_m + t Bt^T Z)^{-1} Z^T,
// which only needs the small SPD matrix M = I_m + t Bt^T P Bt (the dense
// counterpart of the r x r solve of §2.2).  With M = L L^T and Y = Z L^{-T}:
//     T3(t) P = P - t Y Y^T.
// Kernels: (1) Z = P Bt with per-block partial Gram sums Bt^T Z, (2) M from the
// partials (deterministic reduction order), its Cholesky and L^{-1} (FP64; in
// registers for m <= 8), (3) Y = Z L^{-T}, (4) the rank-m update
// P <- P - t Y Y^T (+ q Q); where that is little work (4) forms the rows of Y it needs itself.
// Each kernel takes a batch of independent problems (grouped launch): the
// blocks of every problem are laid end to end and each block finds its
// problem by a binary search over the per-problem block offsets, so a
// problem is computed identically alone or in a batch.
// Everything is FP64.  (1) and (4) stream P once each with coalesced,
// 16-byte vector loads; the row dot-products of (1) are warp reductions.
#include "dme_internal.h"
#include "pdl.cuh"

#include <algorithm>
#include <cstring>
#include <vector>

namespace dme {

constexpr int RZ_MB = 8;        // columns of Bt per pass
constexpr int RZ_DIRECT = 4;    // most columns of Bt read as they lie
constexpr int RZ_WIDE = 1700;   // kernel (1) takes eight rows a block from this n on, if it stages Bt
constexpr int RU_TILE = 32;     // update tile
constexpr int RS_SUM = 8;       // largest m whose partial Gram sums one block adds
// Whether the update forms the rows of Y it needs from Z and L^{-1} (n^2 m (m + 1) / 64 FMAs
// more) or reads those of a launch of its own (5 to 8 us).  T3, us, formed / read: n = 625, m = 8
// 49.1 / 49.9; n = 1024, m = 5 49.3 / 49.8, m = 8 72.3 / 68.3; n = 1500, m = 4 61.9 / 60.3, m = 8 111 / 102;
// n = 2025, m = 3 72.3 / 72.3, m = 4 95.5 / 91.8; n = 4096, m = 2 188 / 185, m = 8 588 / 490.
inline bool ru_fused(int n, int m) { return m <= 8 && (long long)n * n * (m * (m + 1)) <= 50000000; }

constexpr int RZ_PARTS = 608;   // most blocks of kernel (1), and so most partial Gram matrices
// Rows of P per block and step in kernel (1): four with two warps each, or eight with one.
inline int rz_rows(int n, int m) { return m > RZ_DIRECT && n >= RZ_WIDE ? 8 : 4; }
inline int rz_groups(int n, int m) { return (n + rz_rows(n, m) - 1) / rz_rows(n, m); }
inline int rz_blocks(int n, int m) {
    return rz_groups(n, m) < RZ_PARTS ? rz_groups(n, m) : RZ_PARTS;
}

size_t riccati_work_doubles(int n, int m) {
    // Z (n m) | Y (n m) | Gpart (blocks m m) | Linv (m m)
    return (size_t)2 * n * m + (size_t)rz_blocks(n, m) * m * m + (size_t)m * m + 8;
}

// One problem of a (possibly grouped) Riccati update; the block-prefix fields
// map a global block index of each kernel to (problem, local block).
struct RicDesc {
    double* P;
    const double* Bt;
    double* Z;
    double* Y;
    double* Gpart;
    double* Linv;
    const double* Qadd;
    double t, q;
    int n, m;
    int* status;
    int sz, sy, su;     // first block of this problem in the z, y and update grids
    unsigned short parts;           // rz_blocks, rz_rows, ru_fused (ric_shape)
    unsigned char rows, fused;
};

static void ric_shape(RicDesc& d, int n, int m) {
    d.n = n;
    d.m = m;
    d.parts = (unsigned short)rz_blocks(n, m);
    d.rows = (unsigned char)rz_rows(n, m);
    d.fused = ru_fused(n, m);
}

constexpr int kRicLocal = 8;
struct RicBatch {
    RicDesc local[kRicLocal];
    const RicDesc* dev;     // used instead of `local` when nd > kRicLocal
    int nd;
};

__device__ __forceinline__ const RicDesc* ric_descs(const RicBatch& b) { return b.dev ? b.dev : b.local; }

// largest i with start(i) <= blk
template <int FIELD>
__device__ __forceinline__ int ric_find(const RicDesc* d, int nd, int blk) {
    int lo = 0, hi = nd - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        const int st = FIELD == 0 ? d[mid].sz : (FIELD == 1 ? d[mid].sy : d[mid].su);
        if (st <= blk) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// (1) Z[r][c] = sum_k P[r][k] Bt[k][c], four or eight rows at a time (rz_rows; row groups b,
// b + gridDim, ...), two warps or one a row (each of two on half of the row's 64-column steps,
// the halves added in order), and the block's partial Gram sums Gpart[b][i][c] =
// sum_{its rows} Bt[r][i] Z[r][c], one entry a thread, in a fixed order (deterministic, no
// atomics).  MB columns per pass.
// Bound: the FP64 pipe (two FMAs per SM and cycle): n^2 m FMAs, so a pass computes no
// column that is not there, and four rows a block give n / 4 blocks; at most RZ_PARTS of
// them, since one block adds the partial sums (n = 4096, m = 8, 1024 of them: 16 us of its FP64 pipe).
// Up to four columns of Bt are read as they lie; more of them, at a stride of m doubles per
// lane, would keep L1 busier than the FP64 pipe (n = 4096, m = 8: 535 us), so they are staged
// column by column in pairs: sB[c][k / 2] = (Bt[k][c], Bt[k + 1][c]).  Eight rows then share a
// staging, where there are blocks enough (T3, m = 8, four rows / eight: n = 1500 115 / 123 us, 1700
// 131 / 138, 1849 178 / 152, 2025 206 / 171, 4096 626 / 612; m = 32: n = 1500 535 / 505, 2025 717 / 700).
constexpr int RZ_KC = 512, RZ_SB = RZ_KC / 2 + 1;    // (+ 1: the columns' stores in different banks)

template <int MB, bool STAGED, int KSTEP>
__device__ __forceinline__ void riccati_z_row(const RicDesc& d, int row, int kfirst, int c0, int kbeg, int kend,
                                              const double2 (*sB)[RZ_SB], double (&acc)[RZ_MB]) {
    const int n = d.n, m = d.m;
    const double* __restrict__ prow = d.P + (size_t)row * n;
    const double* __restrict__ Bt = d.Bt + c0;
    const bool vec = (n % 2) == 0;
#pragma unroll 2
    for (int k = kbeg + kfirst; k < kend; k += KSTEP) {
        const bool two = k + 1 < kend;
        double p0, p1 = 0.0;
        if (vec) {
            const double2 v = *reinterpret_cast<const double2*>(prow + k);
            p0 = v.x;
            p1 = v.y;
        } else {
            p0 = prow[k];
            if (two) p1 = prow[k + 1];
        }
#pragma unroll
        for (int c = 0; c < MB; ++c) {
            double b0, b1;
            if (STAGED) {
                const double2 b = sB[c][(k - kbeg) >> 1];
                b0 = b.x;
                b1 = b.y;
            } else {
                b0 = Bt[(size_t)k * m + c];
                b1 = two ? Bt[(size_t)(k + 1) * m + c] : 0.0;
            }
            acc[c] = fma(p1, b1, fma(p0, b0, acc[c]));
        }
    }
}

// WIDE: eight rows a block, a warp each; else four with two warps each.  A batch of both kinds
// takes two launches, in which the other kind's blocks return at once.
template <bool WIDE>
__global__ void __launch_bounds__(256) riccati_z_kernel(const __grid_constant__ RicBatch batch) {
    pdl_trigger();
    pdl_wait();
    __shared__ double2 sB[RZ_MB][RZ_SB];
    __shared__ double sH[8][RZ_MB], sZ[WIDE ? 8 : 4][RZ_MB];
    const RicDesc* ds = ric_descs(batch);
    const int ip = ric_find<0>(ds, batch.nd, blockIdx.x);
    const RicDesc& d = ds[ip];
    const int lb = blockIdx.x - d.sz;
    const int n = d.n, m = d.m;
    constexpr int ROWS = WIDE ? 8 : 4, KSTEP = WIDE ? 64 : 128;
    if (d.rows != ROWS) return;
    const double* __restrict__ Bt = d.Bt;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
    const int parts = d.parts, groups = (n + ROWS - 1) / ROWS;
    const int kfirst = 2 * lane + (WIDE ? 0 : 64 * (warp & 1));
    for (int c0 = 0; c0 < m; c0 += RZ_MB) {
        const int mb = min(RZ_MB, m - c0);
        const int gi = tid / mb, gj = tid % mb;               // this thread's Gram entry (m mb <= 256)
        double gram = 0.0;
        for (int g = lb; g < groups; g += parts) {
            const int row = g * ROWS + (WIDE ? warp : warp >> 1);
            double acc[RZ_MB];
#pragma unroll
            for (int c = 0; c < RZ_MB; ++c) acc[c] = 0.0;
            if (mb <= RZ_DIRECT) {
                if (row < n) {
                    switch (mb) {
                        case 1: riccati_z_row<1, false, KSTEP>(d, row, kfirst, c0, 0, n, sB, acc); break;
                        case 2: riccati_z_row<2, false, KSTEP>(d, row, kfirst, c0, 0, n, sB, acc); break;
                        case 3: riccati_z_row<3, false, KSTEP>(d, row, kfirst, c0, 0, n, sB, acc); break;
                        default: riccati_z_row<4, false, KSTEP>(d, row, kfirst, c0, 0, n, sB, acc); break;
                    }
                }
            } else {
                for (int k0 = 0; k0 < n; k0 += RZ_KC) {
                    __syncthreads();
                    for (int e = tid; e < (RZ_KC / 2) * mb; e += blockDim.x) {
                        const int kp = e / mb, c = e % mb, k = k0 + 2 * kp;      // consecutive in memory over c
                        double2 v;
                        v.x = k < n ? Bt[(size_t)k * m + c0 + c] : 0.0;
                        v.y = k + 1 < n ? Bt[(size_t)(k + 1) * m + c0 + c] : 0.0;
                        sB[c][kp] = v;
                    }
                    __syncthreads();
                    if (row >= n) continue;
                    const int kend = min(n, k0 + RZ_KC);
                    switch (mb) {
                        case 5: riccati_z_row<5, true, KSTEP>(d, row, kfirst, c0, k0, kend, sB, acc); break;
                        case 6: riccati_z_row<6, true, KSTEP>(d, row, kfirst, c0, k0, kend, sB, acc); break;
                        case 7: riccati_z_row<7, true, KSTEP>(d, row, kfirst, c0, k0, kend, sB, acc); break;
                        default: riccati_z_row<8, true, KSTEP>(d, row, kfirst, c0, k0, kend, sB, acc); break;
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < RZ_MB; ++c) {
                if (c >= mb) break;
                double v = acc[c];
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
                if (lane == 0) sH[warp][c] = v;
            }
            __syncthreads();
            if (tid < ROWS * mb) {
                const int r = tid / mb, c = tid % mb, rr = g * ROWS + r;
                double v = 0.0;
                if (rr < n) {
                    if constexpr (WIDE) v = sH[r][c];
                    else v = sH[2 * r][c] + sH[2 * r + 1][c];
                }
                sZ[r][c] = v;
                if (rr < n) d.Z[(size_t)rr * m + c0 + c] = v;
            }
            __syncthreads();
            if (gi < m)
                for (int r = 0; r < ROWS; ++r) {
                    const int rr = g * ROWS + r;
                    if (rr < n) gram = fma(Bt[(size_t)rr * m + gi], sZ[r][gj], gram);
                }
        }
        if (gi < m) d.Gpart[(size_t)lb * m * m + (size_t)gi * m + c0 + gj] = gram;
        __syncthreads();
    }
}

// (1c) For m > RS_SUM: the partial sums added over the whole chip, 32 entries a block, a warp
// per eighth of the parts, into part 0; in one block their m^2 FP64 adds a part kept that SM's pipe
// busy for 0.27 us each (n = 2025, m = 32: 254 us with the factor, 70 with this launch).
__global__ void __launch_bounds__(256) riccati_gsum_kernel(const __grid_constant__ RicBatch batch) {
    pdl_trigger();
    pdl_wait();
    __shared__ double sums[8][32];
    const RicDesc& d = ric_descs(batch)[blockIdx.y];
    const int E = d.m * d.m, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;
    if (d.m <= RS_SUM || blockIdx.x * 32 >= E) return;
    const int parts = d.parts;
    double s = 0.0;
    if (e < E) {
#pragma unroll 8
        for (int b = warp; b < parts; b += 8) s += d.Gpart[(size_t)b * E + e];
    }
    sums[warp][lane] = s;
    __syncthreads();
    if (warp == 0 && e < E) {
        for (int w = 1; w < 8; ++w) s += sums[w][lane];
        d.Gpart[e] = s;
    }
}

// Threads of riccati_small_kernel for a problem: few partial sums leave most of 1024 threads
// nothing but the tree over them; many need the loads in flight (n = 4096, m = 8: 35 us with
// 256 threads, 20 with 1024).  The order of the sums follows from it, not from the launch's
// size, so a problem gives the same bits alone and in a batch.
__host__ __device__ __forceinline__ int rs_threads(int parts, int m) {
    return m <= 16 && (m > RS_SUM ? 1 : parts) * m * m <= 4096 ? 256 : 1024;
}

// M = I + t (G + G^T) / 2 for m <= RS_MAX, its Cholesky and L^{-1} in one warp: row `lane` of
// M in registers, the pivot row handed out by shuffles (through shared memory, with the
// columns of L^{-1} in local arrays, n = 4096, m = 8 took 28 us of which the sums were 12).
constexpr int RS_MAX = 8;
__device__ __forceinline__ void riccati_factor_small(const RicDesc& d, const double (&G)[32][33], int lane) {
    const int m = d.m;
    double a[RS_MAX], rinv[RS_MAX];
#pragma unroll
    for (int j = 0; j < RS_MAX; ++j)
        a[j] = (lane < m && j < m) ? (lane == j ? 1.0 : 0.0) + d.t * 0.5 * (G[lane][j] + G[j][lane]) : 0.0;
#pragma unroll
    for (int j = 0; j < RS_MAX; ++j) {
        if (j >= m) break;
        const double dj = __shfl_sync(0xffffffffu, a[j], j);
        if (!(dj > 0.0)) {
            if (lane == 0) atomicOr(d.status, DEV_NOTSPD);
            return;
        }
        rinv[j] = rsqrt(dj);
        const double lj = a[j] * rinv[j];                     // L[lane][j], lane >= j
        a[j] = lj;
#pragma unroll
        for (int k = j + 1; k < RS_MAX; ++k) a[k] = fma(-lj, __shfl_sync(0xffffffffu, lj, k), a[k]);
    }
    // column `lane` of L^{-1}: y_r = (e_r - sum_{k < r} L[r][k] y_k) / L[r][r]
    double y[RS_MAX];
#pragma unroll
    for (int r = 0; r < RS_MAX; ++r) {
        if (r >= m) break;
        double s = (r == lane) ? 1.0 : 0.0;
#pragma unroll
        for (int k = 0; k < r; ++k) s = fma(-__shfl_sync(0xffffffffu, a[k], r), y[k], s);
        y[r] = (r < lane) ? 0.0 : s * rinv[r];
        if (lane < m) d.Linv[r * m + lane] = y[r];
    }
}

// (2) M = I + t sym(sum_b Gpart[b]); M = L L^T; Linv = L^{-1}.  One block per
// problem.  The sum over blocks is a fixed two-level order (strided partial
// sums, then a tree), so the result does not depend on scheduling.
__global__ void __launch_bounds__(1024) riccati_small_kernel(const __grid_constant__ RicBatch batch) {
    pdl_trigger();
    pdl_wait();
    __shared__ double red[1024];
    __shared__ double L[32][33];
    const RicDesc& d = ric_descs(batch)[blockIdx.x];
    const int m = d.m;
    const int nblocks = m > RS_SUM ? 1 : d.parts;
    const double t = d.t;
    const int E = m * m;
    const int G = max(1, rs_threads(nblocks, m) / E);
    const int tid = threadIdx.x;
    const int e = tid % E, g = tid / E;
    double sacc = 0.0;
    if (g < G)
        for (int b = g; b < nblocks; b += G) sacc += d.Gpart[(size_t)b * E + e];
    red[tid] = (g < G) ? sacc : 0.0;
    __syncthreads();
    // tree over groups: group g adds group g + half (fixed order)
    for (int half = 1; half < G; half <<= 1) {
        if (g < G && (g % (2 * half)) == 0 && g + half < G) red[tid] += red[tid + half * E];
        __syncthreads();
    }
    if (tid < E) L[tid / m][tid % m] = red[tid];
    __syncthreads();
    if (tid >= 32) return;
    if (m <= RS_MAX) {
        riccati_factor_small(d, L, tid);
        return;
    }
    const int lane = tid;
    // symmetrise and add the identity: M = I + t (G + G^T)/2
    double Mv[32];
    for (int e2 = lane; e2 < E; e2 += 32) {
        const int i = e2 / m, j = e2 % m;
        Mv[e2 / 32] = (i == j ? 1.0 : 0.0) + t * 0.5 * (L[i][j] + L[j][i]);
    }
    __syncwarp();
    for (int e2 = lane; e2 < E; e2 += 32) L[e2 / m][e2 % m] = Mv[e2 / 32];
    __syncwarp();
    // Cholesky in place (lower)
    for (int j = 0; j < m; ++j) {
        double dj = L[j][j];
        for (int k = 0; k < j; ++k) dj -= L[j][k] * L[j][k];
        if (!(dj > 0.0)) {
            if (lane == 0) atomicOr(d.status, DEV_NOTSPD);
            return;
        }
        dj = sqrt(dj);
        __syncwarp();
        for (int i = j + 1 + lane; i < m; i += 32) {
            double s2 = L[i][j];
            for (int k = 0; k < j; ++k) s2 -= L[i][k] * L[j][k];
            L[i][j] = s2 / dj;
        }
        __syncwarp();
        if (lane == 0) L[j][j] = dj;
        __syncwarp();
    }
    // Linv column by column (forward substitution on e_c); lane c owns column c
    for (int c = lane; c < m; c += 32) {
        double x[32];
        for (int r = 0; r < m; ++r) {
            double s2 = (r == c) ? 1.0 : 0.0;
            for (int k = 0; k < r; ++k) s2 -= L[r][k] * x[k];
            x[r] = (r < c) ? 0.0 : s2 / L[r][r];
        }
        for (int r = 0; r < m; ++r) d.Linv[r * m + c] = x[r];
    }
}

// (1b) The partial Gram sums of (1) from a Z computed elsewhere (same blocks and order).
__global__ void riccati_gpart_kernel(const __grid_constant__ RicBatch batch) {
    pdl_trigger();
    pdl_wait();
    const RicDesc* ds = ric_descs(batch);
    const RicDesc& d = ds[ric_find<0>(ds, batch.nd, blockIdx.x)];
    const int lb = blockIdx.x - d.sz, n = d.n, m = d.m;
    const int parts = d.parts, rows = d.rows, groups = (n + rows - 1) / rows;
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
        const int i = e / m, c = e % m;
        double sacc = 0.0;
        for (int g = lb; g < groups; g += parts)
            for (int r = 0; r < rows; ++r) {
                const int rr = g * rows + r;
                if (rr < n) sacc = fma(d.Bt[(size_t)rr * m + i], d.Z[(size_t)rr * m + c], sacc);
            }
        d.Gpart[(size_t)lb * m * m + e] = sacc;
    }
}

// (3) Y[i][r] = sum_{c <= r} Linv[r][c] Z[i][c]   (Y = Z L^{-T}); Y = 0 when the
// m x m matrix was not SPD (an update with Y then leaves P as it is).
__device__ __forceinline__ double riccati_y_entry(const RicDesc& d, int i, int r) {
    double s = 0.0;
    for (int c = 0; c <= r; ++c) s = fma(d.Linv[r * d.m + c], d.Z[(size_t)i * d.m + c], s);
    return s;
}

__global__ void riccati_y_kernel(const __grid_constant__ RicBatch batch) {
    pdl_trigger();
    pdl_wait();
    const RicDesc* ds = ric_descs(batch);
    const RicDesc& d = ds[ric_find<1>(ds, batch.nd, blockIdx.x)];
    const int i = (blockIdx.x - d.sy) * blockDim.x + threadIdx.x;
    const int m = d.m;
    if (i >= d.n) return;
    const bool skip = (*d.status & DEV_NOTSPD) != 0;
    for (int r = 0; r < m; ++r) d.Y[(size_t)i * m + r] = skip ? 0.0 : riccati_y_entry(d, i, r);
}

// (4) P[i][j] <- P[i][j] - t sum_r Y[i][r] Y[j][r] (+ q Q[i][j]).  The result is
// symmetric (the sum is taken in the same order for (i, j) and (j, i)), so only
// the 32 x 32 tiles on or above the diagonal are computed: each reads its
// upper block of P, writes it, and for an off-diagonal tile also writes the
// transposed block below the diagonal from a shared-memory copy (coalesced).
// Half of the FP64 work and of the traffic on P of a full update.  Fused problems
// (ru_fused) form the Y rows of the tile from Z and Linv here (m (m + 1) FMAs per
// row against 32 m of the tile's own), which saves them a launch.  The tile's entries
// of P (and Q) are loaded together before the first is stored: one by one, each load
// waited behind the store before it (64-wide tiles, n = 81: 16 us).
__global__ void __launch_bounds__(256) riccati_update_kernel(const __grid_constant__ RicBatch batch) {
    pdl_trigger();
    pdl_wait();
    const RicDesc* ds = ric_descs(batch);
    const RicDesc& d = ds[ric_find<2>(ds, batch.nd, blockIdx.x)];
    if (*d.status & DEV_NOTSPD) return;
    __shared__ double Yi[RU_TILE][33], Yj[RU_TILE][33];
    __shared__ double Vt[RU_TILE][RU_TILE + 1];
    const int n = d.n, m = d.m;
    const int T = (n + RU_TILE - 1) / RU_TILE;
    // upper-triangle tile (ti <= tj), row by row
    int rem = blockIdx.x - d.su, ti = 0;
    while (rem >= T - ti) {
        rem -= T - ti;
        ++ti;
    }
    const int tj = ti + rem;
    const int i0 = ti * RU_TILE, j0 = tj * RU_TILE;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 32 x 8
    double pv[4], qv[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        const int i = i0 + ty + 8 * h, j = j0 + tx;
        const bool in = i < n && j < n;
        const size_t off = (size_t)i * n + j;
        pv[h] = in ? d.P[off] : 0.0;
        qv[h] = in && d.Qadd ? d.Qadd[off] : 0.0;
    }
    const bool fuse = d.fused != 0;
    for (int e = threadIdx.x; e < RU_TILE * m; e += blockDim.x) {
        const int r = e / m, c = e % m;
        const int gi = i0 + r, gj = j0 + r;
        Yi[r][c] = gi < n ? (fuse ? riccati_y_entry(d, gi, c) : d.Y[(size_t)gi * m + c]) : 0.0;
        Yj[r][c] = gj < n ? (fuse ? riccati_y_entry(d, gj, c) : d.Y[(size_t)gj * m + c]) : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        const int di = ty + 8 * h, i = i0 + di, j = j0 + tx;
        if (i >= n || j >= n) continue;
        double s = 0.0;
        for (int c = 0; c < m; ++c) s = fma(Yi[di][c], Yj[tx][c], s);
        double v = pv[h] - d.t * s;
        if (d.Qadd) v += d.q * qv[h];
        d.P[(size_t)i * n + j] = v;
        Vt[di][tx] = v;
    }
    if (ti == tj) return;
    __syncthreads();
    // mirror: P[j][i] = V[i][j] for the block below the diagonal
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        const int dj = ty + 8 * h, j = j0 + dj, i = i0 + tx;
        if (j < n && i < n) d.P[(size_t)j * n + i] = Vt[tx][dj];
    }
}

dme_status launch_riccati_from_z(const double* Bt, int n, int m, double t, double* work, int* status,
                                 cudaStream_t st) {
    RicBatch b;
    std::memset(&b, 0, sizeof(b));
    b.nd = 1;
    RicDesc& d = b.local[0];
    d.P = nullptr;
    d.Bt = Bt;
    d.Z = work;
    d.Y = d.Z + (size_t)n * m;
    d.Gpart = d.Y + (size_t)n * m;
    d.Linv = d.Gpart + (size_t)rz_blocks(n, m) * m * m;
    d.t = t;
    ric_shape(d, n, m);
    d.status = status;
    DME_CUDA_TRY(pdl_launch(riccati_gpart_kernel, rz_blocks(n, m), 64, 0, st, b));
    if (m > RS_SUM) DME_CUDA_TRY(pdl_launch(riccati_gsum_kernel, (m * m + 31) / 32, 256, 0, st, b));
    DME_CUDA_TRY(pdl_launch(riccati_small_kernel, 1, rs_threads(d.parts, m), 0, st, b));
    DME_CUDA_TRY(pdl_launch(riccati_y_kernel, (n + 127) / 128, 128, 0, st, b));
    return DME_OK;
}

RicItem make_ric_item(double* P, const double* Bt, int n, int m, double t, const double* Qadd, double q,
                      double* work, int* status) {
    RicItem it;
    it.P = P;
    it.Bt = Bt;
    it.n = n;
    it.m = m;
    it.t = t;
    it.Qadd = Qadd;
    it.q = q;
    it.work = work;
    it.status = status;
    return it;
}

dme_status launch_riccati_grouped(const std::vector<RicItem>& items, void* dev_desc, cudaStream_t st,
                                  DescArena* arena) {
    if (items.empty()) return DME_OK;
    std::vector<RicDesc> ds(items.size());
    int sz = 0, sy = 0, su = 0;
    for (size_t k = 0; k < items.size(); ++k) {
        const RicItem& it = items[k];
        RicDesc& d = ds[k];
        const int n = it.n, m = it.m;
        d.P = it.P;
        d.Bt = it.Bt;
        d.Z = it.work;
        d.Y = d.Z + (size_t)n * m;
        d.Gpart = d.Y + (size_t)n * m;
        d.Linv = d.Gpart + (size_t)rz_blocks(n, m) * m * m;
        d.Qadd = it.Qadd;
        d.t = it.t;
        d.q = it.q;
        ric_shape(d, n, m);
        d.status = it.status;
        d.sz = sz;
        d.sy = sy;
        d.su = su;
        sz += rz_blocks(n, m);
        sy += (n + 127) / 128;
        const int tn = (n + RU_TILE - 1) / RU_TILE;
        su += tn * (tn + 1) / 2;
    }
    RicBatch b;
    std::memset(&b, 0, sizeof(b));
    b.nd = (int)ds.size();
    if (ds.size() <= (size_t)kRicLocal) {
        for (size_t k = 0; k < ds.size(); ++k) b.local[k] = ds[k];
        b.dev = nullptr;
    } else {
        if (arena) {
            dev_desc = arena->put(ds.data(), ds.size() * sizeof(RicDesc));
            if (!dev_desc) return set_error("grouped Riccati: descriptor arena full"), DME_ENOMEM;
        } else {
            if (!dev_desc) {
                set_error("grouped Riccati: more than 8 problems need a device descriptor buffer");
                return DME_EINVAL;
            }
            DME_CUDA_TRY(cudaMemcpyAsync(dev_desc, ds.data(), ds.size() * sizeof(RicDesc), cudaMemcpyHostToDevice, st));
        }
        b.dev = reinterpret_cast<const RicDesc*>(dev_desc);
    }
    int mmax = 0, threads = 256;
    bool y = false, wide = false, narrow = false;
    for (const RicItem& it : items) {
        (rz_rows(it.n, it.m) == 8 ? wide : narrow) = true;
        mmax = std::max(mmax, it.m);
        y = y || !ru_fused(it.n, it.m);
        threads = std::max(threads, rs_threads(rz_blocks(it.n, it.m), it.m));
    }
    if (narrow) DME_CUDA_TRY(pdl_launch(riccati_z_kernel<false>, sz, 256, 0, st, b));
    if (wide) DME_CUDA_TRY(pdl_launch(riccati_z_kernel<true>, sz, 256, 0, st, b));
    if (mmax > RS_SUM) DME_CUDA_TRY(pdl_launch(riccati_gsum_kernel, dim3((mmax * mmax + 31) / 32, b.nd), 256, 0, st, b));
    DME_CUDA_TRY(pdl_launch(riccati_small_kernel, b.nd, threads, 0, st, b));
    if (y) DME_CUDA_TRY(pdl_launch(riccati_y_kernel, sy, 128, 0, st, b));
    DME_CUDA_TRY(pdl_launch(riccati_update_kernel, su, 256, 0, st, b));
    DME_CUDA_TRY(cudaGetLastError());
    return DME_OK;
}

size_t riccati_desc_bytes() { return sizeof(RicDesc); }

// K = R^{-1} B^T P for symmetric P, with R = L L^T and Bt = B L^{-T}:
// B^T P = L Bt^T P = L Z^T (Z = P Bt), so K = L^{-T} Z^T, i.e. L^T K = Z^T,
// solved by back substitution for each column j of K (one thread per column).
__global__ void lqr_gain_kernel(const double* __restrict__ Z, const double* __restrict__ L, double* __restrict__ K,
                                int n, int m) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    double x[32];
    for (int r = m - 1; r >= 0; --r) {
        double s = Z[(size_t)j * m + r];
        for (int c = r + 1; c < m; ++c) s -= L[c * m + r] * x[c];
        x[r] = s / L[r * m + r];
        K[(size_t)r * n + j] = x[r];
    }
}

// The gain of step *ctr into Kbase + (*ctr) m n, then ++*ctr (a single thread,
// after the gain kernel in stream order): one record per replayed step.
__global__ void lqr_gain_hist_kernel(const double* __restrict__ Z, const double* __restrict__ L,
                                     double* __restrict__ Kbase, int n, int m, const int* __restrict__ ctr,
                                     int cap) {
    const int k = *ctr;
    if (k >= cap) return;
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    double* K = Kbase + (size_t)k * m * n;
    double x[32];
    for (int r = m - 1; r >= 0; --r) {
        double s = Z[(size_t)j * m + r];
        for (int c = r + 1; c < m; ++c) s -= L[c * m + r] * x[c];
        x[r] = s / L[r * m + r];
        K[(size_t)r * n + j] = x[r];
    }
}

__global__ void counter_inc_kernel(int* ctr) { *ctr += 1; }

static void launch_z(const RicBatch& b, int n, int m, cudaStream_t st) {
    if (rz_rows(n, m) == 8) riccati_z_kernel<true><<<rz_blocks(n, m), 256, 0, st>>>(b);
    else riccati_z_kernel<false><<<rz_blocks(n, m), 256, 0, st>>>(b);
}

dme_status launch_lqr_gain_hist(const double* P, const double* Bt, const double* LR, int n, int m, double* work,
                                double* Kbase, int* ctr, int cap, cudaStream_t st) {
    RicBatch b;
    std::memset(&b, 0, sizeof(b));
    RicDesc& d = b.local[0];
    d.P = const_cast<double*>(P);
    d.Bt = Bt;
    d.Z = work;
    d.Y = d.Z + (size_t)n * m;
    d.Gpart = d.Y + (size_t)n * m;
    ric_shape(d, n, m);
    b.nd = 1;
    launch_z(b, n, m, st);                                   // Z = P Bt (P is only read)
    lqr_gain_hist_kernel<<<(n + 127) / 128, 128, 0, st>>>(d.Z, LR, Kbase, n, m, ctr, cap);
    counter_inc_kernel<<<1, 1, 0, st>>>(ctr);
    DME_CUDA_TRY(cudaGetLastError());
    return DME_OK;
}

dme_status launch_lqr_gain(const double* P, const double* Bt, const double* LR, int n, int m, double* work,
                           double* K, cudaStream_t st) {
    RicBatch b;
    std::memset(&b, 0, sizeof(b));
    RicDesc& d = b.local[0];
    d.P = const_cast<double*>(P);
    d.Bt = Bt;
    d.Z = work;
    d.Y = d.Z + (size_t)n * m;
    d.Gpart = d.Y + (size_t)n * m;
    ric_shape(d, n, m);
    b.nd = 1;
    launch_z(b, n, m, st);                                   // Z = P Bt (P is only read)
    lqr_gain_kernel<<<(n + 127) / 128, 128, 0, st>>>(d.Z, LR, K, n, m);
    DME_CUDA_TRY(cudaGetLastError());
    return DME_OK;
}

void launch_riccati(double* P, const double* Bt, int n, int m, double t, const double* Qadd, double q,
                    double* work, int* status, cudaStream_t st) {
    std::vector<RicItem> v{make_ric_item(P, Bt, n, m, t, Qadd, q, work, status)};
    launch_riccati_grouped(v, nullptr, st);
}

}  // namespace dme
