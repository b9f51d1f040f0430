// The action of the matrix exponential on a block of vectors by Newton
// interpolation at Leja points (the `expleja` step of the paper's low-rank
// algorithms, §3), for a sparse A^T in CSR.  Over each substep the series
//     w_0 = v,  w_{k+1} = (A^T - c I) w_k / g - x_k w_k,   p = sum_k d_k w_k
// needs one SpMM of the n x r block per term and a stopping test on the norms
// of the newest term and of the partial sum.  The block is small (a few MB) and
// the terms are many (the count grows with t ||A||), so one launch per term
// would be bound by launch and host round-trip latency: instead one persistent
// cooperative launch runs every term of every substep of an application.  Each
// thread owns the same entries (row, j) throughout; a term is a pass over them
// (SpMM row, recurrence, accumulation, per-block partial norms) and a grid barrier.
// Bound: the chain of latencies from barrier to barrier (L2 gather, release, arrival,
// poll), then FP64 issue (nnz + 2 FMAs per entry and term, two per SM and cycle).  So
//  - the block after the workers only sums the partial norms, in a fixed order, one term
//    late: its arrival at the barrier of term k carries the decision on term k - 1, and
//    every block takes the same one (one term more than the test asks for);
//  - the barrier is one counter: release arrivals, acquire polls, nobody in between;
//  - a thread's stored entries (in shared memory), its w_k and its sum stay on chip
//    while every thread has at most two entries;
//  - the norms are formed in fp32 from the top bits of the entries: in FP64 the shuffles
//    and block sums alone were 830 FP64 warp instructions per SM and term.
// (n = 3600, r = 18 .. 60, 82 terms: 790 us an action with the terms in global memory and the last
// arriving block summing the norms, 395 now.)
#include "dme_internal.h"

#include <algorithm>

namespace dme {

namespace {

constexpr int LJ_THREADS = 256;
constexpr int LJ_PASS = 2;         // entries per thread held on chip
constexpr int LJ_NNZ = 1536;       // stored entries of A^T of a block's rows held on chip
constexpr unsigned LJ_SPIN_LIMIT = 1u << 22;

// Block sum of two values; the result is valid in thread 0.  Every write of the block
// before it is ordered before what thread 0 does next.
__device__ __forceinline__ void block_sum2(float& a, float& b, float* sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, off);
        b += __shfl_xor_sync(0xffffffffu, b, off);
    }
    if (lane == 0) {
        sh[2 * warp] = a;
        sh[2 * warp + 1] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        a = 0.0f;
        b = 0.0f;
#pragma unroll
        for (int w = 0; w < LJ_THREADS / 32; ++w) {   // fixed order
            a += sh[2 * w];
            b += sh[2 * w + 1];
        }
    }
}

// Thread 0's arrival: everything the block wrote before its last __syncthreads is visible
// to whoever polls the counter.
__device__ __forceinline__ void lj_arrive(unsigned long long* cnt, unsigned long long add) {
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(cnt), "l"(add) : "memory");
}

// Wait until the counter's low word reaches target; the high word (the barrier at which
// the current substep stops) goes to `stop`.  False after a timeout (status set).
__device__ __forceinline__ bool lj_wait(const unsigned long long* cnt, unsigned target, int* status, int2* s_word,
                                        unsigned& stop) {
    if (threadIdx.x == 0) {
        unsigned long long v = 0;
        int ok = 1;
        for (unsigned it = 0;;) {
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(cnt) : "memory");
            if ((unsigned)v >= target) break;
            if (++it > LJ_SPIN_LIMIT) {
                atomicOr(status, DEV_TIMEOUT);
                ok = 0;
                break;
            }
            __nanosleep(20);
        }
        *s_word = make_int2(ok, (int)(v >> 32));
    }
    __syncthreads();
    const int2 w = *s_word;
    stop = (unsigned)w.y;
    return w.x != 0;
}

// The exponent field of |x| (0 for zero and subnormals).
__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }

// |x| 2^(1023 - e0) as a float (20 mantissa bits), from the bits of x: the stopping test's
// norms need a few digits and run beside the FP64 pipe.  Saturates at 2^60.
__device__ __forceinline__ float mag(double x, int e0) {
    const int h = __double2hiint(x) & 0x7FFFFFFF;
    const int e = (h >> 20) - e0;
    if (e < -100 || (h >> 20) == 0) return 0.0f;
    if (e > 60) return 1.152921504606847e18f;
    return __int_as_float(((e + 127) << 23) | ((h & 0xFFFFF) << 3));
}

struct LejaArgs {
    const int* ptr;
    const int* idx;
    const double* val;
    int n, r;
    const double* X;
    int ldx;
    double* Y;
    int ldy;
    double* Wa;
    double* Wb;
    int ldw;
    double c, invg, scale, tol;
    int substeps, terms;
    float* part;                // 2 buffers x 2 gridDim floats
    unsigned long long* cnt;    // arrivals (low word) and the stopping barrier (high word)
    unsigned* em;               // largest exponent field of the substep's v (two, by parity)
    int* status;                // (cnt and em zeroed before the launch)
    double xi[80];
    double dd[80];
};

// The entries (row, j) a thread owns: e = first, first + stride, ... < n r in
// row-major order, walked without a division per entry.
struct Entries {
    int row0, j0, drow, dj, n, r;
    __device__ Entries(int n_, int r_, int blocks) : n(n_), r(r_) {
        const size_t first = (size_t)blockIdx.x * LJ_THREADS + threadIdx.x;
        const size_t stride = (size_t)blocks * LJ_THREADS;
        row0 = (int)(first / r_);
        j0 = (int)(first % r_);
        drow = (int)(stride / r_);
        dj = (int)(stride % r_);
    }
    __device__ __forceinline__ void next(int& row, int& j) const {
        row += drow;
        j += dj;
        if (j >= r) {
            j -= r;
            ++row;
        }
    }
};

// The block after the workers: sums the partial norms of each term while the workers are
// at the next one, and stops after two consecutive terms |d_k| |w_k| <= tol |p|.
__device__ void leja_sums(const LejaArgs& a, float* sh, int2* s_word) {
    const int workers = gridDim.x - 1;
    unsigned b = 0, told = 0, stop;
    for (int sub = 0; sub < a.substeps; ++sub) {
        __syncthreads();
        if (threadIdx.x == 0) lj_arrive(a.cnt, 1);
        if (!lj_wait(a.cnt, ++b * gridDim.x, a.status, s_word, stop)) return;
        int small = 0;
        for (int k = 1; k < a.terms; ++k) {
            unsigned long long add = 1;
            float aw = 0.0f, ap = 0.0f;
            if (k > 1) {
                const float2* part = reinterpret_cast<const float2*>(a.part + (size_t)((k - 1) & 1) * 2 * gridDim.x);
                for (int i = threadIdx.x; i < workers; i += LJ_THREADS) {
                    const float2 v = __ldcg(part + i);
                    aw += v.x;
                    ap += v.y;
                }
            }
            block_sum2(aw, ap, sh);
            ++b;
            if (threadIdx.x == 0) {
                if (k > 1) {
                    const double dk = a.dd[k - 1];
                    small = dk * dk * aw <= a.tol * a.tol * ap ? small + 1 : 0;
                }
                if (small == 2) {
                    add += (unsigned long long)(b - told) << 32;
                    told = b;
                }
                lj_arrive(a.cnt, add);
            }
            if (!lj_wait(a.cnt, b * gridDim.x, a.status, s_word, stop)) return;
            if (stop == b) break;
        }
    }
}

// CACHED: at most LJ_PASS entries per thread and LJ_NNZ stored entries in a block's rows.
template <bool CACHED>
__global__ void __launch_bounds__(LJ_THREADS, CACHED ? 6 : 1) leja_persistent_kernel(const __grid_constant__ LejaArgs a) {
    __shared__ float sh[2 * (LJ_THREADS / 32)];
    __shared__ int2 s_word;
    if (blockIdx.x == gridDim.x - 1) {
        leja_sums(a, sh, &s_word);
        return;
    }
    __shared__ int s_idx[CACHED ? LJ_NNZ : 1];
    __shared__ double s_val[CACHED ? LJ_NNZ : 1];
    const Entries it(a.n, a.r, gridDim.x - 1);
    // CACHED: entry u of the thread is (row, j) = er[u], ej[u] (er < 0: none), its stored
    // entries are qb[u] .. qe[u] of the shared copy
    int er[LJ_PASS], ej[LJ_PASS], qb[LJ_PASS], qe[LJ_PASS];
    double w[LJ_PASS], p[LJ_PASS];
    if constexpr (CACHED) {
        int row = it.row0, j = it.j0, base = 0;
#pragma unroll
        for (int u = 0; u < LJ_PASS; ++u) {
            er[u] = row < a.n ? row : -1;
            ej[u] = j;
            w[u] = p[u] = 0.0;
            qb[u] = qe[u] = 0;
            // the rows of the block's 256 entries of this pass are contiguous
            const size_t first = ((size_t)u * (gridDim.x - 1) + blockIdx.x) * LJ_THREADS, total = (size_t)a.n * a.r;
            if (first < total) {
                const int lo = (int)(first / a.r), hi = (int)(min(first + LJ_THREADS, total) - 1) / a.r;
                const int q0 = a.ptr[lo], q1 = a.ptr[hi + 1];
                for (int q = q0 + threadIdx.x; q < q1; q += LJ_THREADS) {
                    s_idx[base + q - q0] = a.idx[q];
                    s_val[base + q - q0] = a.val[q];
                }
                if (er[u] >= 0) {
                    qb[u] = a.ptr[row] - q0 + base;
                    qe[u] = a.ptr[row + 1] - q0 + base;
                    w[u] = a.X[(size_t)row * a.ldx + j];
                    a.Wa[(size_t)row * a.ldw + j] = w[u];
                }
                base += q1 - q0;
            }
            it.next(row, j);
        }
    } else {
        // v = X (Y may be X: every entry is read and written by its own thread)
        for (int row = it.row0, j = it.j0; row < a.n; it.next(row, j))
            a.Wa[(size_t)row * a.ldw + j] = a.X[(size_t)row * a.ldx + j];
    }
    unsigned b = 0, stop;
    for (int sub = 0; sub < a.substeps; ++sub) {
        int em = 0;                                                        // p = d_0 v
        if constexpr (CACHED) {
#pragma unroll
            for (int u = 0; u < LJ_PASS; ++u) {
                p[u] = a.dd[0] * w[u];
                em = max(em, exp_field(w[u]));
            }
        } else {
            for (int row = it.row0, j = it.j0; row < a.n; it.next(row, j)) {
                const double v = a.Wa[(size_t)row * a.ldw + j];
                a.Y[(size_t)row * a.ldy + j] = a.dd[0] * v;
                em = max(em, exp_field(v));
            }
        }
        em = __reduce_max_sync(0xffffffffu, em);
        if ((threadIdx.x & 31) == 0) atomicMax(a.em + (sub & 1), (unsigned)em);
        __syncthreads();
        if (threadIdx.x == 0) lj_arrive(a.cnt, 1);
        if (!lj_wait(a.cnt, ++b * gridDim.x, a.status, &s_word, stop)) return;
        const int e0 = (int)__ldcg(a.em + (sub & 1));
        // the other parity's word is read again only after the barriers of this substep
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicExch(a.em + ((sub + 1) & 1), 0u);
        const double* W = a.Wa;
        double* Wn = a.Wb;
        for (int k = 1; k < a.terms; ++k) {
            // val holds A^T / g, so w_{k+1} = val w_k - (c/g + x_k) w_k: one FP64
            // FMA per stored entry plus one
            const double beta = a.c * a.invg + a.xi[k - 1], dk = a.dd[k];
            float aw = 0.0f, ap = 0.0f;
            if constexpr (CACHED) {
#pragma unroll
                for (int u = 0; u < LJ_PASS; ++u) {
                    if (er[u] < 0) continue;
                    double wn = -beta * w[u];
#pragma unroll 4
                    for (int q = qb[u]; q < qe[u]; ++q)
                        wn = fma(s_val[q], __ldcg(W + (size_t)s_idx[q] * a.ldw + ej[u]), wn);
                    Wn[(size_t)er[u] * a.ldw + ej[u]] = wn;
                    w[u] = wn;
                    p[u] = fma(dk, wn, p[u]);
                    const float fw = mag(wn, e0), fp = mag(p[u], e0);
                    aw = fmaf(fw, fw, aw);
                    ap = fmaf(fp, fp, ap);
                }
            } else {
                for (int row = it.row0, j = it.j0; row < a.n; it.next(row, j)) {
                    double wn = -beta * __ldcg(W + (size_t)row * a.ldw + j);
                    for (int q = a.ptr[row]; q < a.ptr[row + 1]; ++q)
                        wn = fma(a.val[q], __ldcg(W + (size_t)a.idx[q] * a.ldw + j), wn);
                    Wn[(size_t)row * a.ldw + j] = wn;
                    const double pv = fma(dk, wn, a.Y[(size_t)row * a.ldy + j]);
                    a.Y[(size_t)row * a.ldy + j] = pv;
                    const float fw = mag(wn, e0), fp = mag(pv, e0);
                    aw = fmaf(fw, fw, aw);
                    ap = fmaf(fp, fp, ap);
                }
            }
            block_sum2(aw, ap, sh);
            ++b;
            if (threadIdx.x == 0) {
                __stcg(reinterpret_cast<float2*>(a.part + (size_t)(k & 1) * 2 * gridDim.x) + blockIdx.x,
                       make_float2(aw, ap));
                lj_arrive(a.cnt, 1);
            }
            if (!lj_wait(a.cnt, b * gridDim.x, a.status, &s_word, stop)) return;
            double* t = const_cast<double*>(W);
            W = Wn;
            Wn = t;
            if (stop == b) break;
        }
        // the next substep starts from v = scale p; the last one leaves Y = scale p
        const bool last = sub + 1 == a.substeps;
        if constexpr (CACHED) {
#pragma unroll
            for (int u = 0; u < LJ_PASS; ++u) {
                if (er[u] < 0) continue;
                w[u] = a.scale * p[u];
                if (last) a.Y[(size_t)er[u] * a.ldy + ej[u]] = w[u];
                else a.Wa[(size_t)er[u] * a.ldw + ej[u]] = w[u];
            }
        } else {
            for (int row = it.row0, j = it.j0; row < a.n; it.next(row, j)) {
                const double v = a.scale * a.Y[(size_t)row * a.ldy + j];
                if (last) a.Y[(size_t)row * a.ldy + j] = v;
                else a.Wa[(size_t)row * a.ldw + j] = v;
            }
        }
    }
}

// Y = alpha S X for a sparse S (CSR) and an n x r block X: one thread per entry.
__global__ void __launch_bounds__(256) spmm_kernel(const int* __restrict__ ptr, const int* __restrict__ idx,
                                                   const double* __restrict__ val, int n, int r,
                                                   const double* __restrict__ X, int ldx, double* __restrict__ Y,
                                                   int ldy, double alpha) {
    const size_t total = (size_t)n * r;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const int row = (int)(e / r), j = (int)(e % r);
        double y = 0.0;
        for (int q = ptr[row]; q < ptr[row + 1]; ++q) y = fma(val[q], X[(size_t)idx[q] * ldx + j], y);
        Y[(size_t)row * ldy + j] = alpha * y;
    }
}

}  // namespace

void launch_spmm(const int* ptr, const int* idx, const double* val, int n, int r, const double* X, int ldx, double* Y,
                 int ldy, double alpha, cudaStream_t st) {
    if (n <= 0 || r <= 0) return;
    const size_t total = (size_t)n * r;
    const int grid = (int)std::min<size_t>((total + 255) / 256, 152 * 32);
    spmm_kernel<<<grid, 256, 0, st>>>(ptr, idx, val, n, r, X, ldx, Y, ldy, alpha);
}

// Resident blocks per SM (at most eight) and the SM count.
static int leja_per_sm(bool cached) {
    static const int per[2] = {
        [] {
            int p = 0;
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p, leja_persistent_kernel<false>, LJ_THREADS, 0);
            return std::max(1, std::min(p, 8));
        }(),
        [] {
            int p = 0;
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p, leja_persistent_kernel<true>, LJ_THREADS, 0);
            return std::max(1, std::min(p, 8));
        }()};
    return per[cached];
}

static int leja_blocks(bool cached) {
    static const int sms = [] {
        int dev = 0, s = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&s, cudaDevAttrMultiProcessorCount, dev);
        return std::max(1, s);
    }();
    return std::max(2, sms * leja_per_sm(cached));
}

int leja_grid_max() { return std::max(leja_blocks(false), leja_blocks(true)); }

dme_status launch_leja_apply(const LejaCall& c, cudaStream_t st) {
    if (c.n <= 0 || c.r <= 0) return DME_OK;
    if (c.terms > 80 || c.terms < 1) return set_error("Leja apply: 1 <= terms <= 80"), DME_EINVAL;
    LejaArgs a;
    a.ptr = c.ptr;
    a.idx = c.idx;
    a.val = c.val;
    a.n = c.n;
    a.r = c.r;
    a.X = c.X;
    a.ldx = c.ldx;
    a.Y = c.Y;
    a.ldy = c.ldy;
    a.Wa = c.Wa;
    a.Wb = c.Wb;
    a.ldw = c.ldw;
    a.c = c.c;
    a.invg = c.invg;
    a.scale = c.scale;
    a.tol = c.tol;
    a.substeps = c.substeps;
    a.terms = c.terms;
    a.part = reinterpret_cast<float*>(c.part);
    a.cnt = reinterpret_cast<unsigned long long*>(c.bar);
    a.em = c.bar + 2;
    a.status = c.status;
    for (int i = 0; i < 80; ++i) {
        a.xi[i] = i < c.terms ? c.xi[i] : 0.0;
        a.dd[i] = i < c.terms ? c.dd[i] : 0.0;
    }
    const size_t total = (size_t)c.n * c.r, blocks = (total + LJ_THREADS - 1) / LJ_THREADS;
    // on chip if every thread has at most LJ_PASS entries and the rows that LJ_THREADS
    // consecutive entries can touch store few enough; any other block through global memory
    const long long rows = (LJ_THREADS - 1 + c.r - 1) / c.r + 1;
    const bool cached = blocks <= (size_t)LJ_PASS * (leja_blocks(true) - 1) &&
                        LJ_PASS * std::min<long long>(rows, c.n) * c.row_nnz <= LJ_NNZ;
    const int grid = (int)std::min<size_t>(blocks, (size_t)leja_blocks(cached) - 1) + 1;
    // the barrier counter reaches (barriers per launch) x grid: keep it below 2^31
    const long long per_sub = (long long)c.terms * grid;
    const int chunk = (int)std::max<long long>(1, std::min<long long>(c.substeps, (1ll << 31) / per_sub - 1));
    const void* kern = cached ? reinterpret_cast<const void*>(leja_persistent_kernel<true>)
                              : reinterpret_cast<const void*>(leja_persistent_kernel<false>);
    for (int done = 0; done < c.substeps; done += chunk) {
        a.substeps = std::min(chunk, c.substeps - done);
        if (done > 0) {            // continue from the previous launch's result
            a.X = c.Y;
            a.ldx = c.ldy;
        }
        DME_CUDA_TRY(cudaMemsetAsync(c.bar, 0, 4 * sizeof(unsigned), st));
        void* args[] = {&a};
        DME_TRY(coop_launch(kern, dim3(grid), dim3(LJ_THREADS), args, 0, st, leja_per_sm(cached)));
    }
    return DME_OK;
}

}  // namespace dme
