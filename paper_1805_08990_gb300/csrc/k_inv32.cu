// A single-precision approximate inverse, the preconditioner of the plan's refined solves.
//
// Gauss-Jordan inversion in blocks of 64: the diagonal block is inverted with partial
// pivoting inside it (in shared memory, by every block of the row panel for itself), the
// row panel becomes D^{-1} A_k., and every other block takes a rank-64 update.  There is no
// pivoting across blocks: an inverse that is not good enough shows in the refinement, which
// then gives way to the pivoted FP64 elimination.  Two launches per 64 columns against
// three per 16 there, and FP32 FMAs (128 per cycle and SM) instead of FP64 ones (two).
#include "dme_internal.h"

#include <algorithm>

namespace dme {

namespace {

constexpr int IB = 64;             // block size
constexpr int IW_LD = 68;          // row stride of a block in shared memory

// F (np x np) = X (n x n), the identity beyond it.
__global__ void __launch_bounds__(256) inv_load_kernel(const double* __restrict__ X, int n, float* __restrict__ F, int np) {
    const int i = blockIdx.x;
    for (int j = threadIdx.x; j < np; j += blockDim.x)
        F[(size_t)i * np + j] = (i < n && j < n) ? (float)X[(size_t)i * n + j] : (i == j ? 1.0f : 0.0f);
}

__global__ void __launch_bounds__(256) inv_store_kernel(const float* __restrict__ F, int np, double* __restrict__ X, int n) {
    const int i = blockIdx.x;
    for (int j = threadIdx.x; j < n; j += blockDim.x) X[(size_t)i * n + j] = (double)F[(size_t)i * np + j];
}

// out (64 x 64, 4 x 4 entries a thread) = P W.
__device__ __forceinline__ void mul64(const float* P, const float* W, float (&acc)[4][4]) {
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.0f;
#pragma unroll 8
    for (int k = 0; k < IB; ++k) {
        const float4 w = *reinterpret_cast<const float4*>(W + k * IW_LD + 4 * tx);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const float p = P[(4 * ty + a) * IW_LD + k];
            acc[a][0] = fmaf(p, w.x, acc[a][0]);
            acc[a][1] = fmaf(p, w.y, acc[a][1]);
            acc[a][2] = fmaf(p, w.z, acc[a][2]);
            acc[a][3] = fmaf(p, w.w, acc[a][3]);
        }
    }
}

// Block j of the row panel k: D = A_kk inverted in place by Gauss-Jordan elimination, then
// A_kj <- D^{-1} A_kj (Dinv for j = k); and the column panel's block j copied to Cb.
// A row's four threads hold 16 of its columns each in registers (16 steps unrolled: all 64
// would miss the instruction cache, 41 us a panel); a
// step publishes its column, finds the pivot among the rows not used yet (each warp for
// itself, one reduction of keys made of the magnitude and the row) and publishes the scaled
// pivot row: two barriers.  Rows are not exchanged: with pivot row pr[k] of column k the
// inverse's entry (k, pr[c]) ends in row pr[k], column c.  (As [D | I] in shared memory with
// three barriers a step: 100 us a panel.)
__global__ void __launch_bounds__(256) inv_panel_kernel(float* __restrict__ A, int np, int k0, float* __restrict__ Dinv,
                                                        float* __restrict__ Cb) {
    __shared__ __align__(16) float D[IB * IW_LD], W[IB * IW_LD];
    __shared__ __align__(16) float scol[2][IB], sprow[2][IB];
    __shared__ int pr[IB], kinv[IB];
    const int tid = threadIdx.x, lane = tid & 31;
    const int j0 = blockIdx.x * IB;
    const int r = tid >> 2, q = tid & 3;
    float a[16];
#pragma unroll
    for (int i = 0; i < 16; i += 4) {
        const float4 v = *reinterpret_cast<const float4*>(A + (size_t)(k0 + r) * np + k0 + 16 * q + i);
        a[i] = v.x;
        a[i + 1] = v.y;
        a[i + 2] = v.z;
        a[i + 3] = v.w;
    }
    for (int e = tid; e < IB * IB; e += 256) {
        const int rr = e / IB, c = e % IB;
        W[rr * IW_LD + c] = A[(size_t)(k0 + rr) * np + j0 + c];
        if (j0 != k0) Cb[(size_t)(j0 + rr) * IB + c] = A[(size_t)(j0 + rr) * np + k0 + c];
    }
    unsigned used0 = 0, used1 = 0;                    // rows 0 .. 31, 32 .. 63
#pragma unroll 1
    for (int kq = 0; kq < 4; ++kq)
#pragma unroll
    for (int ki = 0; ki < 16; ++ki) {
        const int k = 16 * kq + ki, b = ki & 1;
        if (q == kq) scol[b][r] = a[ki];
        __syncthreads();
        const unsigned v0 = __float_as_uint(scol[b][lane]) & 0x7FFFFFC0u;
        const unsigned v1 = __float_as_uint(scol[b][lane + 32]) & 0x7FFFFFC0u;
        const unsigned key0 = ((used0 >> lane) & 1) ? 0u : (v0 | (63u - lane));
        const unsigned key1 = ((used1 >> lane) & 1) ? 0u : (v1 | (31u - lane));
        const int p = 63 - (int)(__reduce_max_sync(0xffffffffu, max(key0, key1)) & 63u);
        if (p < 32) used0 |= 1u << p;
        else used1 |= 1u << (p - 32);
        const float rp = 1.0f / scol[b][p];
        if (r == p) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                a[i] *= rp;
                if (q == kq && i == ki) a[i] = rp;
            }
#pragma unroll
            for (int i = 0; i < 16; i += 4)
                *reinterpret_cast<float4*>(&sprow[b][16 * q + i]) = make_float4(a[i], a[i + 1], a[i + 2], a[i + 3]);
            if (q == 0) {
                pr[k] = p;
                kinv[p] = k;
            }
        }
        __syncthreads();
        if (r != p) {
            const float f = scol[b][r];
            if (q == kq) a[ki] = 0.0f;
#pragma unroll
            for (int i = 0; i < 16; i += 4) {
                const float4 v = *reinterpret_cast<const float4*>(&sprow[b][16 * q + i]);
                a[i] = fmaf(-f, v.x, a[i]);
                a[i + 1] = fmaf(-f, v.y, a[i + 1]);
                a[i + 2] = fmaf(-f, v.z, a[i + 2]);
                a[i + 3] = fmaf(-f, v.w, a[i + 3]);
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 16; ++i) D[kinv[r] * IW_LD + pr[16 * q + i]] = a[i];
    __syncthreads();
    const int tx = tid & 15, ty = tid >> 4;
    if (j0 == k0) {
        for (int e = tid; e < IB * IB; e += 256) Dinv[e] = D[(e / IB) * IW_LD + e % IB];
        return;
    }
    float acc[4][4];
    mul64(D, W, acc);
#pragma unroll
    for (int u = 0; u < 4; ++u)
        *reinterpret_cast<float4*>(A + (size_t)(k0 + 4 * ty + u) * np + j0 + 4 * tx) =
            make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]);
}

// Blocks (i, j): A_ij -= C_i A_kj; A_ik = -C_i Dinv; A_kk = Dinv; the row panel stays.
__global__ void __launch_bounds__(256) inv_update_kernel(float* __restrict__ A, int np, int k0,
                                                         const float* __restrict__ Dinv, const float* __restrict__ Cb) {
    __shared__ __align__(16) float P[IB * IW_LD], W[IB * IW_LD];
    const int i0 = blockIdx.y * IB, j0 = blockIdx.x * IB;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    if (i0 == k0) {
        if (j0 == k0)
            for (int e = tid; e < IB * IB; e += 256) A[(size_t)(k0 + e / IB) * np + k0 + e % IB] = Dinv[e];
        return;
    }
    for (int e = tid; e < IB * IB; e += 256) {
        const int r = e / IB, c = e % IB;
        P[r * IW_LD + c] = Cb[(size_t)(i0 + r) * IB + c];
        W[r * IW_LD + c] = j0 == k0 ? Dinv[e] : A[(size_t)(k0 + r) * np + j0 + c];
    }
    __syncthreads();
    float acc[4][4];
    mul64(P, W, acc);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        float4* o = reinterpret_cast<float4*>(A + (size_t)(i0 + 4 * ty + a) * np + j0 + 4 * tx);
        float4 v = j0 == k0 ? make_float4(0.f, 0.f, 0.f, 0.f) : *o;
        v.x -= acc[a][0];
        v.y -= acc[a][1];
        v.z -= acc[a][2];
        v.w -= acc[a][3];
        *o = v;
    }
}

// X += C; per-block partial sums of C^2 and X^2 (fixed order; summed by refine_final_kernel).
__global__ void __launch_bounds__(256) refine_update_kernel(double* __restrict__ X, const double* __restrict__ C, size_t len,
                                                            double* __restrict__ part) {
    __shared__ double sc[8], sx[8];
    double c2 = 0.0, x2 = 0.0;
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < len; e += (size_t)gridDim.x * blockDim.x) {
        const double c = C[e], x = X[e] + c;
        X[e] = x;
        c2 = fma(c, c, c2);
        x2 = fma(x, x, x2);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        c2 += __shfl_xor_sync(0xffffffffu, c2, off);
        x2 += __shfl_xor_sync(0xffffffffu, x2, off);
    }
    if ((threadIdx.x & 31) == 0) {
        sc[threadIdx.x >> 5] = c2;
        sx[threadIdx.x >> 5] = x2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) {
            c2 += sc[w];
            x2 += sx[w];
        }
        part[2 * blockIdx.x] = c2;
        part[2 * blockIdx.x + 1] = x2;
    }
}

__global__ void refine_final_kernel(const double* __restrict__ part, int nb, double* __restrict__ out) {
    double c2 = 0.0, x2 = 0.0;
    for (int k = threadIdx.x; k < nb; k += 32) {
        c2 += part[2 * k];
        x2 += part[2 * k + 1];
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        c2 += __shfl_xor_sync(0xffffffffu, c2, off);
        x2 += __shfl_xor_sync(0xffffffffu, x2, off);
    }
    if (threadIdx.x == 0) {
        out[0] = c2;
        out[1] = x2;
    }
}

constexpr int kRefineBlocks = 608;

}  // namespace

int inv32_pad(int n) { return (n + IB - 1) / IB * IB; }
size_t inv32_floats(int n) { return (size_t)inv32_pad(n) * inv32_pad(n); }
size_t inv32_work_floats(int n) { return (size_t)inv32_pad(n) * IB + IB * IB; }

dme_status launch_inv32(const double* X, int n, double* Y, float* F, float* work, cudaStream_t st) {
    const int np = inv32_pad(n), nb = np / IB;
    float* Cb = work;
    float* Dinv = work + (size_t)np * IB;
    inv_load_kernel<<<np, 256, 0, st>>>(X, n, F, np);
    for (int k = 0; k < nb; ++k) {
        inv_panel_kernel<<<nb, 256, 0, st>>>(F, np, k * IB, Dinv, Cb);
        inv_update_kernel<<<dim3(nb, nb), 256, 0, st>>>(F, np, k * IB, Dinv, Cb);
    }
    inv_store_kernel<<<n, 256, 0, st>>>(F, np, Y, n);
    DME_CUDA_TRY(cudaGetLastError());
    return DME_OK;
}

size_t refine_work_doubles() { return 2 * (size_t)kRefineBlocks + 2; }

void launch_refine_update(double* X, const double* C, size_t len, double* work, cudaStream_t st) {
    refine_update_kernel<<<kRefineBlocks, 256, 0, st>>>(X, C, len, work + 2);
    refine_final_kernel<<<1, 32, 0, st>>>(work + 2, kRefineBlocks, work);
}

}  // namespace dme
