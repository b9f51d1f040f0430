// The FP64 tile product shared by the grouped FP64 GEMM and the residue products'
// native recomputation.
#pragma once

#include "dme_internal.h"

namespace dme {

// One BM x BM output tile (BM = 32 or 64) with 256 threads, each holding a
// TM x TM register tile (TM = BM / 16).  Every output is accumulated over k in
// increasing order with fma, whatever BM is; gemm64_accum covers [kbeg, kend).
template <int BM>
__device__ __forceinline__ void gemm64_accum(const GemmProb& pb, int row0, int col0, int kbeg, int kend,
                                             double (&As)[G64_BK][BM + 1], double (&Bs)[G64_BK][BM + 1],
                                             double (&acc)[BM / 16][BM / 16]) {
    constexpr int TM = BM / 16;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TM; ++j) acc[i][j] = 0.0;

    for (int k0 = kbeg; k0 < kend; k0 += G64_BK) {
#pragma unroll
        for (int q = 0; q < TM; ++q) {
            const int e = tid + 256 * q;     // BM x 16 elements of each operand tile
            int r, k;
            double v = 0.0;
            if (!pb.transA) {
                r = e >> 4;
                k = e & 15;
                int gr = row0 + r, gk = k0 + k;
                if (gr < pb.M && gk < kend) v = pb.A[(size_t)gr * pb.lda + gk];
            } else {
                r = e % BM;
                k = e / BM;
                int gr = row0 + r, gk = k0 + k;
                if (gr < pb.M && gk < kend) v = pb.A[(size_t)gk * pb.lda + gr];
            }
            As[k][r] = v;
            int c;
            double w = 0.0;
            if (!pb.transB) {
                c = e % BM;
                k = e / BM;
                int gc = col0 + c, gk = k0 + k;
                if (gc < pb.N && gk < kend) w = pb.B[(size_t)gk * pb.ldb + gc];
            } else {
                c = e >> 4;
                k = e & 15;
                int gc = col0 + c, gk = k0 + k;
                if (gc < pb.N && gk < kend) w = pb.B[(size_t)gc * pb.ldb + gk];
            }
            Bs[k][c] = w;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < G64_BK; ++k) {
            double a[TM], b[TM];
#pragma unroll
            for (int i = 0; i < TM; ++i) a[i] = As[k][ty + 16 * i];
#pragma unroll
            for (int j = 0; j < TM; ++j) b[j] = Bs[k][tx + 16 * j];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TM; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
}

// C = alpha acc + b1 D1 + b2 D2 + b3 D3 (a triangle problem writes (r, c), r <= c,
// and its mirror).
__device__ __forceinline__ void gemm64_out(const GemmProb& pb, int r, int c, double sum) {
    const size_t off = (size_t)r * pb.ldd + c;
    double v = pb.alpha * sum;
    if (pb.D1) v += pb.b1 * pb.D1[off];
    if (pb.D2) v += pb.b2 * pb.D2[off];
    if (pb.D3) v += pb.b3 * pb.D3[off];
    pb.C[(size_t)r * pb.ldc + c] = v;
    if (pb.tri && r != c) pb.C[(size_t)c * pb.ldc + r] = v;
}

}  // namespace dme
