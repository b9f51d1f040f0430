// Kernels of the low-rank (LDL^T) path: the pivoted QLP factorisation of the
// compressions within a solve, a one-CTA parallel Jacobi eigensolver for the
// last one, the selections that build the compressed basis, the m x m root of
// the factored Riccati flow, and column scaling / copying helpers.
//
// The last compression needs the eigen-decomposition of an r x r Gram matrix
// (r <= 224), so one CTA holds its upper triangle packed in shared memory and
// applies r/2 disjoint rotations per sub-sweep (round-robin pairing); the
// eigenvector matrix is accumulated transposed (rows p, q of V^T change per
// rotation, so the updates are contiguous), in shared memory up to r = 112 and
// in global memory beyond.
#include "dme_internal.h"

#include <algorithm>
#include <cmath>

namespace dme {

namespace {

__device__ __forceinline__ int pk(int a, int b, int r) {   // packed upper triangle, a <= b
    return a * r - (a * (a - 1)) / 2 + (b - a);
}

template <typename T>
__device__ __forceinline__ T pget(const T* A, int x, int y, int r) {
    return x <= y ? A[pk(x, y, r)] : A[pk(y, x, r)];
}

template <typename T>
__device__ __forceinline__ void pset(T* A, int x, int y, int r, T v) {
    if (x <= y) A[pk(x, y, r)] = v;
    else A[pk(y, x, r)] = v;
}

// Round-robin pairing of R (even) indices in sub-sweep t: index 0 stays, the
// others rotate on a circle of R - 1 positions.
__device__ __forceinline__ void rr_pair(int i, int t, int R, int& p, int& q) {
    int a, b;
    if (i == 0) {
        a = 0;
        b = 1 + (t % (R - 1));
    } else {
        a = 1 + ((i + t) % (R - 1));
        b = 1 + ((R - 1 - i + t) % (R - 1));
    }
    p = min(a, b);
    q = max(a, b);
}

constexpr int kJacobiSweeps = 60;

// Symmetric eigen-decomposition of the r x r matrix G (only (G + G^T)/2 is
// used): lam[i] = eigenvalue i, row i of V^T (ldv) = its eigenvector.  A
// rotation is skipped when |a_pq| <= max(1e-14 sqrt(|a_pp a_qq|), 1e-15 max_i
// |a_ii|): what the compression drops with the off-diagonal part is then below
// 1e-14 of the kept terms (the factored path's bar is 1e-11), the FP64 pass
// after the single-precision one (off-diagonal about 1e-7) needs one rotating
// sweep instead of two, and rounding noise below the floor is not chased (a
// Gram matrix formed in floating point carries absolute errors of that size).  The sweeps stop after
// one with no rotation (DEV_NONFINITE in *status after 60 sweeps or on a
// non-finite entry).
// T: the arithmetic (float for a fast first pass, double for the result).
// VS: V^T is accumulated in shared memory too (r <= 112 for double) and copied
// out at the end; otherwise in global memory (Vt_out, double only).
template <typename T, bool VS>
__global__ void __launch_bounds__(1024) jacobi_eig_kernel(const double* __restrict__ G, int ldg, int r,
                                                          double* __restrict__ Vt_out, int ldv_out,
                                                          double* __restrict__ lam, int* status) {
    extern __shared__ __align__(16) unsigned char jsm[];
    const int R = r + (r & 1), P = R / 2;
    T* A = reinterpret_cast<T*>(jsm);
    T* cs = A + (size_t)r * (r + 1) / 2;
    T* sn = cs + P;
    T* tt = sn + P;
    T* Vt = VS ? tt + P : reinterpret_cast<T*>(Vt_out);
    const int ldv = VS ? r : ldv_out;
    constexpr T kRel = sizeof(T) == 4 ? T(1e-7) : T(1e-14);
    constexpr T kFloor = sizeof(T) == 4 ? T(1e-8) : T(1e-15);
    int* pp = reinterpret_cast<int*>(VS ? tt + P + (size_t)r * r : tt + P);
    int* qq = pp + P;
    // (i, j), i <= j, of every rotation block, packed as i << 8 | j (P <= 112)
    unsigned short* blk = reinterpret_cast<unsigned short*>(qq + P);
    const int nblk = P * (P + 1) / 2;
    __shared__ int rotated;
    __shared__ int bad;
    __shared__ T floor_abs;
    const int tid = threadIdx.x, nt = blockDim.x;
    if (tid == 0) bad = 0;
    for (int i = tid; i < P; i += nt) {
        const int base = i * P - i * (i - 1) / 2;      // blocks (i, i..P-1) start here
        for (int j = i; j < P; ++j) blk[base + j - i] = (unsigned short)((i << 8) | j);
    }
    for (int e = tid; e < r * r; e += nt) {
        const int i = e / r, j = e % r;
        if (i <= j) {
            const double v = 0.5 * (G[(size_t)i * ldg + j] + G[(size_t)j * ldg + i]);
            A[pk(i, j, r)] = (T)v;
            if (!isfinite(v)) bad = 1;
        }
        Vt[(size_t)i * ldv + j] = (i == j) ? T(1) : T(0);
    }
    __syncthreads();
    if (bad) {
        if (tid == 0) atomicOr(status, DEV_NONFINITE);
        return;
    }
    int sweep = 0;
    for (; sweep < kJacobiSweeps; ++sweep) {
        if (tid == 0) {
            rotated = 0;
            T dm = 0;
            for (int i = 0; i < r; ++i) dm = max(dm, abs(A[pk(i, i, r)]));
            floor_abs = kFloor * dm;
        }
        __syncthreads();
        for (int t = 0; t < R - 1; ++t) {
            for (int i = tid; i < P; i += nt) {
                int p, q;
                rr_pair(i, t, R, p, q);
                T c = 1, s = 0, tv = 0;
                if (q < r) {
                    const T apq = A[pk(p, q, r)];
                    const T app = A[pk(p, p, r)], aqq = A[pk(q, q, r)];
                    if (abs(apq) > max(kRel * sqrt(abs(app * aqq)), floor_abs)) {
                        const T th = (aqq - app) / (T(2) * apq);
                        tv = (th >= T(0) ? T(1) : T(-1)) / (abs(th) + sqrt(T(1) + th * th));
                        c = T(1) / sqrt(T(1) + tv * tv);
                        s = tv * c;
                        rotated = 1;
                    }
                }
                pp[i] = p;
                qq[i] = q;
                cs[i] = c;
                sn[i] = s;
                tt[i] = tv;
            }
            __syncthreads();
            // every 2 x 2 block between pairs i <= j: X <- J_i^T X J_j
            for (int e = tid; e < nblk; e += nt) {
                const int i = blk[e] >> 8, j = blk[e] & 0xFF;
                const int pi = pp[i], qi = qq[i], pj = pp[j], qj = qq[j];
                const T ci = cs[i], si = sn[i], cj = cs[j], sj = sn[j];
                if (si == T(0) && sj == T(0)) continue;
                if (i == j) {
                    if (qi >= r) continue;
                    const T apq = A[pk(pi, qi, r)];
                    A[pk(pi, pi, r)] -= tt[i] * apq;
                    A[pk(qi, qi, r)] += tt[i] * apq;
                    A[pk(pi, qi, r)] = T(0);
                    continue;
                }
                const bool qiok = qi < r, qjok = qj < r;
                const T x00 = pget(A, pi, pj, r);
                const T x01 = qjok ? pget(A, pi, qj, r) : T(0);
                const T x10 = qiok ? pget(A, qi, pj, r) : T(0);
                const T x11 = (qiok && qjok) ? pget(A, qi, qj, r) : T(0);
                const T y00 = ci * x00 - si * x10, y01 = ci * x01 - si * x11;
                const T y10 = si * x00 + ci * x10, y11 = si * x01 + ci * x11;
                pset(A, pi, pj, r, cj * y00 - sj * y01);
                if (qjok) pset(A, pi, qj, r, sj * y00 + cj * y01);
                if (qiok) pset(A, qi, pj, r, cj * y10 - sj * y11);
                if (qiok && qjok) pset(A, qi, qj, r, sj * y10 + cj * y11);
            }
            // V <- V J: rows p, q of V^T
            for (int e = tid; e < P * r; e += nt) {
                const int i = e / r, k = e % r;
                const T s = sn[i];
                if (s == T(0)) continue;
                const T c = cs[i];
                const int p = pp[i], q = qq[i];
                const T vp = Vt[(size_t)p * ldv + k], vq = Vt[(size_t)q * ldv + k];
                Vt[(size_t)p * ldv + k] = c * vp - s * vq;
                Vt[(size_t)q * ldv + k] = s * vp + c * vq;
            }
            __syncthreads();
        }
        const int any = rotated;
        __syncthreads();
        if (!any) break;
    }
    for (int i = tid; i < r; i += nt) lam[i] = (double)A[pk(i, i, r)];
    if (VS)
        for (int e = tid; e < r * r; e += nt) Vt_out[(size_t)(e / r) * ldv_out + e % r] = (double)Vt[e];
    if (tid == 0 && sweep == kJacobiSweeps && sizeof(T) == 8) atomicOr(status, DEV_NONFINITE);
}

// ---- pivoted QLP of the scaled Gram matrix (compressions between the first and the
// last of a solve).  With M = diag(d)^{1/2} G diag(d)^{1/2} = R^T R (pivoted Cholesky, R in
// the original column order, rank k0) and R R^T = T^T T (Cholesky), the rows of
// X = T^{-T} R are orthonormal, and the columns of Lt X^T (Lt Lt^T = P) have the squared
// norms of T's rows, which follow the eigenvalues of P (Stewart's pivoted QLP): the
// orthogonal change of columns leaves P alone, so dropping column j costs its squared
// norm, and what the pivoted Cholesky leaves out costs at most its last pivot per
// column.  Two r^3 / 3 factorisations replace the Jacobi sweeps (r = 57: 1.1 ms in
// 0.25 ms).  Both factorisations are one block (a chain of r pivots, FP64 issue of
// one SM): the packed upper triangle in shared memory.

//
// Per pivot the chain is scale, update, next pivot, each FP64 instruction of a lone warp
// about 65 cycles: warp 0 keeps the diagonal by itself and forms the next pivot and its
// reciprocal root while the others update the triangle (as one rank-one update between
// barriers, with the root and a divide in every warp: 82 and 60 us at r = 57 instead of
// 42 and 36, 122 and 86 at r = 100 instead of 69 and 42).

// The rank-one update of the strict triangle over positions [a0, m), by warps 1, 2, ...:
// rows q from the front and from the back are paired, so that a pair has m - a0 - 1
// entries and lanes idle only at its end.  col(a) is the column at position a.
template <class Col>
__device__ __forceinline__ void chol_update(double* A, const double* v, int a0, int m, int r, const Col& col) {
    const int lane = threadIdx.x & 31, w = m - a0;
    for (int q = (threadIdx.x >> 5) - 1; q < (w + 1) / 2; q += (blockDim.x >> 5) - 1) {
        const int back = w - 1 - q;
        const int i0 = col(a0 + q), i1 = col(a0 + back);
        const double v0 = v[i0], v1 = v[i1];
        const int len = back == q ? back : w - 1;
        for (int t = lane; t < len; t += 32) {
            const bool front = t < back;
            const int j = col(a0 + (front ? q + 1 + t : t + 1)), i = front ? i0 : i1;
            const int e = i <= j ? pk(i, j, r) : pk(j, i, r);
            A[e] = fma(front ? -v0 : -v1, v[j], A[e]);
        }
    }
}

// One warp: the position of the largest diagonal entry among col(0), ..., col(m - 1) to 20
// bits (lane l has seen l, l + 32, ...: `hi` the largest high word, `pos` its position).
__device__ __forceinline__ int chol_argmax(int hi, int pos) {
    const int top = __reduce_max_sync(0xffffffffu, hi);
    return __reduce_min_sync(0xffffffffu, hi == top ? pos : 0x7fffffff);
}

// The high word of x as an ordering key; negatives, infinities and NaN sort below zero.
__device__ __forceinline__ int chol_key(double x) {
    const int h = __double2hiint(x);
    return h < 0x7FF00000 ? h : -1;
}

__global__ void __launch_bounds__(512) chol_pivot_kernel(const double* __restrict__ G, int ldg, int r,
                                                         const double* __restrict__ d, double tol,
                                                         double* __restrict__ R, int ldr, int* __restrict__ k_out,
                                                         int* status) {
    extern __shared__ __align__(16) double csm[];
    double* A = csm;                                  // packed upper triangle (diagonal unused)
    double* v = A + (size_t)r * (r + 1) / 2;
    double* ds = v + r;                               // sqrt(d)
    double* dg = ds + r;                              // the diagonal
    int* idx = reinterpret_cast<int*>(dg + r);
    __shared__ int s_pos, bad;
    __shared__ double s_piv, s_rp;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    if (tid == 0) bad = 0;
    for (int i = tid; i < r; i += nt) {
        ds[i] = sqrt(d[i]);
        idx[i] = i;
    }
    __syncthreads();
    for (int e = tid; e < r * r; e += nt) {
        const int i = e / r, j = e % r;
        R[(size_t)i * ldr + j] = 0.0;
        if (i <= j) {
            const double g = 0.5 * (G[(size_t)i * ldg + j] + G[(size_t)j * ldg + i]) * (ds[i] * ds[j]);
            A[pk(i, j, r)] = g;
            if (i == j) dg[i] = g;
            if (!isfinite(g)) bad = 1;
        }
    }
    __syncthreads();
    if (bad) {
        if (tid == 0) {
            atomicOr(status, DEV_NONFINITE);
            *k_out = 0;
        }
        return;
    }
    int m = r, k = 0, pos = -1;
    double stop = 0.0;
    for (;; ++k) {
        // position pos (the last pivot) now holds the last column; idx[pos] itself is only
        // rewritten below, where nobody reads it
        const auto col = [&](int a) { return idx[a == pos ? m : a]; };
        if (tid < 32) {
            int hi = -1, at = 0;
            for (int a = lane; a < m; a += 32) {
                const int j = col(a);
                double x = dg[j];
                if (k > 0) {
                    x = fma(-v[j], v[j], x);
                    dg[j] = x;
                }
                if (chol_key(x) > hi) {
                    hi = chol_key(x);
                    at = a;
                }
            }
            at = chol_argmax(hi, at);
            __syncwarp();
            if (lane == 0) {
                double x = 0.0;
                if (m > 0 && at < m) {
                    x = dg[col(at)];
                    if (k > 0 && pos < m) idx[pos] = idx[m];
                }
                s_pos = at;
                s_piv = x;
                s_rp = x > 0.0 ? rsqrt(x) : 0.0;
            }
        } else if (k > 0) {
            chol_update(A, v, 0, m, r, col);
        }
        __syncthreads();
        const double piv = s_piv, rp = s_rp;
        if (k == 0) stop = tol * piv;
        if (m == 0 || !(piv > stop)) break;
        pos = s_pos;
        const int p = idx[pos];
        for (int a = tid; a < m; a += nt) {
            const int j = idx[a];
            const double x = (p == j ? dg[j] : A[p < j ? pk(p, j, r) : pk(j, p, r)]) * rp;
            v[j] = x;
            R[(size_t)k * ldr + j] = x;
        }
        --m;
        __syncthreads();
    }
    if (tid == 0) *k_out = k;
}

// T (upper, rows contiguous) with H = T^T T, rinv[j] = 1 / T[j][j], nrm[j] = the squared
// norm of row j; *k is lowered to the first pivot that is not positive.
__global__ void __launch_bounds__(512) chol_rows_kernel(const double* __restrict__ H, int ldh, int r, int* __restrict__ k,
                                                        double* __restrict__ T, int ldt, double* __restrict__ rinv,
                                                        double* __restrict__ nrm) {
    extern __shared__ __align__(16) double csm[];
    __shared__ double s_rp;
    const int n = min(*k, r);
    double* A = csm;                                  // packed upper triangle (diagonal unused)
    double* v = A + (size_t)r * (r + 1) / 2;
    double* dg = v + r;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    for (int e = tid; e < n * n; e += nt) {
        const int i = e / n, j = e % n;
        if (i <= j) A[pk(i, j, r)] = H[(size_t)i * ldh + j];
        if (i == j) dg[i] = H[(size_t)i * ldh + i];
    }
    __syncthreads();
    int j = 0;
    for (;; ++j) {
        if (tid < 32) {
            for (int a = j + lane; a < n; a += 32) {
                double x = dg[a];
                if (j > 0) {
                    x = fma(-v[a], v[a], x);
                    dg[a] = x;
                }
                if (a == j) s_rp = x > 0.0 ? rsqrt(x) : 0.0;
            }
        } else if (j > 0) {
            if (tid >= nt - 32) {                      // the last row's norm, beside the update
                double s = 0.0;
                for (int a = j - 1 + lane; a < n; a += 32) s = fma(v[a], v[a], s);
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
                if (lane == 0) nrm[j - 1] = s;
            }
            chol_update(A, v, j, n, r, [](int a) { return a; });
        }
        __syncthreads();
        if (j == n) break;
        const double rp = s_rp;
        if (!(rp > 0.0)) break;
        if (tid == 0) rinv[j] = rp;
        for (int a = j + tid; a < n; a += nt) {
            const double x = (a == j ? dg[a] : A[pk(j, a, r)]) * rp;
            v[a] = x;
            T[(size_t)j * ldt + a] = x;
        }
        __syncthreads();
    }
    if (tid == 0) *k = j;
}

// X = T^{-T} R, a warp per column, lane l holding the entries l, l + 32, ...; rows from *k
// on are zero.  The rows of T come in panels through shared memory: with a row loaded ahead
// from L2 each of the k dependent steps took that latency (32 us at r = 56, now 20).
constexpr int QS_ROWS = 16;
__global__ void __launch_bounds__(128) qlp_solve_kernel(const double* __restrict__ T, int ldt,
                                                        const double* __restrict__ rinv, const double* __restrict__ R,
                                                        int ldr, int r, const int* __restrict__ k, double* __restrict__ X,
                                                        int ldx) {
    constexpr int Q = LR_MAX_RANK / 32;
    __shared__ double Ts[QS_ROWS][LR_MAX_RANK], ri[QS_ROWS];
    const int c = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const bool on = c < r;
    const int n = *k;
    double b[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int i = lane + 32 * q;
        b[q] = on && i < n ? R[(size_t)i * ldr + c] : 0.0;
    }
#pragma unroll
    for (int qi = 0; qi < Q; ++qi)
        for (int half = 0; half < 2; ++half) {
            const int i0 = 32 * qi + QS_ROWS * half, rows = min(QS_ROWS, n - i0);
            if (rows <= 0) break;
            __syncthreads();
            double t[QS_ROWS / 4][Q];         // every load of the panel in flight at once
#pragma unroll
            for (int w = 0; w < QS_ROWS / 4; ++w)
#pragma unroll
                for (int q = qi; q < Q; ++q) {
                    const int i = (threadIdx.x >> 5) + 4 * w, kk = lane + 32 * q;
                    t[w][q] = i < rows && kk > i0 + i && kk < n ? T[(size_t)(i0 + i) * ldt + kk] : 0.0;
                }
#pragma unroll
            for (int w = 0; w < QS_ROWS / 4; ++w)
#pragma unroll
                for (int q = qi; q < Q; ++q) Ts[(threadIdx.x >> 5) + 4 * w][lane + 32 * q] = t[w][q];
            if (threadIdx.x < rows) ri[threadIdx.x] = rinv[i0 + threadIdx.x];
            __syncthreads();
            for (int i = 0; i < rows; ++i) {
                const int li = QS_ROWS * half + i;
                const double x = __shfl_sync(0xffffffffu, b[qi], li) * ri[i];
                if (lane == li) b[qi] = x;
                // zeros of Ts leave the entries up to i0 + i alone
#pragma unroll
                for (int q = qi; q < Q; ++q)
                    if (32 * q < n) {
                        const int kk = lane + 32 * q;
                        if (kk > i0 + i && kk < n) b[q] = fma(-Ts[i][kk], x, b[q]);
                    }
            }
        }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int i = lane + 32 * q;
        if (on && i < r) X[(size_t)i * ldx + c] = b[q];
    }
}

// Keep the rows j of X with nrm[j] > tol * max: To[a][rank] = X[j][a] sqrt(d[a]), d_out = 1,
// k_out their count (d_out may alias d).
__global__ void __launch_bounds__(1024) qlp_select_kernel(const double* __restrict__ X, int ldx,
                                                         const double* __restrict__ nrm, const int* __restrict__ k, int r,
                                                         double tol, const double* d, double* __restrict__ To, int ldt,
                                                         double* d_out, int* k_out) {
    __shared__ double rs[LR_MAX_RANK];
    __shared__ int rank[LR_MAX_RANK], kept;
    const int n = *k, tid = threadIdx.x, lane = tid & 31;
    if (tid < 32) {                       // the maximum, then the ranks, 32 rows at a time
        double m = 0.0;
        for (int j = lane; j < n; j += 32) m = fmax(m, nrm[j]);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, off));
        int c = 0;
        for (int j0 = 0; j0 < n; j0 += 32) {
            const int j = j0 + lane;
            const bool in = j < n && nrm[j] > tol * m;
            const unsigned set = __ballot_sync(0xffffffffu, in);
            if (j < n) rank[j] = in ? c + __popc(set & ((1u << lane) - 1)) : -1;
            c += __popc(set);
        }
        if (lane == 0) kept = c;
    } else {
        for (int a = tid - 32; a < r; a += blockDim.x - 32) rs[a] = sqrt(d[a]);
    }
    __syncthreads();
    for (int e = tid; e < n * r; e += blockDim.x) {
        const int j = e / r, a = e % r;
        if (rank[j] >= 0) To[(size_t)a * ldt + rank[j]] = X[(size_t)j * ldx + a] * rs[a];
    }
    for (int j = tid; j < kept; j += blockDim.x) d_out[j] = 1.0;
    if (tid == 0) *k_out = kept;
}

// Order the eigenvalues decreasingly and keep those above tol * max (max > 0):
// k_out = their count, d_out[rank] = lambda, T[a][rank] = V[a][i] * w with
// w = lambda^{-1/2} (inv_sqrt) or 1.  T has r rows (ldt).
__global__ void __launch_bounds__(256) select_kernel(const double* __restrict__ lam, const double* __restrict__ Vt,
                                                     int ldv, int r, double tol, int inv_sqrt, double* __restrict__ T,
                                                     int ldt, double* d_out, int* k_out, const double* rowscale) {
    __shared__ double smax;
    __shared__ int kcount;
    __shared__ double rs[LR_MAX_RANK];   // sqrt(rowscale), read before d_out (which may alias it) is written
    const int tid = threadIdx.x, nt = blockDim.x;
    for (int a = tid; a < r; a += nt) rs[a] = rowscale ? sqrt(rowscale[a]) : 1.0;
    if (tid == 0) {
        double m = 0.0;
        for (int i = 0; i < r; ++i) m = fmax(m, lam[i]);
        smax = m;
        kcount = 0;
    }
    __syncthreads();
    const double thr = tol * smax;
    for (int i = tid; i < r; i += nt) {
        const double li = lam[i];
        if (!(smax > 0.0) || !(li > thr)) continue;
        int rank = 0;
        for (int j = 0; j < r; ++j) {
            const double lj = lam[j];
            rank += (lj > li) || (lj == li && j < i);
        }
        atomicAdd(&kcount, 1);
        d_out[rank] = li;
        const double w = inv_sqrt ? 1.0 / sqrt(li) : 1.0;
        for (int a = 0; a < r; ++a) T[(size_t)a * ldt + rank] = Vt[(size_t)i * ldv + a] * w * rs[a];
    }
    __syncthreads();
    if (tid == 0) *k_out = kcount;
}

// Y = G F^T (r x m) with F = -t K^{-T} (K + I)^{-1}, K the Cholesky factor of
// I + t G^T G (m x m): (I + G F G^T)(I + G F G^T)^T = (I + t G G^T)^{-1} (Andrews' square
// root of the rank-m downdate).  One block: H = G^T G a warp per entry of its upper
// triangle, then the m x m part in one warp, Y by all threads.
__global__ void __launch_bounds__(256) ric_factor_kernel(const double* __restrict__ G, int r, int m, double t,
                                                         double* __restrict__ Y, int* status) {
    __shared__ double K[32][33], F[32][33];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int bad = 0;
    for (int e = warp; e < m * m; e += 8) {
        const int i = e / m, j = e % m;
        if (i > j) continue;
        double s = 0.0;
        for (int q = lane; q < r; q += 32) s = fma(G[(size_t)q * m + i], G[(size_t)q * m + j], s);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (!isfinite(s)) bad = 1;
        if (lane == 0) {
            const double v = (i == j ? 1.0 : 0.0) + t * s;
            K[i][j] = v;
            K[j][i] = v;
        }
    }
    if (__syncthreads_or(bad)) {
        if (tid == 0) atomicOr(status, DEV_NONFINITE);
        return;
    }
    if (warp == 0) {
        // Cholesky in place (lower): I + t G^T G is positive definite
        for (int j = 0; j < m; ++j) {
            double dj = K[j][j];
            for (int k = 0; k < j; ++k) dj -= K[j][k] * K[j][k];
            dj = sqrt(dj);
            __syncwarp();
            if (lane > j && lane < m) {
                double s = K[lane][j];
                for (int k = 0; k < j; ++k) s -= K[lane][k] * K[j][k];
                K[lane][j] = s / dj;
            }
            __syncwarp();
            if (lane == 0) K[j][j] = dj;
            __syncwarp();
        }
        // column `lane` of F: (K + I) x = e, then K^T y = x
        if (lane < m) {
            double x[32];
            for (int i = 0; i < m; ++i) {
                double s = i == lane ? 1.0 : 0.0;
                for (int k = 0; k < i; ++k) s -= K[i][k] * x[k];
                x[i] = s / (K[i][i] + 1.0);
            }
            for (int i = m - 1; i >= 0; --i) {
                double s = x[i];
                for (int k = i + 1; k < m; ++k) s -= K[k][i] * x[k];
                x[i] = s / K[i][i];
                F[i][lane] = -t * x[i];
            }
        }
    }
    __syncthreads();
    for (int e = tid; e < r * m; e += blockDim.x) {
        const int q = e / m, i = e % m;
        double s = 0.0;
        for (int k = 0; k < m; ++k) s = fma(G[(size_t)q * m + k], F[i][k], s);
        Y[(size_t)q * m + i] = s;
    }
}

// Y[i][j] = alpha * X[i][j] * (d ? sqrt(d[j]) : 1) for an n x k block.
// The entries (i, j) of an n x k block a thread visits in a grid-stride loop over
// e = i k + j, walked without a division per entry.
struct BlockEntries {
    int i0, j0, di, dj;
    __device__ BlockEntries(int k) {
        const size_t first = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
        const size_t stride = (size_t)gridDim.x * blockDim.x;
        i0 = (int)(first / k);
        j0 = (int)(first % k);
        di = (int)(stride / k);
        dj = (int)(stride % k);
    }
    __device__ __forceinline__ void next(int& i, int& j, int k) const {
        i += di;
        j += dj;
        if (j >= k) {
            j -= k;
            ++i;
        }
    }
};

// Y = alpha X diag(d)^{1/2} (d NULL: alpha X); the column scales are formed once
// per block (a square root per entry would be FP64-issue bound).
__global__ void __launch_bounds__(256) copy_cols_kernel(double* __restrict__ Y, int ldy, const double* __restrict__ X,
                                                        int ldx, int n, int k, double alpha,
                                                        const double* __restrict__ d) {
    __shared__ double sc[LR_MAX_RANK];
    const bool staged = k <= LR_MAX_RANK;
    if (staged)
        for (int j = threadIdx.x; j < k; j += blockDim.x) sc[j] = d ? alpha * sqrt(d[j]) : alpha;
    __syncthreads();
    const BlockEntries it(k);
    for (int i = it.i0, j = it.j0; i < n; it.next(i, j, k)) {
        const double s = staged ? sc[j] : (d ? alpha * sqrt(d[j]) : alpha);
        Y[(size_t)i * ldy + j] = s * X[(size_t)i * ldx + j];
    }
}

// G_ij *= sqrt(d_i d_j): the Gram matrix of L diag(d)^{1/2} from that of L.
__global__ void sym_scale_kernel(double* __restrict__ G, int ldg, int r, const double* __restrict__ d) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < r * r; e += gridDim.x * blockDim.x) {
        const int i = e / r, j = e % r;
        G[(size_t)i * ldg + j] *= sqrt(d[i]) * sqrt(d[j]);
    }
}

// C = alpha * sum_s W[s] (+ b1 D1), summed in s order; tri: C symmetric from the upper part.
__global__ void splitk_reduce_kernel(const double* __restrict__ Wk, int S, int M, int N, double* __restrict__ C,
                                     int ldc, double alpha, const double* __restrict__ D1, double b1, int tri) {
    const size_t total = (size_t)M * N;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(e / N), j = (int)(e % N);
        if (tri && i > j) continue;
        double acc = 0.0;
        for (int s = 0; s < S; ++s) acc += Wk[(size_t)s * total + e];
        double v = alpha * acc;
        if (D1) v += b1 * D1[(size_t)i * ldc + j];
        C[(size_t)i * ldc + j] = v;
        if (tri && i != j) C[(size_t)j * ldc + i] = v;
    }
}

// Partial products of X^T Y for tall X (K x M) and Y (K x N), M N <= 1024:
// block s sums the rows [s chunk, (s + 1) chunk).  The 256 threads form G =
// 256 / E groups (E = M N rounded up to a power of two, at least 32 so a group
// is whole warps, or 256 / 4 entries per thread when M N > 256); group g takes
// the rows k0 + g, k0 + g + G, ..., and the groups' sums are added in group
// order in shared memory.  part: [S][M][N].
__global__ void __launch_bounds__(256) tsgemm_kernel(const double* __restrict__ X, int ldx, int M,
                                                     const double* __restrict__ Y, int ldy, int N, int K, int chunk,
                                                     double* __restrict__ part, int sym) {
    __shared__ double red[1024];
    const int k0 = blockIdx.x * chunk, k1 = min(K, k0 + chunk);
    // sym (X = Y, M = N): only the M (M + 1) / 2 entries i <= j (half the FP64 FMAs)
    const int MN = sym ? M * (M + 1) / 2 : M * N;
    int E = 32;
    while (E < MN && E < 256) E <<= 1;
    const int per = (MN + 255) / 256;                 // entries per thread when E = 256
    const int G = 256 / E;
    const int g = threadIdx.x / E, t = threadIdx.x % E;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    int ea[4], eb[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int e = t + E * u;
        ea[u] = 0;
        eb[u] = 0;
        if (e < MN && !sym) {
            ea[u] = e / N;
            eb[u] = e % N;
        } else if (e < MN) {                          // e-th entry of the upper triangle, row by row
            int i = 0, rem = e;
            while (rem >= M - i) {
                rem -= M - i;
                ++i;
            }
            ea[u] = i;
            eb[u] = i + rem;
        }
    }
    for (int k = k0 + g; k < k1; k += G) {
        const double* xr = X + (size_t)k * ldx;
        const double* yr = Y + (size_t)k * ldy;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (u < per && t + E * u < MN) acc[u] = fma(xr[ea[u]], yr[eb[u]], acc[u]);
    }
    const size_t base = (size_t)blockIdx.x * M * N;   // part keeps the [M][N] layout (sym: i <= j written)
    if (G == 1) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int e = t + E * u;
            if (u < per && e < MN) part[base + (size_t)ea[u] * N + eb[u]] = acc[u];
        }
        return;
    }
    // G > 1: E <= 128, one entry per thread
    red[threadIdx.x] = acc[0];
    __syncthreads();
    if (g == 0 && t < MN) {
        double v = red[t];
        for (int q = 1; q < G; ++q) v += red[q * E + t];
        part[base + (size_t)ea[0] * N + eb[0]] = v;
    }
}

// C (n x N, ldc) = alpha X op(T) (+ beta D) for X n x K (ldx) and a small op(T)
// (K x N; T stored K x N, or N x K when tT, leading dimension ldt; K, N <= 64)
// staged in shared memory; one thread per output entry.
__global__ void __launch_bounds__(256) tall_small_kernel(const double* __restrict__ X, int ldx, int n, int K,
                                                         const double* __restrict__ Tm, int ldt, int tT, int N,
                                                         double* __restrict__ C, int ldc, double alpha,
                                                         const double* __restrict__ D, double beta) {
    __shared__ double sT[64 * 64];
    for (int e = threadIdx.x; e < K * N; e += blockDim.x) {
        const int k = e / N, j = e % N;
        sT[e] = tT ? Tm[(size_t)j * ldt + k] : Tm[(size_t)k * ldt + j];
    }
    __syncthreads();
    const BlockEntries it(N);
    for (int i = it.i0, j = it.j0; i < n; it.next(i, j, N)) {
        const double* xr = X + (size_t)i * ldx;
        double acc = 0.0;
        for (int k = 0; k < K; ++k) acc = fma(xr[k], sT[k * N + j], acc);
        double v = alpha * acc;
        if (D) v += beta * D[(size_t)i * ldc + j];
        C[(size_t)i * ldc + j] = v;
    }
}

__global__ void fill_kernel(double* __restrict__ x, int k, double v) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < k; i += gridDim.x * blockDim.x) x[i] = v;
}

int grid_of(size_t total) { return (int)std::min<size_t>((total + 255) / 256, 152 * 8); }

}  // namespace

constexpr int kJacobiSmemV = 112;    // largest r whose V^T also fits in shared memory (double)
constexpr int kJacobiF32Max = LR_JACOBI_F32_MAX;   // single-precision pass: V^T in shared memory

template <typename T>
static size_t jacobi_smem(int r, bool vs) {
    const int P = (r + (r & 1)) / 2;
    return sizeof(T) * ((size_t)r * (r + 1) / 2 + 3 * (size_t)P + (vs ? (size_t)r * r : 0)) +
           sizeof(int) * 2 * (size_t)P + sizeof(unsigned short) * (size_t)P * (P + 1) / 2;
}

size_t jacobi_smem_bytes(int r) { return jacobi_smem<double>(r, r <= kJacobiSmemV); }

dme_status launch_jacobi_eig(const double* G, int ldg, int r, double* Vt, int ldv, double* lam, int* status,
                             cudaStream_t st, bool fp32) {
    if (r < 1 || r > LR_MAX_RANK) return set_error("jacobi: size must be in [1, 224]"), DME_EINVAL;
    if (fp32 && r > kJacobiF32Max) return set_error("jacobi: the single-precision pass needs r <= 176"), DME_EINVAL;
    // shared-memory limits, set once (thread-safe static initialisation)
    static const cudaError_t attr = [] {
        cudaError_t e = cudaFuncSetAttribute(jacobi_eig_kernel<double, false>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)jacobi_smem<double>(LR_MAX_RANK, false));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(jacobi_eig_kernel<double, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)jacobi_smem<double>(kJacobiSmemV, true));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(jacobi_eig_kernel<float, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)jacobi_smem<float>(kJacobiF32Max, true));
        return e;
    }();
    DME_CUDA_TRY(attr);
    // enough threads for the P(P+1)/2 rotation blocks of a sub-sweep, no more (fewer warps
    // make the two barriers per sub-sweep cheaper)
    const int P = (r + 1) / 2;
    const int threads = std::min(1024, std::max(64, (P * (P + 1) / 2 + 31) / 32 * 32));
    if (fp32)
        jacobi_eig_kernel<float, true><<<1, threads, jacobi_smem<float>(r, true), st>>>(G, ldg, r, Vt, ldv, lam,
                                                                                     status);
    else if (r <= kJacobiSmemV)
        jacobi_eig_kernel<double, true><<<1, threads, jacobi_smem<double>(r, true), st>>>(G, ldg, r, Vt, ldv, lam,
                                                                                       status);
    else
        jacobi_eig_kernel<double, false><<<1, threads, jacobi_smem<double>(r, false), st>>>(G, ldg, r, Vt, ldv,
                                                                                         lam, status);
    DME_CUDA_TRY(cudaGetLastError());
    return DME_OK;
}

size_t chol_smem(int r) { return sizeof(double) * ((size_t)r * (r + 1) / 2 + 3 * (size_t)r) + sizeof(int) * (size_t)r; }

dme_status launch_chol_pivot(const double* G, int ldg, int r, const double* d, double tol, double* R, int ldr, int* k,
                             int* status, cudaStream_t st) {
    if (r < 1 || r > LR_MAX_RANK) return set_error("pivoted Cholesky: size must be in [1, 224]"), DME_EINVAL;
    static const cudaError_t attr = cudaFuncSetAttribute(
        chol_pivot_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)chol_smem(LR_MAX_RANK));
    DME_CUDA_TRY(attr);
    const int threads = r <= 32 ? 128 : (r <= 96 ? 256 : 512);
    chol_pivot_kernel<<<1, threads, chol_smem(r), st>>>(G, ldg, r, d, tol, R, ldr, k, status);
    DME_CUDA_TRY(cudaGetLastError());
    return DME_OK;
}

dme_status launch_qlp_rows(const double* H, int ldh, int r, const double* R, int ldr, int* k, double* T, int ldt,
                           double* rinv, double* nrm, double* X, int ldx, cudaStream_t st) {
    static const cudaError_t attr = cudaFuncSetAttribute(
        chol_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)chol_smem(LR_MAX_RANK));
    DME_CUDA_TRY(attr);
    const int threads = r <= 32 ? 128 : (r <= 96 ? 256 : 512);
    chol_rows_kernel<<<1, threads, chol_smem(r), st>>>(H, ldh, r, k, T, ldt, rinv, nrm);
    qlp_solve_kernel<<<(r + 3) / 4, 128, 0, st>>>(T, ldt, rinv, R, ldr, r, k, X, ldx);
    DME_CUDA_TRY(cudaGetLastError());
    return DME_OK;
}

void launch_qlp_select(const double* X, int ldx, const double* nrm, const int* k, int r, double tol, const double* d,
                       double* T, int ldt, double* d_out, int* k_out, cudaStream_t st) {
    qlp_select_kernel<<<1, 1024, 0, st>>>(X, ldx, nrm, k, r, tol, d, T, ldt, d_out, k_out);
}

void launch_lr_select(const double* lam, const double* Vt, int ldv, int r, double tol, int inv_sqrt, double* T,
                      int ldt, double* d_out, int* k_out, cudaStream_t st, const double* rowscale) {
    select_kernel<<<1, 256, 0, st>>>(lam, Vt, ldv, r, tol, inv_sqrt, T, ldt, d_out, k_out, rowscale);
}

void launch_sym_scale(double* G, int ldg, int r, const double* d, cudaStream_t st) {
    if (r <= 0) return;
    sym_scale_kernel<<<std::min(1024, (r * r + 255) / 256), 256, 0, st>>>(G, ldg, r, d);
}

void launch_ric_factor(const double* G, int r, int m, double t, double* Y, int* status, cudaStream_t st) {
    if (r <= 0 || m <= 0) return;
    ric_factor_kernel<<<1, 256, 0, st>>>(G, r, m, t, Y, status);
}

void launch_copy_cols(double* Y, int ldy, const double* X, int ldx, int n, int k, double alpha, const double* d,
                      cudaStream_t st) {
    if (n <= 0 || k <= 0) return;
    copy_cols_kernel<<<grid_of((size_t)n * k), 256, 0, st>>>(Y, ldy, X, ldx, n, k, alpha, d);
}

// Many partials of a small result: one block per entry, strided sums then a
// fixed tree (deterministic); same outputs as splitk_reduce_kernel.
__global__ void __launch_bounds__(256) splitk_reduce_wide_kernel(const double* __restrict__ Wk, int S, int M, int N,
                                                                 double* __restrict__ C, int ldc, double alpha,
                                                                 const double* __restrict__ D1, double b1, int tri) {
    __shared__ double red[256];
    const size_t total = (size_t)M * N;
    const int e = blockIdx.x;
    const int i = e / N, j = e % N;
    if (tri && i > j) return;
    double acc = 0.0;
    for (int s = threadIdx.x; s < S; s += 256) acc += Wk[(size_t)s * total + e];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        double v = alpha * red[0];
        if (D1) v += b1 * D1[(size_t)i * ldc + j];
        C[(size_t)i * ldc + j] = v;
        if (tri && i != j) C[(size_t)j * ldc + i] = v;
    }
}

void launch_splitk_reduce(const double* W, int S, int M, int N, double* C, int ldc, double alpha, const double* D1,
                          double b1, int tri, cudaStream_t st) {
    if (M <= 0 || N <= 0) return;
    if (S >= 64 && (size_t)M * N <= 4096) {
        splitk_reduce_wide_kernel<<<M * N, 256, 0, st>>>(W, S, M, N, C, ldc, alpha, D1, b1, tri);
        return;
    }
    splitk_reduce_kernel<<<grid_of((size_t)M * N), 256, 0, st>>>(W, S, M, N, C, ldc, alpha, D1, b1, tri);
}

void launch_tsgemm(const double* X, int ldx, int M, const double* Y, int ldy, int N, int K, int chunk, double* part,
                   cudaStream_t st, int sym) {
    const int S = (K + chunk - 1) / chunk;
    if (S <= 0 || M * N <= 0) return;
    tsgemm_kernel<<<S, 256, 0, st>>>(X, ldx, M, Y, ldy, N, K, chunk, part, sym && X == Y && ldx == ldy && M == N);
}

void launch_tall_small(const double* X, int ldx, int n, int K, const double* Tm, int ldt, int tT, int N, double* C,
                       int ldc, double alpha, const double* D, double beta, cudaStream_t st) {
    if (n <= 0 || N <= 0) return;
    const size_t total = (size_t)n * N;
    const int grid = (int)std::min<size_t>((total + 255) / 256, 152 * 16);
    tall_small_kernel<<<grid, 256, 0, st>>>(X, ldx, n, K, Tm, ldt, tT, N, C, ldc, alpha, D, beta);
}

void launch_fill(double* x, int k, double v, cudaStream_t st) {
    if (k <= 0) return;
    fill_kernel<<<grid_of((size_t)k), 256, 0, st>>>(x, k, v);
}

}  // namespace dme
