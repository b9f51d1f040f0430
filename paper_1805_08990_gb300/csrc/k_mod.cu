// FP64 products A B^T as exact residue products on tcgen05 tensor cores.
//
// GB300 runs FP64 FMAs at 1.25 TFLOP/s for the whole chip and bf16 MMAs at about
// 1900, so an FP64 product is computed in whole numbers instead (after Ozaki,
// Uchino & Imamura, "Ozaki scheme II", 2025: a product of integer matrices from its
// residues modulo pairwise coprime numbers and the Chinese remainder theorem):
//  1. convert: row i of each operand becomes integers rint(x 2^sigma_i), sigma_i such
//     that the row's 2-norm is at most 2^61 (Cauchy-Schwarz: every output is below
//     2^122 in magnitude), and the integers their residues modulo the 16 moduli below
//     (product 2^125.3), centred, each exact in bf16.
//  2. multiply: per modulus one bf16 product with fp32 accumulation; |residue| <= 128
//     and K <= 1024 per pass keep every partial sum at most 2^24, so it is exact in
//     any order; the epilogue reduces it and stores one byte per output.
//  3. combine: x = sum_m y_m w_m mod P in 128-bit integers, rounded to double once,
//     scaled by 2^(-sigma_i - sigma_j), then the addends of the product.
// The only errors are the operands' rounding in step 1 (2^-59 of the row's largest
// entry or less at K = 1024, where a double has 2^-53) and the final rounding.
//
// Certificate.  An FP64 dot product of length K has the a-priori error bound
// K u S, S = sum_k |a_k b_k|, u = 2^-53.  A row's rounding error is absolute (one
// scale per row), so an output whose products are all far below the row's largest
// entries could have a larger one.  A seventeenth plane holds |x| / 2^E rounded
// down to bf16; its product is a lower estimate of S, and an output is accepted only
// when (rho_a |b|_1 + rho_b |a|_1) <= K u S, i.e. when its error bound is no larger
// than the FP64 sum's own.  The others (and all of a row with a non-finite entry or
// an exponent outside +-400) are recomputed in FP64 from the operands by the same
// blocks that combine.
//
// Bound: tensor pipe for n >= 1024 (17 bf16 products), launch latency below.
#include "mod_internal.h"
#include "split_internal.h"
#include "tc_ptx.cuh"

#include <cudaTypedefs.h>

#include <algorithm>
#include <string>

namespace dme {

using namespace tc;

namespace {

using u128 = unsigned __int128;

// ------------------------------------------------------------------ constants
constexpr int MOD_NORM = 61;                  // log2 of a row's largest 2-norm in integer units
constexpr int MOD_MAX_EXP = 400;              // rows with larger exponents (of either sign) go to FP64
constexpr int MOD_CHUNK = 1024;               // K per exact fp32 sum

constexpr u128 mod_product() {
    u128 p = 1;
    for (int m = 0; m < MOD_NM; ++m) p *= (u128)kModuli[m];
    return p;
}

constexpr int centred(int r, int p) { return r > p / 2 ? r - p : r; }

struct ModConst {
    float p[MOD_NM], inv[MOD_NM];
    float c1[MOD_NM], c2[MOD_NM], c3[MOD_NM];     // 2^16, 2^32, 2^48 mod p, centred
    uint32_t w0[MOD_NM], w1[MOD_NM], w2[MOD_NM];  // (P / p) inverse(P / p) mod P, without its low 32 bits
    uint32_t o0, o1, o2;                          // -128 sum_m w_m mod P (bytes hold residue + 128)
    uint64_t plo;                                 // P without its low 32 bits
    uint32_t phi;
    float qscale;                                 // 2^(64 + 10) / (P / 2^32)
};

constexpr ModConst make_mod_const() {
    ModConst c{};
    const u128 P = mod_product();
    for (int m = 0; m < MOD_NM; ++m) {
        const int p = kModuli[m];
        c.p[m] = (float)p;
        c.inv[m] = 1.0f / (float)p;
        const long s = 65536 % p;
        c.c1[m] = (float)centred((int)s, p);
        c.c2[m] = (float)centred((int)(s * s % p), p);
        c.c3[m] = (float)centred((int)(s * s % p * s % p), p);
        const u128 M = P / (u128)p;
        const int r = (int)(M % (u128)p);
        int inv = 1;
        while (r * inv % p != 1) ++inv;
        const u128 w = (M * (u128)inv) % P;       // M inv < 2^125
        const u128 h = (w + ((u128)1 << 31)) >> 32;
        c.w0[m] = (uint32_t)h;
        c.w1[m] = (uint32_t)(h >> 32);
        c.w2[m] = (uint32_t)(h >> 64);
    }
    const u128 ph = (P + ((u128)1 << 31)) >> 32;
    u128 sw = 0;
    for (int m = 0; m < MOD_NM; ++m) sw += ((u128)c.w2[m] << 64) + ((u128)c.w1[m] << 32) + (u128)c.w0[m];
    const u128 o = ph - (sw * 128) % ph;
    c.o0 = (uint32_t)o;
    c.o1 = (uint32_t)(o >> 32);
    c.o2 = (uint32_t)(o >> 64);
    c.plo = (uint64_t)ph;
    c.phi = (uint32_t)(ph >> 64);
    c.qscale = (float)(18889465931478580854784.0 / ((double)c.phi * 18446744073709551616.0 + (double)c.plo));
    return c;
}

__constant__ ModConst c_mod = make_mod_const();
static_assert(mod_product() >> 125 != 0 && mod_product() >> 126 == 0, "2^122 < P / 8: the quotient is never ambiguous");

// The bytes of an odd modulus hold every residue that mod_centred returns: p (1/2 + 2^-8) < 128.
constexpr bool mod_residues_fit() {
    for (int m = 1; m < MOD_NM; ++m)
        if (kModuli[m] * 129 >= 128 * 256) return false;
    return kModuli[0] == 256;
}
static_assert(mod_residues_fit(), "a residue of 128 is only legitimate modulo 256");

// ------------------------------------------------------------------ 1. convert
// |x| / 2^E as a float rounded towards zero (20 mantissa bits), from the bits of x.
__device__ __forceinline__ float mag_scaled(unsigned long long b, int E) {
    const int ex = (int)((b >> 52) & 0x7FF) - 1023 - E;       // |x| / 2^E in [2^ex, 2^(ex+1)), ex <= -1
    // entries below 2^-60 of the row's largest (subnormal ones always are: E >= -399) are raised
    // to it: far too small to pass the certificate, and a product of nonzero entries stays
    // distinguishable from zero
    if (ex < -60) return (b << 1) ? __int_as_float((127 - 60) << 23) : 0.0f;
    return __int_as_float(((ex + 127) << 23) | (int)((b >> 29) & 0x7FFFFF));
}

// rint(x 2^sigma) for |x 2^sigma| < 2^62
__device__ __forceinline__ long long to_int(unsigned long long b, int sigma) {
    const int ex = (int)((b >> 52) & 0x7FF);
    if (ex == 0) return 0;
    const unsigned long long m = (b & ((1ull << 52) - 1)) | (1ull << 52);
    const int s = ex - 1075 + sigma;
    unsigned long long v;
    if (s >= 0) v = m << s;
    else if (s < -54) v = 0;
    else v = (m + (1ull << (-s - 1))) >> (-s);
    return (b >> 63) ? -(long long)v : (long long)v;
}

// The centred residues of four integers, one 8-byte store of bf16 per plane: the
// integers as balanced 16-bit limbs l, x = l0 + l1 c1 + l2 c2 + l3 c3 exactly in fp32
// (below 2^24 in magnitude), then x - p rint(x / p).
__device__ __forceinline__ void store_residues4(const long long (&V)[4], __nv_bfloat16* __restrict__ out,
                                                size_t plane) {
    float l[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        long long v = V[u];
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            const int d = (int)(short)(v & 0xFFFF);
            l[u][t] = (float)d;
            v = (v - d) >> 16;
        }
        l[u][3] = (float)(int)v;
    }
#pragma unroll
    for (int m = 0; m < MOD_NM; ++m) {
        uint32_t r[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float x = fmaf(l[u][3], c_mod.c3[m], fmaf(l[u][2], c_mod.c2[m], fmaf(l[u][1], c_mod.c1[m], l[u][0])));
            const float q = fmaf(x, c_mod.inv[m], 12582912.0f) - 12582912.0f;
            r[u] = __float_as_uint(fmaf(-q, c_mod.p[m], x));       // an integer of at most 8 bits: exact in bf16
        }
        uint2 w;
        w.x = __byte_perm(r[0], r[1], 0x7632);
        w.y = __byte_perm(r[2], r[3], 0x7632);
        *reinterpret_cast<uint2*>(out + m * plane) = w;
    }
}

__device__ __forceinline__ void load4_bits(const double* __restrict__ row, int k, int cols, bool vec,
                                           unsigned long long (&b)[4]) {
    if (vec && k + 3 < cols) {
        const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(row + k);
        const ulonglong2 c = *reinterpret_cast<const ulonglong2*>(row + k + 2);
        b[0] = a.x;
        b[1] = a.y;
        b[2] = c.x;
        b[3] = c.y;
    } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) b[u] = k + u < cols ? (unsigned long long)__double_as_longlong(row[k + u]) : 0ull;
    }
}

// One block of T threads per row, four consecutive entries per thread and step: pass 1
// the largest exponent, pass 2 the norms, pass 3 the residues.  Rows of up to 4 T
// entries stay in registers; longer ones are read again (from L1 / L2).
// Bound: the planes' writes (34 bytes per entry against 8 read).
template <int T>
__global__ void __launch_bounds__(T) mod_convert_kernel(const double* __restrict__ X, int cols, int ld,
                                                        __nv_bfloat16* __restrict__ out, int Kp,
                                                        ModRow* __restrict__ info, int prow) {
    __shared__ int s_e[T / 32];
    __shared__ float s_q[T / 32], s_a[T / 32];
    const int row = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double* x = X + (size_t)row * ld;
    const bool vec = (ld % 2) == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    constexpr int NW = T / 32;
    unsigned long long b[4];
    int emax = -100000;
    for (int k = 4 * tid; k < cols; k += 4 * T) {
        load4_bits(x, k, cols, vec, b);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (b[u] << 1) emax = max(emax, (int)((b[u] >> 52) & 0x7FF) - 1023);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, off));
    if (lane == 0) s_e[warp] = emax;
    __syncthreads();
    emax = s_e[0];
#pragma unroll
    for (int w = 1; w < NW; ++w) emax = max(emax, s_e[w]);
    const bool zero = emax == -100000;
    const bool bad = !zero && (emax > MOD_MAX_EXP || emax < -MOD_MAX_EXP);   // NaN, infinity: emax = 1024
    const int E = emax + 1;
    float sq = 0.0f, sa = 0.0f;
    if (!zero && !bad) {
        for (int k = 4 * tid; k < cols; k += 4 * T) {
            if (cols > 4 * T) load4_bits(x, k, cols, vec, b);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float f = mag_scaled(b[u], E);
                sq = fmaf(f, f, sq);
                sa += f;
            }
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        sq += __shfl_xor_sync(0xffffffffu, sq, off);
        sa += __shfl_xor_sync(0xffffffffu, sa, off);
    }
    if (lane == 0) {
        s_q[warp] = sq;
        s_a[warp] = sa;
    }
    __syncthreads();
    sq = s_q[0];
    sa = s_a[0];
#pragma unroll
    for (int w = 1; w < NW; ++w) {
        sq += s_q[w];
        sa += s_a[w];
    }
    // sums of at most 2^14 floats of relative error 2^-20: 1 + 2^-7 covers them
    sq *= 1.0078125f;
    sa *= 1.0078125f;
    // L: the smallest integer with 2-norm <= 2^L (in units of 2^E), i.e. 4^L >= sq
    int L = 0;
    if (sq > 1.0f) L = ((int)((__float_as_uint(sq) >> 23) & 0xFF) - 127 + 2) >> 1;   // sq < 2^(e+1) <= 4^L
    const int sigma = zero || bad ? 0 : MOD_NORM - E - L;
    if (tid == 0) {
        ModRow r;
        r.sigma = sigma;
        r.rho = zero ? 0.0f : __int_as_float((127 - (MOD_NORM + 1 - L)) << 23);      // half a unit 2^-sigma over 2^E
        r.n1 = bad ? __int_as_float(0x7f800000) : sa;
        r.pad = 0;
        info[row] = r;
    }
    const size_t plane = (size_t)prow * Kp, kblock = (size_t)prow * MOD_BK;
    for (int k = 4 * tid; k < Kp; k += 4 * T) {
        __nv_bfloat16* o = out + (k / MOD_BK) * kblock + (size_t)row * MOD_BK + k % MOD_BK;
        long long V[4] = {0, 0, 0, 0};
        uint32_t f[4] = {0, 0, 0, 0};
        if (!zero && !bad && k < cols) {
            if (cols > 4 * T) load4_bits(x, k, cols, vec, b);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                V[u] = to_int(b[u], sigma);
                f[u] = __float_as_uint(mag_scaled(b[u], E));
            }
        }
        store_residues4(V, o, plane);
        uint2 w;
        w.x = __byte_perm(f[0], f[1], 0x7632);                 // truncated to bf16
        w.y = __byte_perm(f[2], f[3], 0x7632);
        *reinterpret_cast<uint2*>(o + MOD_NM * plane) = w;
    }
}

// ------------------------------------------------------------------ 2. multiply
constexpr int MG_BM = 128;
constexpr uint64_t MG_TIMEOUT_NS = 2000000000ull;

struct ModGemmArgs {
    int M, N, Kp;
    int tri;
    int tiles_m, tiles_n, tiles, units;
    uint8_t* R;
    size_t plane;             // bytes per residue plane of the output
    int ldr;
    const ModRow* ra;
    const ModRow* rb;
    float kfac;               // 2^53 / K
    int* status;
};

// PAIR: two CTAs work on a 256 x 256 tile (tcgen05 cta_group::2: each loads its 128 rows of
// A and 128 of B, and holds its 128 rows of the result).  One plane pair gives one MMA per
// K step, so what a stage of shared memory is good for decides: 32 KB buy 256 cycles of
// MMA in a 128 x 128 tile, 512 in a pair's, and loads came back 3900 cycles after they were
// issued at K = 2048 (six stages of the former: 690 cycles per K block; 128 x 256 tiles in
// clusters of four with a multicast B, four stages of 48 KB: 970 per 512 of MMA; pairs,
// seven stages: 860 with the MMAs issued by one diverged lane, 700 from uniform registers, where
// cuBLAS runs at 640).
template <int BN_, bool PAIR_>
struct ModCfg {
    static constexpr int BN = BN_, CL = PAIR_ ? 2 : 1;
    static constexpr int B_ROWS = BN / CL;                    // rows of B in one CTA
    static constexpr int A_BYTES = MG_BM * MOD_BK * 2, B_BYTES = B_ROWS * MOD_BK * 2;
    static constexpr int STAGE = A_BYTES + B_BYTES;
    static constexpr int STAGES = BN == 64 ? 8 : (BN == 128 ? 6 : 7);
    static constexpr int TM = MG_BM * CL;                     // rows of a unit's tile
    // epilogue warps: 64 (BN = 64: 32) columns each.  Eight warps on 128 columns each took
    // longer over a pass than its MMAs (17 instructions an output then, 5 now)
    static constexpr int EPI = BN == 256 ? 16 : 8, THREADS = 64 + 32 * EPI, NC = 4 * BN / EPI;
    static constexpr int SMEM = STAGES * STAGE + 1024 + 256;
    static constexpr uint32_t IDESC = idesc_bf16_f32(TM, BN);
};
static_assert(ModCfg<256, true>::SMEM <= 232448 && ModCfg<128, false>::SMEM <= 232448 && ModCfg<64, false>::SMEM <= 232448,
              "shared memory per CTA");

// Tiles in groups of eight tile rows, column by column inside a group; a triangle
// product has only the tiles with an entry on or above the diagonal.
template <int BN, int TM>
__device__ __forceinline__ void mod_tile(const ModGemmArgs& p, int t, int& tm, int& tn) {
    int first = 0;
    while (true) {
        const int rows = min(8, p.tiles_m - first);
        if (!p.tri) {
            const int in_group = rows * p.tiles_n;
            if (t < in_group) {
                tm = first + t % rows;
                tn = t / rows;
                return;
            }
            t -= in_group;
        } else {
            for (int c = first * TM / BN; c < p.tiles_n; ++c) {
                const int cnt = min(rows, (c * BN + BN - 1) / TM + 1 - first);
                if (t < cnt) {
                    tm = first + t;
                    tn = c;
                    return;
                }
                t -= cnt;
            }
        }
        first += 8;
    }
}

// Bits whose low byte (low half for sums) is r + 128 (modulo 256 a residue 128 wraps to 0, i.e. -128).
__device__ __forceinline__ uint32_t mod_bits(float r) { return __float_as_uint(r + 8388736.0f); }

// Persistent, one CTA per SM: a unit is one tile (TM x BN) of one plane, worked on by the
// CTAs of a cluster.  Warp 0 loads (TMA, a
// ring of stages), warp 1 issues the MMAs into two TMEM accumulators in turn (one per
// K pass), the others reduce the finished one to bytes meanwhile.
template <int BN, bool PAIR, bool MULTI>
__global__ void __launch_bounds__(ModCfg<BN, PAIR>::THREADS, 1) mod_gemm_kernel(const __grid_constant__ CUtensorMap tA,
                                                                 const __grid_constant__ CUtensorMap tB,
                                                                 const __grid_constant__ ModGemmArgs p) {
    using Cfg = ModCfg<BN, PAIR>;
    constexpr int S = Cfg::STAGES, TM = Cfg::TM, CL = Cfg::CL;
    const int rank = PAIR ? (int)cluster_ctarank() : 0;
    const int first_unit = blockIdx.x / CL, unit_step = gridDim.x / CL;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    // full[S], empty[S], accumulator full[2], accumulator empty[2], drain
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S * Cfg::STAGE);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * S + 5);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(smem_u32(&bars[s]), 1);
            mbar_init(smem_u32(&bars[S + s]), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(smem_u32(&bars[2 * S + a]), 1);
            mbar_init(smem_u32(&bars[2 * S + 2 + a]), Cfg::EPI * CL);      // (the even CTA's is used)
        }
        mbar_init(smem_u32(&bars[2 * S + 4]), 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        if (PAIR) {
            tmem_alloc_pair(smem_u32(tmem_slot), 2 * BN);
            tmem_relinquish_pair();
        } else {
            tmem_alloc(smem_u32(tmem_slot), 2 * BN);
            tmem_relinquish();
        }
    }
    fence_before_sync();
    __syncthreads();
    if (PAIR) cluster_sync();                                  // the barriers are ready in both CTAs
    fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    const int nk = p.Kp / MOD_BK;
    constexpr int CH = MOD_CHUNK / MOD_BK;
    const int nch = (nk + CH - 1) / CH;

    if (warp == 0) {
        if (lane == 0) {
            uint32_t issued = 0, last_ph = 0;
            int kit = 0;
            bool ok = true;
            tma_prefetch_desc(&tA);
            tma_prefetch_desc(&tB);
            for (int u = first_unit; u < p.units && ok; u += unit_step) {
                const int m = u / p.tiles;
                int tm, tn;
                mod_tile<BN, TM>(p, u - m * p.tiles, tm, tn);
                for (int it = 0; it < nk; ++it, ++kit) {
                    const int s = kit % S;
                    const uint32_t ph = (kit / S) & 1;
                    if (*abort_flag || (kit >= S && !mbar_wait(smem_u32(&bars[S + s]), ph ^ 1, MG_TIMEOUT_NS))) {
                        atomicOr(p.status, DEV_TIMEOUT);
                        *abort_flag = 1;
                        ok = false;
                        break;
                    }
                    const uint32_t full = smem_u32(&bars[s]);
                    uint8_t* st = smem + s * Cfg::STAGE;
                    if (PAIR) {
                        // both CTAs' loads complete on the even one's barrier
                        const uint32_t lead = cluster_map(full, 0);
                        if (rank == 0) mbar_arrive_expect_tx(full, 2 * Cfg::STAGE);
                        tma_load_3d_pair(smem_u32(st), &tA, lead, 0, tm * TM + rank * MG_BM, m * nk + it);
                        tma_load_3d_pair(smem_u32(st + Cfg::A_BYTES), &tB, lead, 0, tn * BN + rank * Cfg::B_ROWS, m * nk + it);
                        if (rank != 0) continue;
                    } else {
                        mbar_arrive_expect_tx(full, Cfg::STAGE);
                        tma_load_3d(smem_u32(st), &tA, full, 0, tm * TM, m * nk + it);
                        tma_load_3d(smem_u32(st + Cfg::A_BYTES), &tB, full, 0, tn * BN, m * nk + it);
                    }
                    issued |= 1u << s;
                    last_ph = (last_ph & ~(1u << s)) | (ph << s);
                }
            }
            // every load has landed before the CTA may exit (a pair's loads: the even CTA waits,
            // the odd one for it at the cluster barrier below)
            for (int s = 0; s < S; ++s)
                if (((issued >> s) & 1u) && !mbar_wait(smem_u32(&bars[s]), (last_ph >> s) & 1u, MG_TIMEOUT_NS))
                    *abort_flag = 1;
        }
    } else if (warp == 1) {
        // the warp together, one lane issuing: addresses and descriptors in uniform registers
        const bool leader = elect_one();
        if (rank == 0) {
            int kit = 0, ai = 0;
            bool ok = true;
            for (int u = first_unit; u < p.units && ok; u += unit_step) {
                // the magnitudes' sum needs no exact passes
                const bool one = !MULTI || u / p.tiles == MOD_NM;
                for (int it = 0; it < nk; ++it, ++kit) {
                    const int kc = one ? it : it % CH;
                    const uint32_t acc = tmem + (uint32_t)((ai & 1) * BN);
                    if (kc == 0) {
                        if (ai >= 2) ok = mbar_wait(smem_u32(&bars[2 * S + 2 + (ai & 1)]), ((ai >> 1) - 1) & 1, MG_TIMEOUT_NS);
                        fence_after_sync();
                    }
                    const int s = kit % S;
                    ok = ok && mbar_wait(smem_u32(&bars[s]), (kit / S) & 1, MG_TIMEOUT_NS);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) {
                        if (leader) atomicOr(p.status, DEV_TIMEOUT);
                        *abort_flag = 1;
                        break;
                    }
                    fence_after_sync();
                    const uint32_t a0 = smem_u32(smem + s * Cfg::STAGE);
                    const uint64_t ad = desc_kmajor_sw128(a0), bd = desc_kmajor_sw128(a0 + Cfg::A_BYTES);
                    const uint32_t open = kc == 0 ? 0u : 1u;
                    const bool done = it == nk - 1 || (!one && kc == CH - 1);
                    if (leader) {
#pragma unroll
                        for (int kk = 0; kk < MOD_BK / 16; ++kk) {
                            const uint32_t add = kk == 0 ? open : 1u;
                            if (PAIR) mma_bf16_pair(acc, ad + 2 * kk, bd + 2 * kk, Cfg::IDESC, add);
                            else mma_bf16(acc, ad + 2 * kk, bd + 2 * kk, Cfg::IDESC, add);
                        }
                        if (PAIR) {
                            mma_commit_pair(smem_u32(&bars[S + s]));
                            if (done) mma_commit_pair(smem_u32(&bars[2 * S + (ai & 1)]));
                        } else {
                            mma_commit(smem_u32(&bars[S + s]));
                            if (done) mma_commit(smem_u32(&bars[2 * S + (ai & 1)]));
                        }
                    }
                    __syncwarp();
                    if (done) ++ai;
                }
            }
            // every MMA issued has completed before TMEM is released
            if (leader) {
                if (PAIR) mma_commit_pair(smem_u32(&bars[2 * S + 4]));
                else mma_commit(smem_u32(&bars[2 * S + 4]));
            }
            __syncwarp();
        }
        // (both CTAs of a pair wait: the odd one's barriers have then had every arrival)
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bars[2 * S + 4]), 0, MG_TIMEOUT_NS))) {
            if (leader) atomicOr(p.status, DEV_TIMEOUT);
            *abort_flag = 1;
        }
    } else {
        const int q = warp & 3, ew = warp - 2;
        constexpr int NC = Cfg::NC;                            // columns per thread
        const int c0 = NC * (ew / 4);
        int ai = 0;
        bool ok = true;
        for (int u = first_unit; u < p.units && ok; u += unit_step) {
            const int m = u / p.tiles;
            int tm, tn;
            mod_tile<BN, TM>(p, u - m * p.tiles, tm, tn);
            const int i = tm * TM + rank * MG_BM + 32 * q + lane, j0 = tn * BN + c0;
            const bool mag = m == MOD_NM;
            const int passes = (!MULTI || mag) ? 1 : nch;
            const float pm = mag ? 1.0f : c_mod.p[m], inv = mag ? 1.0f : c_mod.inv[m];
            const float bias = 8388608.0f + 128.0f * (float)passes;
            uint32_t sum[MULTI ? NC / 2 : 1];                  // two 16-bit sums of passes a word
            if (MULTI) {
#pragma unroll
                for (int c = 0; c < NC / 2; ++c) sum[MULTI ? c : 0] = 0;
            }
            for (int ps = 0; ps < passes; ++ps, ++ai) {
                if (*abort_flag || !mbar_wait(smem_u32(&bars[2 * S + (ai & 1)]), (ai >> 1) & 1, MG_TIMEOUT_NS)) {
                    if (lane == 0) atomicOr(p.status, DEV_TIMEOUT);
                    *abort_flag = 1;
                    ok = false;
                }
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                fence_after_sync();
                const uint32_t ta = tmem + (uint32_t)((ai & 1) * BN) + ((uint32_t)(32 * q) << 16) + (uint32_t)c0;
#pragma unroll
                for (int h = 0; h < NC / 32; ++h) {
                    uint32_t v[32];
                    tmem_ld_32x32b_x32(ta + 32 * h, v);
                    tmem_ld_wait();
                    if (mag) {
                        // accepted (0): the error bound is within K u S, or every product is zero
                        const ModRow ra = i < p.M ? p.ra[i] : ModRow{0, 0.0f, 0.0f, 0};
                        uint32_t w[8];
#pragma unroll
                        for (int c = 0; c < 32; ++c) {
                            const int j = min(j0 + 32 * h + c, p.N - 1);
                            const float thr = (ra.rho * p.rb[j].n1 + p.rb[j].rho * ra.n1) * p.kfac;
                            const float s = __uint_as_float(v[c]);
                            const uint32_t bad = !(s >= thr || (s == 0.0f && thr < 1e30f)) ? 1u : 0u;
                            w[c / 4] = (c % 4 == 0) ? bad : (w[c / 4] | (bad << (8 * (c % 4))));
                        }
                        if (i < p.M) {
                            uint4* o = reinterpret_cast<uint4*>(p.R + (size_t)m * p.plane + (size_t)i * p.ldr + j0 + 32 * h);
                            o[0] = make_uint4(w[0], w[1], w[2], w[3]);
                            o[1] = make_uint4(w[4], w[5], w[6], w[7]);
                        }
                        continue;
                    }
                    if (MULTI) {
#pragma unroll
                        for (int c = 0; c < 32; c += 2) {
                            const uint32_t r0 = mod_bits(mod_centred(__uint_as_float(v[c]), pm, inv));
                            const uint32_t r1 = mod_bits(mod_centred(__uint_as_float(v[c + 1]), pm, inv));
                            sum[MULTI ? 16 * h + c / 2 : 0] += __byte_perm(r0, r1, 0x5410);
                        }
                        if (ps < passes - 1) continue;
                    }
                    uint32_t w[8];
#pragma unroll
                    for (int c = 0; c < 32; c += 4) {
                        uint32_t r[4];
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            float x;
                            if (MULTI) {
                                // a half word: the passes' residues + 128 each
                                const uint32_t s2 = sum[MULTI ? 16 * h + (c + t) / 2 : 0];
                                const uint32_t s = (t & 1) ? (s2 >> 16) : (s2 & 0xFFFFu);
                                x = __uint_as_float(0x4B000000u | s) - bias;
                            } else {
                                x = __uint_as_float(v[c + t]);
                            }
                            r[t] = mod_bits(mod_centred(x, pm, inv));
                        }
                        w[c / 4] = __byte_perm(__byte_perm(r[0], r[1], 0x0040), __byte_perm(r[2], r[3], 0x0040), 0x5410);
                    }
                    if (i < p.M) {
                        uint4* o = reinterpret_cast<uint4*>(p.R + (size_t)m * p.plane + (size_t)i * p.ldr + j0 + 32 * h);
                        o[0] = make_uint4(w[0], w[1], w[2], w[3]);
                        o[1] = make_uint4(w[4], w[5], w[6], w[7]);
                    }
                }
                fence_before_sync();
                __syncwarp();
                if (lane == 0) {
                    const uint32_t eb = smem_u32(&bars[2 * S + 2 + (ai & 1)]);
                    if (PAIR) mbar_arrive_cluster(cluster_map(eb, 0));
                    else mbar_arrive(eb);
                }
            }
        }
    }
    fence_before_sync();
    __syncthreads();
    fence_after_sync();
    // no CTA of a pair leaves, or frees its TMEM, while the other's loads, MMAs or arrivals may
    // still reach it
    if (PAIR) {
        cluster_sync();
        if (warp == 1) tmem_dealloc_pair(tmem, 2 * BN);
    } else if (warp == 1) {
        tmem_dealloc(tmem, 2 * BN);
    }
}

// ------------------------------------------------------------------ 3. combine
// The signed 128-bit integer v times 2^e as a double: its 64 leading bits, rounded to the
// nearest (ties to even), all in integers (a conversion per output on the FP64 pipe, two a
// cycle and SM, would cost as much as the rest).
__device__ __forceinline__ double int_scaled(__int128 v, int e) {
    const bool neg = v < 0;
    const u128 a = neg ? (u128)(-v) : (u128)v;
    const unsigned long long hi = (unsigned long long)(a >> 64), lo = (unsigned long long)a;
    if ((hi | lo) == 0) return 0.0;
    const int z = hi ? __clzll((long long)hi) : 64 + __clzll((long long)lo);
    const unsigned long long t = (unsigned long long)((a << z) >> 64);      // top bit set
    unsigned long long m = t >> 11;
    const unsigned rem = (unsigned)t & 0x7FFu;
    m += rem > 0x400u || (rem == 0x400u && (m & 1));
    // m in [2^52, 2^53]: its top bit adds one to the exponent field below
    const unsigned long long b =
        m + ((unsigned long long)(1023 + 126 - z + e) << 52) + (neg ? 1ull << 63 : 0ull);
    return __longlong_as_double((long long)b);
}

// A block of the combine: MC_ROWS rows of a 32 x 32 tile, four outputs a thread.
constexpr int MC_ROWS = 8, MC_THREADS = 8 * MC_ROWS;
// Most outputs of a strip (256) recomputed one by one, a warp each; more, and the whole strip is.
// The list's time grows with its length: 64, 128, 192 outputs against the strip at n = 256 93, 118,
// 143 / 122 us, n = 576 210, 319, 428 / 453, n = 1024 714, 1256, 1781 / 1968 (S P S^T, two products,
// all strips alike).  Where strips differ, the longest list decides: a localised state at
// n = 225 takes 136 us with lists of up to 8, 197 with up to 128.
constexpr int MC_LIST = 64;

// FP64 sums of a strip from the operands (k in increasing order, fma), four outputs a thread;
// the next 16 k are loaded beside the FMAs.
__device__ __noinline__ void mod_native_strip(const GemmProb& pb, int row0, int col0, double (*As)[MC_ROWS + 1],
                                              double (*Bs)[33], double (*sS)[33]) {
    constexpr int NT = MC_THREADS, ROWS = MC_ROWS, NB = 16 * 32 / NT;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    double a[2], b[NB];
    auto load = [&](int k0) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int e = tid + NT * q, r = row0 + (pb.transA ? e % ROWS : e >> 4), k = k0 + (pb.transA ? e / ROWS : e & 15);
            a[q] = r < pb.M && k < pb.K ? (pb.transA ? pb.A[(size_t)k * pb.lda + r] : pb.A[(size_t)r * pb.lda + k]) : 0.0;
        }
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int e = tid + NT * q, c = col0 + (pb.transB ? e >> 4 : e & 31), k = k0 + (pb.transB ? e & 15 : e >> 5);
            b[q] = c < pb.N && k < pb.K ? (pb.transB ? pb.B[(size_t)c * pb.ldb + k] : pb.B[(size_t)k * pb.ldb + c]) : 0.0;
        }
    };
    double acc[2][2] = {};
    load(0);
    for (int k0 = 0; k0 < pb.K; k0 += 16) {
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int e = tid + NT * q;
            As[pb.transA ? e / ROWS : e & 15][pb.transA ? e % ROWS : e >> 4] = a[q];
        }
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int e = tid + NT * q;
            Bs[pb.transB ? e & 15 : e >> 5][pb.transB ? e >> 4 : e & 31] = b[q];
        }
        __syncthreads();
        if (k0 + 16 < pb.K) load(k0 + 16);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const double a0 = As[k][ty], a1 = As[k][ty + ROWS / 2], b0 = Bs[k][tx], b1 = Bs[k][tx + 16];
            acc[0][0] = fma(a0, b0, acc[0][0]);
            acc[0][1] = fma(a0, b1, acc[0][1]);
            acc[1][0] = fma(a1, b0, acc[1][0]);
            acc[1][1] = fma(a1, b1, acc[1][1]);
        }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) sS[ty + ROWS / 2 * i][tx + 16 * j] = acc[i][j];
}

// Four outputs a thread from their 16 residues (one word per plane), the sums staged in shared
// memory; outputs without a certificate replaced by FP64 sums (a warp each, or the whole
// strip); then the product's epilogue, coalesced (and its mirror for a triangle).
// Strips of 8 rows: where most outputs fail (a state localised around one node, P0 = 0) the FP64
// pipe bounds the product, and blocks of a whole tile left SMs idle.  T12 step of such a state /
// of a dense one, us: n = 196 123 / 34 (tiles of 32 rows, 33 outputs sending the tile to FP64:
// 174 / 35; the FP64 pipe alone 145), n = 256 144 / 34 (204 / 36; 174), n = 576 604 / 64 (836 / 66;
// 781), n = 1024 2695 / 111 (3016 / 113; 3168), n = 2025 19090 / 424 (21290 / 426; 22760).  Eight
// factored steps from one node's C: n = 1024 2.1 ms (5.4; 2.1), n = 2304 4.6 (12.8; 12.1).
__global__ void __launch_bounds__(MC_THREADS) mod_combine_kernel(const __grid_constant__ GemmProb pb,
                                                                 const uint8_t* __restrict__ R, size_t plane, int ldr,
                                                                 const ModRow* __restrict__ ra, const ModRow* __restrict__ rb,
                                                                 int certify, int tiles_n) {
    constexpr int ROWS = MC_ROWS, STRIPS = 32 / ROWS, WARPS = MC_THREADS / 32;
    __shared__ double sS[ROWS][33];
    __shared__ double As[16][ROWS + 1], Bs[16][33];
    __shared__ int s_cnt;
    __shared__ int s_list[MC_LIST];
    const int tile = blockIdx.x / STRIPS;
    int ti, tj;
    if (pb.tri) {
        // tile t of the upper triangle, column by column: tj (tj + 1) / 2 <= t
        tj = (int)((sqrtf(8.0f * (float)tile + 1.0f) - 1.0f) * 0.5f);
        while ((tj + 1) * (tj + 2) / 2 <= tile) ++tj;
        while (tj * (tj + 1) / 2 > tile) --tj;
        ti = tile - tj * (tj + 1) / 2;
    } else {
        ti = tile / tiles_n;
        tj = tile % tiles_n;
    }
    const int i0 = ti * 32 + (blockIdx.x % STRIPS) * ROWS, j0 = tj * 32;
    if (threadIdx.x == 0) s_cnt = 0;
    __syncthreads();
    {
        const int r = threadIdx.x >> 3, c = 4 * (threadIdx.x & 7);
        const int i = i0 + r, j = j0 + c;
        if (i < pb.M && j < pb.N) {
            const uint8_t* src = R + (size_t)i * ldr + j;
            uint32_t y[MOD_NM];
#pragma unroll
            for (int m = 0; m < MOD_NM; ++m) y[m] = *reinterpret_cast<const uint32_t*>(src + (size_t)m * plane);
            uint32_t flags = certify ? *reinterpret_cast<const uint32_t*>(src + (size_t)MOD_NM * plane) : 0u;
            const ModRow rr = ra[i];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (j + u >= pb.N) break;
                unsigned long long a0 = c_mod.o0, a1 = c_mod.o1, a2 = c_mod.o2;
#pragma unroll
                for (int m = 0; m < MOD_NM; ++m) {
                    const uint32_t v = (y[m] >> (8 * u)) & 0xFFu;
                    a0 += (unsigned long long)v * c_mod.w0[m];
                    a1 += (unsigned long long)v * c_mod.w1[m];
                    a2 += (unsigned long long)v * c_mod.w2[m];
                }
                // x = sum - q P with q = rint(sum / P); |x| < P / 8, so q is never ambiguous
                const unsigned long long top = a2 + (a1 >> 32);
                const uint32_t q = __float2uint_rn((float)(uint32_t)(top >> 10) * c_mod.qscale);
                const u128 s = ((u128)a2 << 64) + ((u128)a1 << 32) + (u128)a0;
                const u128 qp = (u128)q * (u128)c_mod.plo + ((u128)((unsigned long long)q * c_mod.phi) << 64);
                const ModRow rc = rb[j + u];
                sS[r][c + u] = int_scaled((__int128)(s - qp), 32 - rr.sigma - rc.sigma);
                const bool bad = certify ? ((flags >> (8 * u)) & 0xFFu) != 0 : !(rr.n1 < 1e38f && rc.n1 < 1e38f);
                if (bad && !(pb.tri && i > j + u)) {
                    const int e = atomicAdd(&s_cnt, 1);
                    if (e < MC_LIST) s_list[e] = r * 32 + c + u;
                }
            }
        }
    }
    __syncthreads();
    const int cnt = s_cnt;
    if (cnt > MC_LIST) {
        mod_native_strip(pb, i0, j0, As, Bs, sS);
        __syncthreads();
    } else if (cnt > 0) {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        for (int e = warp; e < cnt; e += WARPS) {
            const int i = i0 + s_list[e] / 32, j = j0 + s_list[e] % 32;
            double a = 0.0;
            for (int k = lane; k < pb.K; k += 32) {
                const double x = pb.transA ? pb.A[(size_t)k * pb.lda + i] : pb.A[(size_t)i * pb.lda + k];
                const double w = pb.transB ? pb.B[(size_t)j * pb.ldb + k] : pb.B[(size_t)k * pb.ldb + j];
                a = fma(x, w, a);
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
            if (lane == 0) sS[s_list[e] / 32][s_list[e] % 32] = a;
        }
        __syncthreads();
    }
    const int cc = threadIdx.x & 31;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        const int r = (threadIdx.x >> 5) + WARPS * h, i = i0 + r, j = j0 + cc;
        if (i < pb.M && j < pb.N && !(pb.tri && i > j)) {
            const size_t off = (size_t)i * pb.ldd + j;
            double v = sS[r][cc];
            if (pb.alpha != 1.0) v *= pb.alpha;
            if (pb.D1) v += pb.b1 * pb.D1[off];
            if (pb.D2) v += pb.b2 * pb.D2[off];
            if (pb.D3) v += pb.b3 * pb.D3[off];
            pb.C[(size_t)i * pb.ldc + j] = v;
            if (pb.tri) sS[r][cc] = v;
        }
    }
    if (!pb.tri) return;
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        // the mirror: row j0 + r of the lower triangle, column i0 + ic
        const int ic = threadIdx.x % ROWS, r = threadIdx.x / ROWS + 8 * h, j = j0 + r, i = i0 + ic;
        if (j < pb.N && i < pb.M && i < j) pb.C[(size_t)j * pb.ldc + i] = sS[ic][r];
    }
}

int mod_sms() {
    static const int sms = [] {
        int dev = 0, c = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&c, cudaDevAttrMultiProcessorCount, dev);
        return std::max(c, 1);
    }();
    return sms;
}

dme_status mod_map(const ModBuf& b, int box_rows, CUtensorMap* out) {
    cuuint64_t dims[3] = {(cuuint64_t)MOD_BK, (cuuint64_t)b.rows, (cuuint64_t)MOD_PLANES * (b.Kp / MOD_BK)};
    cuuint64_t strides[2] = {(cuuint64_t)MOD_BK * 2, (cuuint64_t)b.rows * MOD_BK * 2};
    cuuint32_t box[3] = {(cuuint32_t)MOD_BK, (cuuint32_t)box_rows, 1};
    return encode_bf16_map(out, b.data, 3, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B);
}

template <int BN, bool PAIR, bool MULTI>
dme_status mod_gemm_launch(const CUtensorMap& tA, const CUtensorMap& tB, const ModGemmArgs& a, int groups, cudaStream_t st) {
    using Cfg = ModCfg<BN, PAIR>;
    static const cudaError_t attr = cudaFuncSetAttribute(
        mod_gemm_kernel<BN, PAIR, MULTI>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::SMEM);
    DME_CUDA_TRY(attr);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(std::min(a.units, groups) * Cfg::CL);
    cfg.blockDim = dim3(Cfg::THREADS);
    cfg.dynamicSmemBytes = Cfg::SMEM;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = Cfg::CL;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = PAIR ? 1 : 0;
    DME_CUDA_TRY(cudaLaunchKernelEx(&cfg, mod_gemm_kernel<BN, PAIR, MULTI>, tA, tB, a));
    return DME_OK;
}

// CTA pairs that the device holds at once (0: none).
int mod_pairs() {
    static const int n = [] {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2 * mod_sms());
        cfg.blockDim = dim3(ModCfg<256, true>::THREADS);
        cfg.dynamicSmemBytes = ModCfg<256, true>::SMEM;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 2;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int c = 0;
        if (cudaFuncSetAttribute(mod_gemm_kernel<256, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 ModCfg<256, true>::SMEM) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&c, mod_gemm_kernel<256, true, true>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        return std::min(c, mod_sms() / 2);
    }();
    return n;
}

// Tiles of TM x BN of an M x N product (a triangle: those with an entry on or above the
// diagonal).
int mod_tile_count(int M, int N, int tri, int tm, int bn) {
    const int rows = (M + tm - 1) / tm, cols = (N + bn - 1) / bn;
    if (!tri) return rows * cols;
    int t = 0;
    for (int c = 0; c < cols; ++c) t += std::min(rows, (c * bn + bn - 1) / tm + 1);
    return t;
}

}  // namespace

dme_status mod_place(ModBuf& b, void* mem) {
    b.data = static_cast<__nv_bfloat16*>(mem);
    b.row = reinterpret_cast<ModRow*>(static_cast<char*>(mem) + mod_plane_bytes(b.rows, b.k));
    DME_TRY(mod_map(b, 64, &b.t64));
    return mod_map(b, 128, &b.t128);
}

void launch_mod_convert(const double* X, int rows, int k, int ld, const ModBuf& b, cudaStream_t st) {
    if (rows <= 0 || rows > b.rows) return;
    if (b.Kp <= 256) mod_convert_kernel<64><<<rows, 64, 0, st>>>(X, k, ld, b.data, b.Kp, b.row, b.rows);
    else if (b.Kp <= 512) mod_convert_kernel<128><<<rows, 128, 0, st>>>(X, k, ld, b.data, b.Kp, b.row, b.rows);
    else mod_convert_kernel<256><<<rows, 256, 0, st>>>(X, k, ld, b.data, b.Kp, b.row, b.rows);
}

dme_status launch_mod_gemm(const ModBuf& A, const ModBuf& B, const GemmProb& g, uint8_t* ws, bool certify, int* status,
                           cudaStream_t st) {
    if (g.M <= 0 || g.N <= 0) return DME_OK;
    if (g.M > A.rows || g.N > B.rows || A.Kp != B.Kp || g.K != A.k || (g.tri && g.M != g.N))
        return set_error("residue product: the planes do not hold the operands"), DME_EINVAL;
    ModGemmArgs a;
    a.M = g.M;
    a.N = g.N;
    a.Kp = A.Kp;
    a.tri = g.tri;
    a.R = ws;
    a.ldr = mod_ldr(g.N);
    a.plane = (size_t)g.M * a.ldr;
    a.ra = A.row;
    a.rb = B.row;
    a.kfac = 9007199254740992.0f / (float)g.K;
    a.status = status;
    const int planes = certify ? MOD_PLANES : MOD_NM;
    const bool multi = a.Kp > MOD_CHUNK;
    auto shape = [&](int tm, int bn) {
        a.tiles_m = (g.M + tm - 1) / tm;
        a.tiles_n = (g.N + bn - 1) / bn;
        a.tiles = mod_tile_count(g.M, g.N, g.tri, tm, bn);
        a.units = a.tiles * planes;
    };
    if (g.N <= 64) {
        shape(MG_BM, 64);
        DME_TRY(multi ? (mod_gemm_launch<64, false, true>(A.t128, B.t64, a, mod_sms(), st))
                      : (mod_gemm_launch<64, false, false>(A.t128, B.t64, a, mod_sms(), st)));
    } else {
        // the shape with the shorter run: waves x measured cycles per K block of 64 (pairs:
        // 600 to 700, less the longer the run; the smaller tile 690).  Below
        // K = 512 a unit is all latency and the smaller tile is faster (n = 256: 8.4 us
        // against 12.1)
        const int np = mod_pairs();
        const long w1 = ((long)mod_tile_count(g.M, g.N, g.tri, 128, 128) * planes + mod_sms() - 1) / mod_sms();
        const long w2 = np > 0 ? ((long)mod_tile_count(g.M, g.N, g.tri, 256, 256) * planes + np - 1) / np : 0;
        if (np > 0 && a.Kp >= 512 && w2 * 600 < w1 * 690) {
            shape(256, 256);
            DME_TRY(multi ? (mod_gemm_launch<256, true, true>(A.t128, B.t128, a, np, st))
                          : (mod_gemm_launch<256, true, false>(A.t128, B.t128, a, np, st)));
        } else {
            shape(MG_BM, 128);
            DME_TRY(multi ? (mod_gemm_launch<128, false, true>(A.t128, B.t128, a, mod_sms(), st))
                          : (mod_gemm_launch<128, false, false>(A.t128, B.t128, a, mod_sms(), st)));
        }
    }
    const int tn = (g.N + 31) / 32, tm = (g.M + 31) / 32;
    const int strips = (g.tri ? tn * (tn + 1) / 2 : tm * tn) * (32 / MC_ROWS);
    mod_combine_kernel<<<strips, MC_THREADS, 0, st>>>(g, a.R, a.plane, a.ldr, a.ra, a.rb, certify ? 1 : 0, tn);
    DME_CUDA_TRY(cudaGetLastError());
    return DME_OK;
}

}  // namespace dme
