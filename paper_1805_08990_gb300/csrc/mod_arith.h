// The moduli of the residue products and the reduction their epilogue uses, for the device
// and for a host compiler.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define DME_MOD_FN __host__ __device__ __forceinline__
#else
#define DME_MOD_FN inline
#endif

namespace dme {

constexpr int MOD_NM = 16;            // moduli

// Pairwise coprime, product 2^125.3.  All but 256 are at most 253: a residue of mod_centred is
// then at most 127 (below).  (255 is coprime to the others too, but reduces some sums above
// 2^23 to +128, which the byte of the result cannot tell from -128.)
constexpr int kModuli[MOD_NM] = {256, 253, 251, 249, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193};

// x mod p for an integer |x| <= 2^24 in fp32, inv = 1 / p rounded: in [-127, 127] for the odd
// moduli, [-128, 128] for 256.  The fma rounds x inv to an integer exactly once, so its
// argument is off by at most 2^24 2^-32 (1 / p < 2^-7 has an error of 2^-32 at most; none
// for 256), and |residue| <= p (1/2 + 2^-8) < 128 for p <= 253.
DME_MOD_FN float mod_centred(float x, float p, float inv) {
    const float q = fmaf(x, inv, 12582912.0f) - 12582912.0f;
    return fmaf(-q, p, x);
}

}  // namespace dme
