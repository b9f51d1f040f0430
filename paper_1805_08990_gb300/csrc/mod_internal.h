// FP64 products as exact residue products on the tensor cores.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "dme_internal.h"
#include "mod_arith.h"

namespace dme {

constexpr int MOD_PLANES = 17;        // residues, then the magnitudes |x| / 2^E
constexpr int MOD_BK = 64;            // K per stage (one 128-byte swizzle row of bf16)

// One row of an operand: its entries are rint(x 2^sigma); rho bounds the rounding
// error of one entry and n1 the row's 1-norm, both in units of 2^E > max |x|
// (n1 = infinity for a row the residues cannot hold).
struct ModRow {
    int sigma;
    float rho, n1;
    int pad;
};

// Residue planes of a rows x k operand: [MOD_PLANES][Kp / 64][rows][64] bf16 (the rows of a
// tile's K block are contiguous), Kp = k rounded up to 64 (zero padded), and the rows' scales.
struct ModBuf {
    __nv_bfloat16* data = nullptr;
    ModRow* row = nullptr;
    int rows = 0, k = 0, Kp = 0;
    CUtensorMap t64, t128;            // boxes of 64 k x (64, 128) rows of one plane
};

inline int mod_kpad(int k) { return (k + MOD_BK - 1) / MOD_BK * MOD_BK; }
inline size_t mod_plane_bytes(int rows, int k) { return (size_t)MOD_PLANES * rows * mod_kpad(k) * 2; }
// One allocation: the planes (a multiple of 128 bytes), then the rows' scales.
inline size_t mod_buf_bytes(int rows, int k) { return mod_plane_bytes(rows, k) + (size_t)rows * sizeof(ModRow); }
// Workspace of an M x N product: a byte per residue and output, and the certificate.
inline int mod_ldr(int N) { return (N + 255) / 256 * 256; }
inline size_t mod_ws_bytes(int M, int N) { return (size_t)MOD_PLANES * M * mod_ldr(N); }

// Put buf (rows, k, Kp set) into mod_buf_bytes of memory and encode its tensor maps.
dme_status mod_place(ModBuf& buf, void* mem);
// Residue planes of the rows of X (rows x k, leading dimension ld; rows <= buf.rows).
void launch_mod_convert(const double* X, int rows, int k, int ld, const ModBuf& buf, cudaStream_t st);
// g (C = alpha op(A) op(B) + addends, triangle mode as gemm64_grouped) from the residue
// planes of the rows of op(A) and of the rows of op(B)^T.  g's A and B are the operands
// themselves, for the outputs recomputed in FP64.  certify: outputs whose error bound is
// not below the FP64 sum's own are recomputed; else only those of rows and columns that
// the residues cannot hold.  ws: mod_ws_bytes(M, N).
dme_status launch_mod_gemm(const ModBuf& A, const ModBuf& B, const GemmProb& g, uint8_t* ws, bool certify, int* status,
                           cudaStream_t st);

}  // namespace dme
