// The factorisation of a 128-column QR block from its Gram matrix (qr_block.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "soap_internal.h"

namespace soap {

constexpr int kQrBlock = 128;
constexpr int kQrGramParts = 4;   // partial Gram matrices per matrix at most
constexpr int kQrTraceParts = 8;  // partial sums of the trace

// A block factored from its Gram matrix is kept if the inverse of that matrix scaled to a unit diagonal,
// G^^-1 (qr_block.cu), is bounded in norm by about 26: by its trace's excess over kbo or by its Frobenius
// norm. max|H^T H - I| of a block, simulated in 32 bits, is 0.3-1.8e-6 up to an excess of 24 (unit
// columns with one small singular value, shared by all of them or not), as it is in the steady state,
// 1-3e-6 at 32 to 48, 2-5e-6 at 61 and 1e-5 at 250; of blocks of training runs 0.9-1.4e-6 up to a
// Frobenius norm of 28, whatever their excess; the column loop's 0.2-0.4e-6. In such runs the trace keeps
// a third of the blocks of steps 4 to 8 that the pivots leave, the Frobenius norm nineteen in twenty.
// A step of 256 x 512 with the rule: 749 -> 757 us, QR of 16 x 2048^2: 6413 -> 6461 us.
constexpr float kQrMaxExcess = 24.f;
constexpr float kQrMaxInverse = 28.f;

// What qr_block_fast did with a matrix's block (state[b]).
enum : int {
  kQrBlockFast = 0,     // factored, if the inverse's bound allows it
  kQrBlockColumns = 1,  // left to the column loop
  kQrBlockZero = 2,     // every column below the zero-column threshold: no reflectors
};

struct QrBlockArgs {
  const float* At;      // [batch][n][n] working P^T
  float* Vt;            // [batch][n][n] Householder vectors as rows
  float* Vt_lo;
  float* Vpos;          // [batch][n][128] the block's Householder vectors, position-major
  float* Vpos_lo;
  float* T;             // [batch][128][128] the block's T, and T^T
  float* T_lo;
  float* Tt;
  float* Tt_lo;
  float* Gpart;         // [batch][kQrGramParts][128][128]
  float* Rf;            // [batch][n][128] rows of D R (from the diagonal on)
  float* Wf;            // [batch][n][128] rows of W (from the diagonal on)
  int* state;           // [batch]
  uint8_t* skip;        // [batch][n]
  float* dsign;         // [batch][n]
  const float* thresh;  // [batch]
  int* status;
  int n, k0, kbo;
};

cudaError_t qr_block_fast(const QrBlockArgs& p, int batch, cudaStream_t s);

#ifdef __CUDACC__
// After qr_block_fast, for a block that it factored: the excess, and R^-1 (128 x 128, upper triangular,
// zeros elsewhere) scaled so that G^^-1 is its product with its transpose.
__device__ __forceinline__ float qr_block_excess(const float* Gpart, int b, int kbo) {
  const float* t = Gpart + ((int64_t)b * kQrGramParts + 1) * kQrBlock * kQrBlock;
  float x = 0.f;
#pragma unroll
  for (int i = 0; i < kQrTraceParts; ++i) x += t[i];
  return x - (float)kbo;
}
__device__ __forceinline__ const float* qr_block_inverse(const float* Gpart, int b) {
  return Gpart + ((int64_t)b * kQrGramParts + 2) * kQrBlock * kQrBlock;
}
#endif

}  // namespace soap
