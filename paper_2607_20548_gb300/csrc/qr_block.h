// The factorisation of a 128-column QR block from its Gram matrix (qr_block.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "soap_internal.h"

namespace soap {

constexpr int kQrBlock = 128;
constexpr int kQrGramParts = 4;  // partial Gram matrices per matrix at most

// What qr_block_fast did with a matrix's block (state[b]).
enum : int {
  kQrBlockFast = 0,     // factored
  kQrBlockColumns = 1,  // left to the column loop: nothing was written but the state
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

}  // namespace soap
