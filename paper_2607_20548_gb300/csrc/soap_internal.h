// Internal declarations shared by the libsoap translation units (not part of the ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/soap.h"
#include "profile.h"

namespace soap {

// Sticky device status bits (combined with atomicOr by the kernels).
enum : int {
  kStatusNonFinite = 1,
  kStatusQrBreakdown = 2,
  kStatusTimeout = 4,
};

// A batched matrix operand: matrix b starts at (ptrs ? ptrs[b] : base + b * stride) + offset.
struct Operand {
  const float* base;
  const float* const* ptrs;  // device array of per-matrix pointers, or nullptr
  int64_t stride;
  int64_t offset;
  int64_t ld;
};

struct MutOperand {
  float* base;
  float* const* ptrs;
  int64_t stride;
  int64_t offset;
  int64_t ld;
};

inline Operand strided(const float* base, int64_t ld, int64_t stride, int64_t offset = 0) {
  return Operand{base, nullptr, stride, offset, ld};
}
inline MutOperand strided_mut(float* base, int64_t ld, int64_t stride, int64_t offset = 0) {
  return MutOperand{base, nullptr, stride, offset, ld};
}

// C_b = alpha * op(A_b) op(B_b) + beta * C_b for b < batch (fp32-accurate).
// Returns a cudaError_t from the launch.
cudaError_t gemm(bool trans_a, bool trans_b, int M, int N, int K, float alpha, Operand A,
                 Operand B, float beta, MutOperand C, int batch, cudaStream_t stream);

// CUDA-core fp32 engine (exact fp32 FMAs); any shape.
cudaError_t gemm_simt(bool trans_a, bool trans_b, int M, int N, int K, float alpha, Operand A,
                      Operand B, float beta, MutOperand C, int batch, cudaStream_t stream);

// ---- tcgen05 fp32 engine (four TF32 products): C_b = alpha * A_b B_(b mod B.batch)^T + beta * C_b
// An operand is `batch` row-major (rows x K) matrices split as hi = trunc_tf32(x) (the fp32
// array itself may serve: the tensor core drops the 13 low mantissa bits) and lo = x - hi.
struct TcOperand {
  const float* hi;
  const float* lo;
  int64_t ld;      // elements between rows
  int64_t stride;  // elements between matrices
  int batch;       // distinct matrices (0: one per launch batch entry)
};
struct TcEpilogue {
  float* C;              // output, matrix b at b * c_stride
  int64_t ldc;
  int64_t c_stride;
  float* C_lo;           // optional: also write out - tf32(out) here (same layout, ld_lo)
  int64_t ld_lo;
  int64_t lo_stride;
  int transpose;         // write C^T (C_b is then N x M with leading dimension ldc)
  float alpha, beta;     // beta != 0 reads C
  int* status;           // device status word for a timed-out wait (may be nullptr)
  // set by gemm_tc_nt from the library's wait settings (soap_wait_limit), not by callers:
  uint64_t wait_ns = 0;       // bounded waits give up after this long
  const int* hold = nullptr;  // testing the timeout path: the epilogue first waits for *hold != 0
};
// `family` tags the launch for the library's profiler. With a split workspace (room for
// ksplit * batch * M * N floats) a launch of few tiles and long K may split K over more CTAs
// and add the partial sums in a second kernel (row-major C with beta = 0 only).
cudaError_t gemm_tc_nt(int M, int N, int K, int batch, const TcOperand& A, const TcOperand& B,
                       const TcEpilogue& ep, cudaStream_t stream, int family = kFamGemmTc,
                       float* split_ws = nullptr, size_t split_ws_floats = 0);
// Bound of the tensor-core products' device waits (0: 2 s) and, for testing the timeout path, a
// device flag their epilogues first wait for (nullptr: none); applies to later launches.
void set_wait_limit(uint64_t ns, const int* hold);
// The settings in force (0: the default bound).
void get_wait_limit(uint64_t* ns, const int** hold);

// ---- fp32-accurate products of operands kept as three bf16 planes (gemm_b3.cu) -----------------
// x = h + m + l to 2^-26, each plane the rounding to nearest bf16 of what the ones before it leave.
// `count` row-major rows x cols matrices as planes: element (i, j) of matrix b of plane q at
// q * plane + b * stride + i * ld + j; rows start on 16 bytes (TMA).
inline int64_t plane_ld(int64_t cols) { return (cols + 7) & ~(int64_t)7; }
struct Planes {
  __nv_bfloat16* p = nullptr;
  int64_t plane = 0, stride = 0, ld = 0;
  __host__ __device__ Planes at(int64_t b, int64_t row = 0, int64_t col = 0) const {  // from matrix b, row, column on
    Planes o = *this;
    o.p += b * stride + row * ld + col;
    return o;
  }
};
inline size_t planes_bytes(int64_t rows, int64_t cols, int64_t count) {
  return (size_t)(6 * count * rows * plane_ld(cols));
}
inline Planes planes_in(void* base, int64_t rows, int64_t cols, int64_t count) {
  const int64_t ld = plane_ld(cols);
  return Planes{static_cast<__nv_bfloat16*>(base), count * rows * ld, rows * ld, ld};
}
struct B3Operand {
  const __nv_bfloat16* p;
  int64_t plane, ld, stride;
  int batch;               // distinct matrices (0: one per launch batch entry)
};
inline B3Operand b3_op(const Planes& x, int batch) { return B3Operand{x.p, x.plane, x.ld, x.stride, batch}; }
struct B3Epilogue {
  float* C;                // fp32 output (or nullptr), matrix b at b * c_stride ...
  float* const* C_ptrs;    // ... or a device array of per-matrix output pointers (16-byte aligned)
  int64_t ldc, c_stride;
  __nv_bfloat16* P;        // output as planes (or nullptr)
  int64_t p_plane, p_ld, p_stride;
  int transpose;           // write C^T (N x M)
  float alpha, beta;       // beta != 0 reads C
  int* status;             // device status word for a timed-out wait (may be nullptr)
  uint64_t wait_ns;        // set by gemm_b3 from the library's wait settings
  const int* hold;
  // the C of beta != 0 as planes (layout of P; not transposed): P itself, or P null. Its rows and columns
  // before cin_from are not read: they are those of diag(d), d_i at cin_diag[b * cin_diag_stride + i].
  const __nv_bfloat16* cin = nullptr;
  const float* cin_diag = nullptr;
  int64_t cin_diag_stride = 0;
  int cin_from = 0;
};
// C_b = alpha A_b B_(b mod B.batch)^T + beta C_b, in fp32 or as planes. The dimension that C's rows
// run along must be a multiple of 4, C and its rows 16-byte aligned.
cudaError_t gemm_b3(int M, int N, int K, int batch, const B3Operand& A, const B3Operand& B, const B3Epilogue& ep,
                    cudaStream_t s, int family = kFamGemmTc);
// C_b = alpha A_b A_b^T + beta C_b (M x M): only the tiles on or below the diagonal are computed,
// each below it also stored in the mirror position; C in fp32 (read) and as planes.
cudaError_t gemm_b3_syrk(int M, int K, int batch, const B3Operand& A, const B3Epilogue& ep, cudaStream_t s,
                         int family = kFamGemmTc);

#ifdef __CUDACC__
// The three planes of a value, and of four (one 8-byte word of each plane).
__device__ __forceinline__ void b3_split(float x, __nv_bfloat16& h, __nv_bfloat16& m, __nv_bfloat16& l) {
  h = __float2bfloat16_rn(x);
  const float r = x - __bfloat162float(h);
  m = __float2bfloat16_rn(r);
  l = __float2bfloat16_rn(r - __bfloat162float(m));
}
__device__ __forceinline__ void b3_split2(float x, float y, uint32_t& h, uint32_t& m, uint32_t& l) {
  const __nv_bfloat162 hh = __floats2bfloat162_rn(x, y);
  const float2 hf = __bfloat1622float2(hh);
  const float rx = x - hf.x, ry = y - hf.y;
  const __nv_bfloat162 mm = __floats2bfloat162_rn(rx, ry);
  const float2 mf = __bfloat1622float2(mm);
  const __nv_bfloat162 ll = __floats2bfloat162_rn(rx - mf.x, ry - mf.y);
  h = reinterpret_cast<const uint32_t&>(hh);
  m = reinterpret_cast<const uint32_t&>(mm);
  l = reinterpret_cast<const uint32_t&>(ll);
}
__device__ __forceinline__ void b3_split4(float4 x, uint2& h, uint2& m, uint2& l) {
  b3_split2(x.x, x.y, h.x, m.x, l.x);
  b3_split2(x.z, x.w, h.y, m.y, l.y);
}
__device__ __forceinline__ void b3_store(__nv_bfloat16* p, int64_t plane, float x) {
  b3_split(x, p[0], p[plane], p[2 * plane]);
}
__device__ __forceinline__ float4 b3_load4(const __nv_bfloat16* p, int64_t plane) {  // h + m + l, 8-byte aligned
  float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int pl = 2; pl >= 0; --pl) {  // the smallest plane first
    const uint2 w = *reinterpret_cast<const uint2*>(p + pl * plane);
    const float2 a = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162&>(w.x));
    const float2 b = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162&>(w.y));
    o.x += a.x; o.y += a.y; o.z += b.x; o.w += b.y;
  }
  return o;
}
__device__ __forceinline__ void b3_store4(__nv_bfloat16* p, int64_t plane, float4 x) {  // 8-byte aligned
  uint2 h, m, l;
  b3_split4(x, h, m, l);
  *reinterpret_cast<uint2*>(p) = h;
  *reinterpret_cast<uint2*>(p + plane) = m;
  *reinterpret_cast<uint2*>(p + 2 * plane) = l;
}
#endif

// hi = trunc_tf32(x), lo = x - hi (exact), elementwise over n values.
cudaError_t split_tf32(const float* x, float* hi, float* lo, int64_t n, cudaStream_t stream);

// Householder QR (explicit Q) of `batch` contiguous n x n matrices (n a multiple of 4).
// Workspace of qr_q / qr_q_t; `lookahead` adds the buffers of the two-stream schedule.
size_t qr_workspace_bytes(int n, int batch, bool lookahead = false);
// P read only; Q written. Uses the tensor-core QR on P^T (staged in the workspace).
cudaError_t qr_q(int n, int batch, const float* P, float* Q, uint8_t* skip, float tol,
                 void* workspace, size_t workspace_bytes, int* status, cudaStream_t stream);
// Where the factored matrix P^T must be placed before qr_q_t.
void qr_input_buffers(void* workspace, int n, int batch, float** At);
// QR of P whose transpose is already in qr_input_buffers(). Leaves Q^T in the workspace, contiguous
// at *Qt (if given), and, if Q is given, writes Q.
// The look-ahead schedule of qr_q_t: a second (low-priority) stream and its events.
struct QrLookahead {
  cudaStream_t far;     // trailing updates beyond the next block, and the Q accumulation's factors
  cudaEvent_t vt;       // this block's V T^T and the next block's rows are ready (caller's stream)
  cudaEvent_t far_done; // the far update of the previous block is done (recorded on `far`)
  cudaEvent_t vq[2];    // what the Q accumulation needs of the block using buffer 0 / 1 is done (on `far`)
};
// With `la` (all members set, and a workspace sized with lookahead) the trailing update of each
// 128-column block, except the next block's rows, and the block's part of the Q accumulation's
// factors run on la->far and overlap the next block's panels; everything is joined back on `stream` before return.
cudaError_t qr_q_t(int n, int batch, float* Q, uint8_t* skip, float tol, void* workspace, size_t workspace_bytes,
                   int* status, cudaStream_t stream, const QrLookahead* la = nullptr, float** Qt = nullptr);

// bf16 tensor-core product out_b = alpha A_b B_b^T + beta Cin_b (A_b M x K, B_b N x K, bf16
// row-major; fp32 accumulation). Outputs: out (bf16, ld, stride; Cin has the same layout) and, if
// given, out_t (bf16, transposed: element (r, c) at c * ld_t + r). M, N and K must be multiples of
// 8. `symmetric` promises a symmetric result (B = A, and Cin, if read, symmetric): one half of it
// is computed and mirrored.
struct Bf16Epilogue {
  __nv_bfloat16* out;
  int64_t ld, stride;
  const __nv_bfloat16* cin;
  __nv_bfloat16* out_t;
  int64_t ld_t, stride_t;
  float alpha, beta;
  int* status;
  bool symmetric;
};
cudaError_t gemm_bf16_nt(int M, int N, int K, int batch, const __nv_bfloat16* A, int64_t lda, int64_t a_stride,
                         const __nv_bfloat16* B, int64_t ldb, int64_t b_stride, const Bf16Epilogue& ep,
                         cudaStream_t stream);

// Muon's elementwise kernels (batched over `batch` rows x cols matrices of a class).
// M <- beta1 M + (1 - beta1) G and norm2[b] += ||M_b||_F^2 (norm2 zeroed by the caller);
// non-finite gradients set kStatusNonFinite.
cudaError_t muon_momentum(const float* const* grads, float* M, double* norm2, int64_t elems, int batch, float beta1,
                          int* status, cudaStream_t stream);
// X_0 = M / max(||M||_F, eps) in bf16, as X (r x c) and X^T (c x r) with (r, c) = (rows, cols),
// or, if `transposed`, (r, c) = (cols, rows) and X = M^T scaled.
cudaError_t muon_init_x(const float* M, const double* norm2, float eps, __nv_bfloat16* X, __nv_bfloat16* Xt,
                        int rows, int cols, int batch, bool transposed, cudaStream_t stream);
// W <- (1 - lr wd) W - lr scale O, O bf16 rows x cols.
cudaError_t muon_update(float* const* params, const __nv_bfloat16* O, int64_t elems, int batch, float lr, float wd,
                        float scale, cudaStream_t stream);

// Elementwise kernels of the step.
// M_hat <- b1 M_hat + (1-b1) G and Gc <- G for each matrix of a class.
cudaError_t momentum_and_copy(const float* const* grads, float* Gc, float* Mhat, int64_t elems,
                              int batch, float beta1, int* status, cudaStream_t stream);
// v <- b2 v + (1-b2) G'^2; N = m' / (sqrt(v) + eps) (bias-corrected if t > 0 given), written as
// the planes Np if given (cols a multiple of 4), else over Gp; guard rows/cols zeroed.
cudaError_t adam_in_basis(float* Gp, const float* Mp, float* V, int rows, int cols, int batch,
                          float beta1, float beta2, float eps, float bc1, float bc2,
                          const uint8_t* skipL, const uint8_t* skipR, const Planes& Np, int* status,
                          cudaStream_t s);
// Tensor-core operand preparation (rows and cols multiples of 4): the planes of G and of G^T, and
// the momentum EMA M_hat <- b1 M_hat + (1-b1) G in place, with its planes (Mc); M_hat is stored
// in G's orientation or (if mhat_transposed) as M_hat^T, and so are its planes.
cudaError_t momentum_split(const float* const* grads, const Planes& Gn, const Planes& Gt, const Planes& Mc, float* Mhat,
                           int rows, int cols, int batch, float beta1, bool mhat_transposed, int* status,
                           cudaStream_t stream);
// Packed symmetric storage: the lower-triangular 32 x 32 tiles of an n x n matrix, tile (I, J)
// (I >= J) at tile index I (I + 1) / 2 + J, each row-major; packed_floats(n) per matrix.
int64_t packed_floats(int n);
// F_b (full, n x n) and, if Fp is given, its planes from the packed tiles P_b.
cudaError_t unpack_sym(const float* P, float* F, const Planes& Fp, int n, int batch, cudaStream_t stream);
// P_b from the lower triangle of F_b.
cudaError_t pack_sym(const float* F, float* P, int n, int batch, cudaStream_t stream);
// Device pointer table written from a host array through kernel parameters (no host buffer
// has to outlive the call, and nothing waits on the host).
constexpr int kPtrChunk = 480;
struct PtrChunk {
  void* p[kPtrChunk];
};
cudaError_t put_ptrs(void** dst, void* const* src, int64_t n, cudaStream_t stream);
// dst_b = src_b^T for `batch` contiguous rows x cols matrices.
cudaError_t transpose(const float* src, float* dst, int rows, int cols, int batch, cudaStream_t stream);
// For `batch` n x n matrices X (n a multiple of 4), any output left out if null: the planes of X
// and of X^T, and X^T itself.
cudaError_t planes_transpose(const float* X, const Planes& Xp, const Planes& Xtp, float* Xt, int n, int batch,
                             cudaStream_t stream);
// The planes of `batch` rows x cols matrices with leading dimension ld, `stride` apart, or of their
// transposes, whose row i is scaled by d_i (at b * d_stride + i) if d is given; with tri > 0 the
// tri x tri blocks left of the diagonal ones are taken as zero, whatever they hold (rows, cols and
// tri multiples of 4).
cudaError_t split_blocks(const float* X, int64_t ld, int64_t stride, bool transposed, const float* d, int64_t d_stride,
                         int tri, const Planes& Xp, int rows, int cols, int batch, cudaStream_t stream);
// The planes of `rows` contiguous rows of cols values (cols a multiple of 4).
cudaError_t split_planes(const float* X, const Planes& Xp, int64_t rows, int cols, cudaStream_t stream);
// W <- (1 - lr*wd) W - lr * D (both sides identity).
cudaError_t weight_update(float* const* params, const float* D, int64_t elems, int batch,
                          float lr, float wd, cudaStream_t stream);
// KL-Shampoo factor form: lam[b][i] = sum_k C[b][i][k] Qt[b][i][k], the diagonal of Q^T F Q
// from C = Q^T F and the planes of Q^T (n a multiple of 4).
cudaError_t diag_dot(const float* C, const Planes& Qt, float* lam, int n, int batch, cudaStream_t stream);
// The planes of X[b][:, j] * sqrt(coef / (max(lam[b][j], 0) + eps)) (cols a multiple of 4).
cudaError_t scale_cols_split(const float* X, const Planes& Xp, const float* lam, int rows, int cols, int batch,
                             float coef, float eps, cudaStream_t stream);
// Sets `batch` n x n matrices to the identity.
cudaError_t set_identity(float* Q, int n, int batch, cudaStream_t stream);

}  // namespace soap
