// Elementwise parts of the SOAP step (HBM-bound; grid-stride, float4 where aligned).
//
//  * momentum_and_copy: the first moment kept in the ORIGINAL basis,
//      M_hat <- beta1 M_hat + (1 - beta1) G,
//    which is Alg. 1's re-projection m <- Q_new^T (Q_old m Q_old^T) Q_new followed
//    by m <- beta1 m + (1 - beta1) Q_new^T G Q_new, written as M_hat = Q m Q^T
//    (exact for the square orthogonal Q of both sides). It also copies G into the
//    library's contiguous gradient arena and flags non-finite gradients.
//  * adam_in_basis: v <- beta2 v + (1 - beta2) G'^2 and N = m / (sqrt(v) + eps)
//    (Alg. 1 "Calculate Adam update"; v is never re-projected), with the zero-column
//    guard.
//  * weight_update: W <- (1 - lr wd) W - lr N for a matrix with no preconditioned
//    side (Alg. 1 "Weight decay and update" with Q_L = Q_R = I).
//  * diag_dot, scale_cols_split: the KL-Shampoo factor form's approximate eigenvalues
//    lam = diag(Q^T F Q) and the column weights sqrt(coef / (lam + eps)) applied to G Q
//    (Alg. 1 "Accumulate Kronecker Factors (KL-Shampoo)").
#include <algorithm>

#include "profile.h"
#include "soap_internal.h"

namespace soap {
namespace {

constexpr int kThreads = 256;

// The tensor core reads an fp32 word as tf32 by dropping its 13 low mantissa bits, so
// an fp32 array serves directly as the "hi" operand. Its lo part is x - trunc(x) (exact
// in fp32) rounded to the nearest tf32, so that the tensor core's own truncation of it
// is exact and hi + lo is x to within half a tf32 unit of lo, without bias.
__device__ __forceinline__ float tf32_trunc(float x) { return __uint_as_float(__float_as_uint(x) & 0xFFFFE000u); }
__device__ __forceinline__ float lo_part(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x - tf32_trunc(x)));
  return __uint_as_float(r);
}

inline int blocks_for(int64_t elems, int batch) {
  int64_t want = (elems / 4 + kThreads - 1) / kThreads;
  if (want < 1) want = 1;
  // about 8 blocks of 256 threads per SM over the whole launch (152 SMs)
  const int64_t cap = std::max<int64_t>(4, (8 * 152) / std::max(1, batch));
  return (int)(want < cap ? want : cap);
}

__global__ void momentum_copy_kernel(const float* const* grads, float* Gc, float* Mh,
                                     int64_t elems, float beta1, int* status) {
  const int b = blockIdx.y;
  const float* g = grads[b];
  float* gc = Gc + (int64_t)b * elems;
  float* mh = Mh + (int64_t)b * elems;
  const float c1 = 1.f - beta1;
  int bad = 0;
  const bool vec = ((reinterpret_cast<uintptr_t>(g) | reinterpret_cast<uintptr_t>(gc) |
                     reinterpret_cast<uintptr_t>(mh)) & 15) == 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t start = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int64_t tail = 0;
  if (vec) {
    const int64_t n4 = elems / 4;
    for (int64_t i = start; i < n4; i += stride) {
      float4 x = reinterpret_cast<const float4*>(g)[i];
      float4 m = reinterpret_cast<float4*>(mh)[i];
      bad |= !isfinite(x.x) | !isfinite(x.y) | !isfinite(x.z) | !isfinite(x.w);
      m.x = fmaf(beta1, m.x, c1 * x.x);
      m.y = fmaf(beta1, m.y, c1 * x.y);
      m.z = fmaf(beta1, m.z, c1 * x.z);
      m.w = fmaf(beta1, m.w, c1 * x.w);
      reinterpret_cast<float4*>(gc)[i] = x;
      reinterpret_cast<float4*>(mh)[i] = m;
    }
    tail = n4 * 4;
  }
  for (int64_t i = tail + start; i < elems; i += stride) {
    const float x = g[i];
    bad |= !isfinite(x);
    mh[i] = fmaf(beta1, mh[i], c1 * x);
    gc[i] = x;
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(status, kStatusNonFinite);
}

// One Adam step in the basis for one element (v updated, N returned).
__device__ __forceinline__ float adam_one(float g, float m, float& v, float beta2, float c2, float eps, float inv_bc1,
                                          float inv_sqrt_bc2) {
  const float vn = fmaf(beta2, v, c2 * g * g);
  v = vn;
  return (m * inv_bc1) / (sqrtf(vn) * inv_sqrt_bc2 + eps);
}

// N goes to the planes Np if they are given (cols a multiple of 4 then), else over G'.
__global__ void adam_kernel(float* Gp, const float* Mp, float* V, int rows, int cols, float beta2,
                            float eps, float inv_bc1, float inv_sqrt_bc2, const uint8_t* skipL,
                            const uint8_t* skipR, Planes Np, int* status) {
  const int b = blockIdx.y;
  const int64_t elems = (int64_t)rows * cols;
  float* gp = Gp + (int64_t)b * elems;
  const float* mp = Mp + (int64_t)b * elems;
  float* v = V + (int64_t)b * elems;
  const uint8_t* sl = skipL ? skipL + (int64_t)b * rows : nullptr;
  const uint8_t* sr = skipR ? skipR + (int64_t)b * cols : nullptr;
  const float c2 = 1.f - beta2;
  int bad = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t start = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if ((cols & 3) == 0) {
    // four elements of one row per thread and step, 16-byte accesses (every matrix of the
    // arena starts on a 16-byte boundary when cols is a multiple of 4)
    for (int64_t i4 = start; i4 < elems / 4; i4 += stride) {
      const float4 g = reinterpret_cast<const float4*>(gp)[i4];
      const float4 m = reinterpret_cast<const float4*>(mp)[i4];
      float4 vv = reinterpret_cast<const float4*>(v)[i4];
      float4 o;
      o.x = adam_one(g.x, m.x, vv.x, beta2, c2, eps, inv_bc1, inv_sqrt_bc2);
      o.y = adam_one(g.y, m.y, vv.y, beta2, c2, eps, inv_bc1, inv_sqrt_bc2);
      o.z = adam_one(g.z, m.z, vv.z, beta2, c2, eps, inv_bc1, inv_sqrt_bc2);
      o.w = adam_one(g.w, m.w, vv.w, beta2, c2, eps, inv_bc1, inv_sqrt_bc2);
      const int row = (int)(4 * i4 / cols), col = (int)(4 * i4 - (int64_t)row * cols);
      if (sl || sr) {
        if (sl && sl[row]) o = make_float4(0.f, 0.f, 0.f, 0.f);
        if (sr) {
          if (sr[col]) o.x = 0.f;
          if (sr[col + 1]) o.y = 0.f;
          if (sr[col + 2]) o.z = 0.f;
          if (sr[col + 3]) o.w = 0.f;
        }
      }
      bad |= !isfinite(o.x) | !isfinite(o.y) | !isfinite(o.z) | !isfinite(o.w);
      reinterpret_cast<float4*>(v)[i4] = vv;
      if (Np.p) b3_store4(Np.p + b * Np.stride + row * Np.ld + col, Np.plane, o);
      else reinterpret_cast<float4*>(gp)[i4] = o;
    }
  } else {
    for (int64_t i = start; i < elems; i += stride) {
      float vi = v[i];
      float nv = adam_one(gp[i], mp[i], vi, beta2, c2, eps, inv_bc1, inv_sqrt_bc2);
      v[i] = vi;
      if ((sl && sl[i / cols]) || (sr && sr[i % cols])) nv = 0.f;
      bad |= !isfinite(nv);
      gp[i] = nv;
    }
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(status, kStatusNonFinite);
}

__global__ void weight_update_kernel(float* const* params, const float* D, int64_t elems, float lr,
                                     float wd) {
  const int b = blockIdx.y;
  float* w = params[b];
  const float* d = D + (int64_t)b * elems;
  const float keep = 1.f - lr * wd;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < elems; i += stride)
    w[i] = fmaf(keep, w[i], -lr * d[i]);
}

__global__ void identity_kernel(float* Q, int n) {
  const int b = blockIdx.y;
  float* q = Q + (int64_t)b * n * n;
  const int64_t nn = (int64_t)n * n;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nn; i += stride)
    q[i] = (i / n == i % n) ? 1.f : 0.f;
}


// A 64 x 32 tile's work: 256 threads, four consecutive elements of a row each, two rows per thread
// going in, and the same of the transposed tile coming out, so that both orientations are read and
// written in 16-byte (planes: 8-byte) units. rows and cols are multiples of 4.
constexpr int kTr = 64, kTc = 32;
struct TileIn {
  int r, c;  // row, first column inside the tile
  __device__ TileIn(int i) : r((threadIdx.x >> 3) + 32 * i), c(4 * (threadIdx.x & 7)) {}
};
struct TileOut {
  int c, r;  // row of the transpose (a column of the tile), first column of it
  __device__ TileOut(int i) : c((threadIdx.x >> 4) + 16 * i), r(4 * (threadIdx.x & 15)) {}
};
struct TileBuf {
  float v[kTr][kTc + 1];
  __device__ void put(const TileIn& t, float4 x) {
    v[t.r][t.c] = x.x;
    v[t.r][t.c + 1] = x.y;
    v[t.r][t.c + 2] = x.z;
    v[t.r][t.c + 3] = x.w;
  }
  __device__ float4 get(const TileOut& t) const {
    return make_float4(v[t.r][t.c], v[t.r + 1][t.c], v[t.r + 2][t.c], v[t.r + 3][t.c]);
  }
};
__device__ __forceinline__ bool bad4(float4 x) {
  return !isfinite(x.x) | !isfinite(x.y) | !isfinite(x.z) | !isfinite(x.w);
}
__device__ __forceinline__ float4 ema4(float beta, float4 m, float c1, float4 x) {
  return make_float4(fmaf(beta, m.x, c1 * x.x), fmaf(beta, m.y, c1 * x.y), fmaf(beta, m.z, c1 * x.z),
                     fmaf(beta, m.w, c1 * x.w));
}

// One 64 x 32 tile of one matrix per block. Reads G and writes the tensor-core operands into the
// step's workspace, as planes: G, G^T, and the momentum EMA M_hat <- b1 M_hat + (1-b1) G, stored
// back into the optimizer state (Mh) and written beside G (or G^T, if M_hat is kept transposed:
// the working orientation of a matrix preconditioned on its left side only), so that one batched
// product rotates both. Bound by memory: 12 bytes an element of gradient and state, 18 of planes.
template <bool MT>
__global__ void __launch_bounds__(256) momentum_split_kernel(const float* const* grads, Planes Gn, Planes Gt, Planes Mc,
                                                             float* Mh, int rows, int cols, float beta1, int* status) {
  __shared__ TileBuf tile;
  const int b = blockIdx.z;
  const int r0 = blockIdx.y * kTr, c0 = blockIdx.x * kTc;
  const int64_t mn = (int64_t)rows * cols;
  const float* g = grads[b];
  const float c1 = 1.f - beta1;
  int bad = 0;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const TileIn t(i);
    const int r = r0 + t.r, c = c0 + t.c;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < rows && c < cols) {
      x = *reinterpret_cast<const float4*>(g + (int64_t)r * cols + c);
      bad |= bad4(x);
      b3_store4(Gn.p + b * Gn.stride + r * Gn.ld + c, Gn.plane, x);
      if (!MT) {
        float4* mp = reinterpret_cast<float4*>(Mh + b * mn + (int64_t)r * cols + c);
        const float4 m = ema4(beta1, *mp, c1, x);
        *mp = m;
        b3_store4(Mc.p + b * Mc.stride + r * Mc.ld + c, Mc.plane, m);
      }
    }
    tile.put(t, x);
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const TileOut t(i);
    const int c = c0 + t.c, r = r0 + t.r;  // G^T[c][r]
    if (r < rows && c < cols) {
      const float4 x = tile.get(t);
      b3_store4(Gt.p + b * Gt.stride + c * Gt.ld + r, Gt.plane, x);
      if (MT) {
        float4* mp = reinterpret_cast<float4*>(Mh + b * mn + (int64_t)c * rows + r);
        const float4 m = ema4(beta1, *mp, c1, x);
        *mp = m;
        b3_store4(Mc.p + b * Mc.stride + c * Mc.ld + r, Mc.plane, m);
      }
    }
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(status, kStatusNonFinite);
}

// Packed symmetric storage of an n x n factor: only its lower-triangular 32 x 32 tiles, tile
// (I, J) with I >= J at tile index I (I + 1) / 2 + J, each tile row-major; entries beyond n
// are zero. A diagonal tile is stored whole (its upper half mirrors its lower half).
__device__ __forceinline__ void tri_tile(int t, int& I, int& J) {
  int i = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
  while ((i + 1) * (i + 2) / 2 <= t) ++i;
  while (i * (i + 1) / 2 > t) --i;
  I = i;
  J = t - i * (i + 1) / 2;
}

// Full matrix (and, if Fp is given, its planes) from packed tiles: one lower tile per
// block (32 x 8 threads), written in place and, off the diagonal, mirrored through shared
// memory.
__global__ void unpack_sym_kernel(const float* P, float* F, Planes Fp, int n, int64_t packed) {
  __shared__ float tile[32][33];
  const int b = blockIdx.y;
  int I, J;
  tri_tile(blockIdx.x, I, J);
  const float* p = P + (int64_t)b * packed + (int64_t)blockIdx.x * 1024;
  float* f = F + (int64_t)b * n * n;
  for (int i = threadIdx.y; i < 32; i += 8) {
    const float x = p[i * 32 + threadIdx.x];
    tile[i][threadIdx.x] = x;
    const int r = I * 32 + i, c = J * 32 + threadIdx.x;
    if (r < n && c < n) {
      f[(int64_t)r * n + c] = x;
      if (Fp.p) b3_store(Fp.p + b * Fp.stride + r * Fp.ld + c, Fp.plane, x);
    }
  }
  if (I == J) return;  // uniform over the block
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int r = J * 32 + i, c = I * 32 + threadIdx.x;
    if (r < n && c < n) {
      const float x = tile[threadIdx.x][i];
      f[(int64_t)r * n + c] = x;
      if (Fp.p) b3_store(Fp.p + b * Fp.stride + r * Fp.ld + c, Fp.plane, x);
    }
  }
}

// Packed tiles from the lower triangle of a full matrix (the upper triangle is not read
// except inside diagonal tiles, where the lower half is mirrored over it).
__global__ void pack_sym_kernel(const float* F, float* P, int n, int64_t packed) {
  __shared__ float tile[32][33];
  const int b = blockIdx.y;
  int I, J;
  tri_tile(blockIdx.x, I, J);
  const float* f = F + (int64_t)b * n * n;
  float* p = P + (int64_t)b * packed + (int64_t)blockIdx.x * 1024;
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int r = I * 32 + i, c = J * 32 + threadIdx.x;
    tile[i][threadIdx.x] = (r < n && c < n) ? f[(int64_t)r * n + c] : 0.f;
  }
  if (I == J) __syncthreads();  // uniform over the block
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int j = threadIdx.x;
    p[i * 32 + j] = (I != J || i >= j) ? tile[i][j] : tile[j][i];
  }
}

// Writes n (<= kPtrChunk) device pointers handed over as a kernel parameter (the launch copies
// them, so the host array may be reused as soon as the launch call returns).
__global__ void put_ptrs_kernel(void** dst, PtrChunk c, int n) {
  const int i = threadIdx.x;
  if (i < n) dst[i] = c.p[i];
}

// dst_b = src_b^T for `batch` contiguous rows x cols matrices (32 x 32 tiles, 32 x 8 threads).
__global__ void transpose_kernel(const float* src, float* dst, int rows, int cols) {
  __shared__ float tile[32][33];
  const int b = blockIdx.z;
  const int64_t mn = (int64_t)rows * cols;
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int r = r0 + i, c = c0 + threadIdx.x;
    tile[i][threadIdx.x] = (r < rows && c < cols) ? src[(int64_t)b * mn + (int64_t)r * cols + c] : 0.f;
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int c = c0 + i, r = r0 + threadIdx.x;
    if (r < rows && c < cols) dst[(int64_t)b * mn + (int64_t)c * rows + r] = tile[threadIdx.x][i];
  }
}

// The planes of X^T, and of X if Xp is given, and X^T itself if Xt is given, for `batch` n x n
// matrices (n a multiple of 4), one 64 x 32 tile per block.
__global__ void __launch_bounds__(256) planes_transpose_kernel(const float* X, Planes Xp, Planes Xtp, float* Xt, int n) {
  __shared__ TileBuf tile;
  const int b = blockIdx.z;
  const int r0 = blockIdx.y * kTr, c0 = blockIdx.x * kTc;
  const int64_t nn = (int64_t)n * n;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const TileIn t(i);
    const int r = r0 + t.r, c = c0 + t.c;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < n && c < n) {
      x = *reinterpret_cast<const float4*>(X + b * nn + (int64_t)r * n + c);
      if (Xp.p) b3_store4(Xp.p + b * Xp.stride + r * Xp.ld + c, Xp.plane, x);
    }
    tile.put(t, x);
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const TileOut t(i);
    const int c = c0 + t.c, r = r0 + t.r;
    if (r < n && c < n) {
      const float4 x = tile.get(t);
      if (Xtp.p) b3_store4(Xtp.p + b * Xtp.stride + c * Xtp.ld + r, Xtp.plane, x);
      if (Xt) *reinterpret_cast<float4*>(Xt + b * nn + (int64_t)c * n + r) = x;
    }
  }
}

// lam[b][i] = sum_k C[b][i][k] Qt[b][i][k] = (Q^T F Q)_ii for C = Q^T F, Q^T as planes: one warp
// per row.
__global__ void diag_dot_kernel(const float* C, Planes Qt, float* lam, int n) {
  const int b = blockIdx.y;
  const int row = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (row >= n) return;
  const float4* c = reinterpret_cast<const float4*>(C + (int64_t)b * n * n + (int64_t)row * n);
  const __nv_bfloat16* q = Qt.p + b * Qt.stride + row * Qt.ld;
  float acc = 0.f;
  for (int k = lane; k < n / 4; k += 32) {
    const float4 x = c[k];
    float y[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int pl = 2; pl >= 0; --pl) {  // the smallest plane first
      const uint2 w = *reinterpret_cast<const uint2*>(q + pl * Qt.plane + 4 * k);
      const float2 lo = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162&>(w.x));
      const float2 hi = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162&>(w.y));
      y[0] += lo.x;
      y[1] += lo.y;
      y[2] += hi.x;
      y[3] += hi.y;
    }
    acc = fmaf(x.x, y[0], acc);
    acc = fmaf(x.y, y[1], acc);
    acc = fmaf(x.z, y[2], acc);
    acc = fmaf(x.w, y[3], acc);
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) lam[(int64_t)b * n + row] = acc;
}

// The planes of X[b][i][j] * sqrt(coef / (max(lam[b][j], 0) + eps)) (cols a multiple of 4).
__global__ void scale_cols_split_kernel(const float* X, Planes Xp, const float* lam, int rows, int cols, float coef,
                                        float eps) {
  const int b = blockIdx.y;
  const int64_t e4 = (int64_t)rows * cols / 4;
  const float4* x = reinterpret_cast<const float4*>(X + (int64_t)b * rows * cols);
  const float* l = lam + (int64_t)b * cols;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < e4; i += stride) {
    const int r = (int)(i * 4 / cols), j = (int)(i * 4 - (int64_t)r * cols);
    float4 v = x[i];
    v.x *= sqrtf(coef / (fmaxf(l[j], 0.f) + eps));
    v.y *= sqrtf(coef / (fmaxf(l[j + 1], 0.f) + eps));
    v.z *= sqrtf(coef / (fmaxf(l[j + 2], 0.f) + eps));
    v.w *= sqrtf(coef / (fmaxf(l[j + 3], 0.f) + eps));
    b3_store4(Xp.p + b * Xp.stride + r * Xp.ld + j, Xp.plane, v);
  }
}

// The planes of `rows` rows of cols values (cols a multiple of 4).
__global__ void split_planes_kernel(const float* X, Planes Xp, int64_t rows, int cols) {
  const int64_t e4 = rows * cols / 4, stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < e4; i += stride) {
    const int64_t r = i * 4 / cols, j = i * 4 - r * cols;
    b3_store4(Xp.p + r * Xp.ld + j, Xp.plane, reinterpret_cast<const float4*>(X)[i]);
  }
}

// 64 rows x 32 columns at a time: the planes as they are, or of the transpose, its rows scaled by d if
// given; with `tri` the blocks of `tri` rows and columns left of the diagonal ones are taken as zero.
__global__ void __launch_bounds__(256) split_blocks_kernel(const float* X, int64_t ld, int64_t stride,
                                                           bool transposed, const float* d, int64_t d_stride, int tri,
                                                           Planes Xp, int rows, int cols) {
  __shared__ TileBuf tile;
  const int b = blockIdx.z;
  const int r0 = blockIdx.y * kTr, c0 = blockIdx.x * kTc;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const TileIn t(i);
    const int r = r0 + t.r, c = c0 + t.c;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < rows && c < cols) {
      if (!tri || c / tri >= r / tri) x = *reinterpret_cast<const float4*>(X + b * stride + r * ld + c);
      if (!transposed) b3_store4(Xp.p + b * Xp.stride + r * Xp.ld + c, Xp.plane, x);
    }
    if (transposed) tile.put(t, x);
  }
  if (!transposed) return;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const TileOut t(i);
    const int c = c0 + t.c, r = r0 + t.r;
    if (r < rows && c < cols) {
      float4 x = tile.get(t);
      const float f = d ? d[b * d_stride + c] : 1.f;
      x.x *= f; x.y *= f; x.z *= f; x.w *= f;
      b3_store4(Xp.p + b * Xp.stride + c * Xp.ld + r, Xp.plane, x);
    }
  }
}

// hi (if given) and lo parts; with `vec` (every pointer 16-byte aligned) four values at a time,
// four units in flight per thread: bound by memory (12 bytes a value; 4-byte accesses took
// 47 us for 16.8 M values, these 36).
__global__ void __launch_bounds__(256) split_kernel(const float* x, float* hi, float* lo, int64_t n, bool vec) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (vec) {
    const int64_t n4 = n / 4;
    auto put = [&](int64_t u, float4 v) {
      if (hi)
        reinterpret_cast<float4*>(hi)[u] = make_float4(tf32_trunc(v.x), tf32_trunc(v.y), tf32_trunc(v.z), tf32_trunc(v.w));
      reinterpret_cast<float4*>(lo)[u] = make_float4(lo_part(v.x), lo_part(v.y), lo_part(v.z), lo_part(v.w));
    };
    const float4* x4 = reinterpret_cast<const float4*>(x);
    int64_t u = i;
    for (; u + 3 * stride < n4; u += 4 * stride) {
      float4 v[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = x4[u + e * stride];
#pragma unroll
      for (int e = 0; e < 4; ++e) put(u + e * stride, v[e]);
    }
    for (; u < n4; u += stride) put(u, x4[u]);
    i += 4 * n4;
  }
  for (; i < n; i += stride) {
    const float v = x[i];
    if (hi) hi[i] = tf32_trunc(v);
    lo[i] = lo_part(v);
  }
}

}  // namespace

cudaError_t momentum_split(const float* const* grads, const Planes& Gn, const Planes& Gt, const Planes& Mc, float* Mhat,
                           int rows, int cols, int batch, float beta1, bool mhat_transposed, int* status,
                           cudaStream_t s) {
  if (rows <= 0 || cols <= 0 || batch <= 0) return cudaSuccess;
  if (batch > 65535 || (rows + kTr - 1) / kTr > 65535 || ((rows | cols) & 3)) return cudaErrorInvalidValue;
  const double e = (double)rows * cols * batch;
  ProfScope prof(kFamElementwise, 3.0 * e, 30.0 * e, s);
  dim3 grid((cols + kTc - 1) / kTc, (rows + kTr - 1) / kTr, batch);
  if (mhat_transposed)
    momentum_split_kernel<true><<<grid, 256, 0, s>>>(grads, Gn, Gt, Mc, Mhat, rows, cols, beta1, status);
  else
    momentum_split_kernel<false><<<grid, 256, 0, s>>>(grads, Gn, Gt, Mc, Mhat, rows, cols, beta1, status);
  return cudaGetLastError();
}

int64_t packed_floats(int n) {
  const int64_t t = (n + 31) / 32;
  return t * (t + 1) / 2 * 1024;
}

cudaError_t unpack_sym(const float* P, float* F, const Planes& Fp, int n, int batch, cudaStream_t s) {
  if (n <= 0 || batch <= 0) return cudaSuccess;
  if (batch > 65535) return cudaErrorInvalidValue;
  const int64_t tiles = packed_floats(n) / 1024;
  const double e = (double)n * n * batch;
  ProfScope prof(kFamElementwise, 0.0, (2.0 + (Fp.p ? 10.0 : 4.0)) * e, s);
  unpack_sym_kernel<<<dim3((unsigned)tiles, batch), dim3(32, 8), 0, s>>>(P, F, Fp, n, packed_floats(n));
  return cudaGetLastError();
}

cudaError_t pack_sym(const float* F, float* P, int n, int batch, cudaStream_t s) {
  if (n <= 0 || batch <= 0) return cudaSuccess;
  if (batch > 65535) return cudaErrorInvalidValue;
  const int64_t tiles = packed_floats(n) / 1024;
  const double e = (double)n * n * batch;
  ProfScope prof(kFamElementwise, 0.0, 4.0 * e, s);
  pack_sym_kernel<<<dim3((unsigned)tiles, batch), dim3(32, 8), 0, s>>>(F, P, n, packed_floats(n));
  return cudaGetLastError();
}

cudaError_t put_ptrs(void** dst, void* const* src, int64_t n, cudaStream_t s) {
  for (int64_t i = 0; i < n; i += kPtrChunk) {
    PtrChunk c;
    const int k = (int)std::min<int64_t>(kPtrChunk, n - i);
    for (int j = 0; j < k; ++j) c.p[j] = src[i + j];
    ProfScope prof(kFamOther, 0.0, 8.0 * k, s);
    put_ptrs_kernel<<<1, 512, 0, s>>>(dst + i, c, k);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t transpose(const float* src, float* dst, int rows, int cols, int batch, cudaStream_t s) {
  if (rows <= 0 || cols <= 0 || batch <= 0) return cudaSuccess;
  if (batch > 65535 || (rows + 31) / 32 > 65535) return cudaErrorInvalidValue;
  ProfScope prof(kFamOther, 0.0, 8.0 * rows * (double)cols * batch, s);
  dim3 grid((cols + 31) / 32, (rows + 31) / 32, batch);
  transpose_kernel<<<grid, dim3(32, 8), 0, s>>>(src, dst, rows, cols);
  return cudaGetLastError();
}

cudaError_t planes_transpose(const float* X, const Planes& Xp, const Planes& Xtp, float* Xt, int n, int batch,
                             cudaStream_t s) {
  if (n <= 0 || batch <= 0) return cudaSuccess;
  if ((n & 3) || batch > 65535) return cudaErrorInvalidValue;
  const double e = (double)n * n * batch;
  ProfScope prof(kFamElementwise, 0.0, (4.0 + (Xp.p ? 6 : 0) + (Xtp.p ? 6 : 0) + (Xt ? 4 : 0)) * e, s);
  dim3 grid((n + kTc - 1) / kTc, (n + kTr - 1) / kTr, batch);
  planes_transpose_kernel<<<grid, 256, 0, s>>>(X, Xp, Xtp, Xt, n);
  return cudaGetLastError();
}

cudaError_t split_blocks(const float* X, int64_t ld, int64_t stride, bool transposed, const float* d, int64_t d_stride,
                         int tri, const Planes& Xp, int rows, int cols, int batch, cudaStream_t s) {
  if (rows <= 0 || cols <= 0 || batch <= 0) return cudaSuccess;
  if (((rows | cols | ld | stride | tri) & 3) || batch > 65535) return cudaErrorInvalidValue;
  ProfScope prof(kFamElementwise, 0.0, 10.0 * rows * cols * batch, s);
  const dim3 grid((cols + kTc - 1) / kTc, (rows + kTr - 1) / kTr, batch);
  split_blocks_kernel<<<grid, 256, 0, s>>>(X, ld, stride, transposed, d, d_stride, tri, Xp, rows, cols);
  return cudaGetLastError();
}

cudaError_t split_planes(const float* X, const Planes& Xp, int64_t rows, int cols, cudaStream_t s) {
  if (rows <= 0 || cols <= 0) return cudaSuccess;
  if (cols & 3) return cudaErrorInvalidValue;
  ProfScope prof(kFamElementwise, 0.0, 10.0 * rows * cols, s);
  split_planes_kernel<<<blocks_for(rows * cols, 1), kThreads, 0, s>>>(X, Xp, rows, cols);
  return cudaGetLastError();
}

cudaError_t split_tf32(const float* x, float* hi, float* lo, int64_t n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  ProfScope prof(kFamElementwise, 2.0 * n, 12.0 * n, s);
  const bool vec = ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(hi) | reinterpret_cast<uintptr_t>(lo)) & 15) == 0;
  const int64_t want = ((vec ? n / 4 : n) + kThreads - 1) / kThreads + 1;
  split_kernel<<<(int)std::min<int64_t>(want, vec ? 8 * 152 : 4096), kThreads, 0, s>>>(x, hi, lo, n, vec);
  return cudaGetLastError();
}

cudaError_t diag_dot(const float* C, const Planes& Qt, float* lam, int n, int batch, cudaStream_t s) {
  if (n <= 0 || batch <= 0) return cudaSuccess;
  if ((n & 3) || batch > 65535) return cudaErrorInvalidValue;
  const double e = (double)n * n * batch;
  ProfScope prof(kFamElementwise, 2.0 * e, 10.0 * e, s);
  diag_dot_kernel<<<dim3((n + 7) / 8, batch), 256, 0, s>>>(C, Qt, lam, n);
  return cudaGetLastError();
}

cudaError_t scale_cols_split(const float* X, const Planes& Xp, const float* lam, int rows, int cols, int batch,
                             float coef, float eps, cudaStream_t s) {
  const int64_t elems = (int64_t)rows * cols;
  if (elems <= 0 || batch <= 0) return cudaSuccess;
  if ((cols & 3) || batch > 65535) return cudaErrorInvalidValue;
  ProfScope prof(kFamElementwise, 4.0 * elems * batch, 10.0 * elems * batch, s);
  scale_cols_split_kernel<<<dim3(blocks_for(elems, batch), batch), kThreads, 0, s>>>(X, Xp, lam, rows, cols, coef,
                                                                                     eps);
  return cudaGetLastError();
}

cudaError_t momentum_and_copy(const float* const* grads, float* Gc, float* Mhat, int64_t elems,
                              int batch, float beta1, int* status, cudaStream_t s) {
  if (elems <= 0 || batch <= 0) return cudaSuccess;
  ProfScope prof(kFamElementwise, 3.0 * elems * batch, 16.0 * elems * batch, s);
  momentum_copy_kernel<<<dim3(blocks_for(elems, batch), batch), kThreads, 0, s>>>(grads, Gc, Mhat, elems,
                                                                                   beta1, status);
  return cudaGetLastError();
}

cudaError_t adam_in_basis(float* Gp, const float* Mp, float* V, int rows, int cols, int batch,
                          float beta1, float beta2, float eps, float bc1, float bc2,
                          const uint8_t* skipL, const uint8_t* skipR, const Planes& Np, int* status,
                          cudaStream_t s) {
  (void)beta1;
  const int64_t elems = (int64_t)rows * cols;
  if (elems <= 0 || batch <= 0) return cudaSuccess;
  if (Np.p && (cols & 3)) return cudaErrorInvalidValue;
  ProfScope prof(kFamElementwise, 8.0 * elems * batch, (Np.p ? 22.0 : 20.0) * elems * batch, s);
  adam_kernel<<<dim3(blocks_for(elems, batch), batch), kThreads, 0, s>>>(
      Gp, Mp, V, rows, cols, beta2, eps, 1.f / bc1, 1.f / sqrtf(bc2), skipL, skipR, Np, status);
  return cudaGetLastError();
}

cudaError_t weight_update(float* const* params, const float* D, int64_t elems, int batch, float lr,
                          float wd, cudaStream_t s) {
  if (elems <= 0 || batch <= 0) return cudaSuccess;
  ProfScope prof(kFamElementwise, 3.0 * elems * batch, 12.0 * elems * batch, s);
  weight_update_kernel<<<dim3(blocks_for(elems, batch), batch), kThreads, 0, s>>>(params, D, elems, lr, wd);
  return cudaGetLastError();
}

cudaError_t set_identity(float* Q, int n, int batch, cudaStream_t s) {
  if (n <= 0 || batch <= 0) return cudaSuccess;
  ProfScope prof(kFamOther, 0, 4.0 * n * n * batch, s);
  identity_kernel<<<dim3(blocks_for((int64_t)n * n, batch), batch), kThreads, 0, s>>>(Q, n);
  return cudaGetLastError();
}

}  // namespace soap
