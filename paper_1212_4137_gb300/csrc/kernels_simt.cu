// kernels_simt.cu -- layout preparation, start initialisation, the y-step, and the FP32
// CUDA-core contractions of one AM sweep (Algorithm 2): u = A x (dense or over the support of
// x) and v = A^T y.
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <algorithm>
#include <cstdint>

#include "block_util.cuh"
#include "spca_internal.cuh"
#include "sweep_bodies.cuh"

namespace spca {

// ------------------------------------------------------------------ layout preparation
__global__ void k_transpose_f32(const float *__restrict__ src, int64_t rows, int64_t cols,
                                int64_t lds, float *__restrict__ dst, int64_t ldd) {
  __shared__ float tile[32][33];
  const int64_t c0 = (int64_t)blockIdx.x * 32;
  // row blocks of 32 on grid y, strided: rows may exceed 32 x 65535 (the grid's y limit)
  for (int64_t r0 = (int64_t)blockIdx.y * 32; r0 < rows; r0 += (int64_t)gridDim.y * 32) {
    for (int k = threadIdx.y; k < 32; k += blockDim.y) {
      const int64_t r = r0 + k, c = c0 + threadIdx.x;
      tile[k][threadIdx.x] = (r < rows && c < cols) ? src[r * lds + c] : 0.0f;
    }
    __syncthreads();
    for (int k = threadIdx.y; k < 32; k += blockDim.y) {
      const int64_t c = c0 + k, r = r0 + threadIdx.x;  // dst row = src column
      if (c < cols && r < rows) dst[c * ldd + r] = tile[threadIdx.x][k];
    }
    __syncthreads();
  }
}

cudaError_t launch_transpose_f32(const float *src, int64_t rows, int64_t cols, int64_t lds,
                                 float *dst, int64_t ldd, cudaStream_t st) {
  const int64_t rb = (rows + 31) / 32;
  dim3 grid((unsigned)((cols + 31) / 32), (unsigned)(rb < 65535 ? rb : 65535));
  k_transpose_f32<<<grid, dim3(32, 8), 0, st>>>(src, rows, cols, lds, dst, ldd);
  return cudaGetLastError();
}

__global__ void k_convert_f64_f32(const double *__restrict__ src, int64_t rows, int64_t cols,
                                  int64_t lds, float *__restrict__ dst, int64_t ldd) {
  const int64_t total = rows * cols;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / cols, c = e - r * cols;
    dst[r * ldd + c] = (float)src[r * lds + c];
  }
}

cudaError_t launch_convert_f64_f32(const double *src, int64_t rows, int64_t cols, int64_t lds,
                                   float *dst, int64_t ldd, cudaStream_t st) {
  k_convert_f64_f32<<<1216, 256, 0, st>>>(src, rows, cols, lds, dst, ldd);
  return cudaGetLastError();
}

__global__ void k_copy_f32(const float *__restrict__ src, int64_t rows, int64_t cols, int64_t lds,
                           float *__restrict__ dst, int64_t ldd) {
  const int64_t total = rows * cols;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / cols, c = e - r * cols;
    dst[r * ldd + c] = src[r * lds + c];
  }
}

cudaError_t launch_copy_f32(const float *src, int64_t rows, int64_t cols, int64_t lds, float *dst,
                            int64_t ldd, cudaStream_t st) {
  k_copy_f32<<<1216, 256, 0, st>>>(src, rows, cols, lds, dst, ldd);
  return cudaGetLastError();
}

__global__ void k_check_finite(const float *__restrict__ a, int64_t rows, int64_t cols, int64_t ld,
                               int *flag) {
  const int64_t total = rows * cols;
  int bad = 0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / cols, c = e - r * cols;
    bad |= !isfinite(a[r * ld + c]);
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, 1);
}

cudaError_t launch_check_finite(const float *a, int64_t rows, int64_t cols, int64_t ld, int *flag,
                                cudaStream_t st) {
  k_check_finite<<<1216, 256, 0, st>>>(a, rows, cols, ld, flag);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ a1: start initialisation
// (start_init_body: sweep_bodies.cuh)
// block per start (or per listed slot)
__global__ void __launch_bounds__(256) k_start_init(const float *__restrict__ x0, int64_t ld0,
                                                    uint64_t key, int p, float *__restrict__ X,
                                                    int64_t ldX, StartState s, double gamma0,
                                                    const int *__restrict__ slot_list,
                                                    const int *__restrict__ slot_start,
                                                    const int *__restrict__ count) {
  __shared__ float redf[32];
  if (slot_list && (int)blockIdx.x >= *count) return;
  const int c = slot_list ? slot_list[blockIdx.x] : (int)blockIdx.x;   // the slot (row of X)
  const int64_t start = slot_list ? slot_start[c] : c;                 // the start it takes
  start_init_body(x0, ld0, key, p, X, ldX, s, gamma0, c, start, redf);
}

// key = mix(seed ^ mix(stream)), stream 5 = starts (same definition as the host generator)
uint64_t start_key(uint64_t seed) {
  auto mixh = [](uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
  };
  return mixh(seed ^ mixh(5ull));
}

cudaError_t launch_start_init(const float *x0, int64_t ld0, uint64_t seed, int r, int p, float *X,
                              int64_t ldX, StartState s, double gamma0, const int *slot_list,
                              const int *slot_start, const int *count, cudaStream_t st) {
  k_start_init<<<r, 256, 0, st>>>(x0, ld0, start_key(seed), p, X, ldX, s, gamma0, slot_list, slot_start, count);
  return cudaGetLastError();
}

// The starts of a solve or of a group's new members (start_pack_body: sweep_bodies.cuh), the CTA that
// finishes last making the first active list.
// One kernel reads x0, checks it, normalises it and writes what the first sweep reads; it replaces a
// copy of x0, a check, an in-place normalisation (three passes), row scales, a plane split and the
// active list.  Bound by HBM: 4 p bytes read and 4 p written per start (two FP16 planes, or FP32).
// 1024 starts, p = 20000, tensor cores: 48 us for the kernel (290 us for the launches it replaces and the
// copy).
__global__ void __launch_bounds__(1024) k_start_pack(const float *x0, int64_t ld0, uint64_t key, int p, float *X,
                                                    int64_t ldX, XPack pk, StartState s, double gamma0, int *flag,
                                                    int r, int *act, int *rank, Ctrl *ctrl) {
  __shared__ float redf[32];
  __shared__ unsigned redu[32];
  const int c = (int)blockIdx.x;
  start_pack_body(x0, ld0, key, p, X, ldX, pk, s, gamma0, flag, c, redf, redu);
  last_makes_active_list(r, s.status, nullptr, r, act, rank, ctrl, nullptr);
}

cudaError_t launch_start_pack(const float *x0, int64_t ld0, uint64_t seed, int r, int p, float *X, int64_t ldX,
                              XPack pk, StartState s, double gamma0, int *flag, int *act, int *rank, Ctrl *ctrl,
                              cudaStream_t st) {
  // seeded normals are FP64 work of the first 256 threads; few long starts: more threads for the packing
  const int threads = x0 && r <= 152 && p > 4096 ? 1024 : 256;
  k_start_pack<<<r, threads, 0, st>>>(x0, ld0, start_key(seed), p, X, ldX, pk, s, gamma0, flag, r, act, rank, ctrl);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ rows between leading dimensions
// cols floats of each row from src (lds apart) to dst (ldd apart), neither aligned beyond a float: a CTA per
// row and 4096 floats, a thread's 16 loads in flight.  Bound by memory; 1024 rows of 20011 floats 23 us,
// where a 2-D copy call took about 90.
constexpr int kCopyPer = 16;
__global__ void __launch_bounds__(256) k_copy_rows(const float *__restrict__ src, int64_t lds, float *__restrict__ dst,
                                                   int64_t ldd, int cols) {
  const float *s = src + (int64_t)blockIdx.y * lds;
  float *d = dst + (int64_t)blockIdx.y * ldd;
  const int64_t j0 = (int64_t)blockIdx.x * (256 * kCopyPer) + threadIdx.x;
  float v[kCopyPer];
#pragma unroll
  for (int k = 0; k < kCopyPer; ++k) v[k] = j0 + 256 * k < cols ? __ldg(s + j0 + 256 * k) : 0.0f;
#pragma unroll
  for (int k = 0; k < kCopyPer; ++k)
    if (j0 + 256 * k < cols) d[j0 + 256 * k] = v[k];
}

cudaError_t launch_copy_rows(const float *src, int64_t lds, float *dst, int64_t ldd, int64_t cols, int rows,
                             cudaStream_t st) {
  k_copy_rows<<<dim3((unsigned)((cols + 256 * kCopyPer - 1) / (256 * kCopyPer)), (unsigned)rows), 256, 0, st>>>(
      src, lds, dst, ldd, (int)cols);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ y-step (Table 3 S1, S2)
// (ystep_body: sweep_bodies.cuh)
// skip: the sweep's y is written by the gather kernel when *skip != 0; flags: the stream-K flags that
// the next contraction needs zeroed (null: none)
__device__ __forceinline__ void zero_flags(int *flags, int nflags) {
  if (flags && blockIdx.x == 0 && blockIdx.y == 0)
    for (int i = threadIdx.x; i < nflags; i += blockDim.x) flags[i] = 0;
}
__global__ void __launch_bounds__(256) k_ystep(int form, const float *__restrict__ U, int64_t ldu,
                                               int n, float *__restrict__ Y,
                                               __half *__restrict__ Ypl, int64_t pstride,
                                               const int *__restrict__ rank, StartState s,
                                               float *__restrict__ X, int64_t ldX, int p,
                                               const int *__restrict__ skip, int *flags, int nflags) {
  __shared__ float redf[32];
  zero_flags(flags, nflags);
  if (skip && *skip != 0) return;   // (the gather kernel has done it)
  ystep_body(form, U, ldu, n, Y, Ypl, pstride, rank, s, X, ldX, p, (int)blockIdx.x, redf);
}

// The same for long u (n > 2 kYChunk), where one CTA per start would be latency-bound: a CTA per
// chunk of kYChunk entries and start; L2 variance first sums u_i^2 per chunk (k_ystep_norm), then
// every CTA of the start adds the chunk sums in chunk order and writes its chunk of y.
__global__ void __launch_bounds__(256) k_ystep_norm(const float *__restrict__ U, int64_t ldu, int n, StartState s,
                                                    float *__restrict__ ysum) {
  __shared__ float redf[32];
  const int b = blockIdx.x, c = blockIdx.y;
  if (s.status[c] != ST_ACTIVE) return;
  const float *u = U + (int64_t)c * ldu;
  const int i0 = b * kYChunk + threadIdx.x, i1 = min(n, (b + 1) * kYChunk);
  constexpr int E = kYChunk / 256;   // a thread's entries, all loads in flight
  float v[E], part = 0.0f;
#pragma unroll
  for (int k = 0; k < E; ++k) v[k] = i0 + 256 * k < i1 ? u[i0 + 256 * k] : 0.0f;
#pragma unroll
  for (int k = 0; k < E; ++k) part = fmaf(v[k], v[k], part);
  const float t = block_sum_f(part, redf);
  if (threadIdx.x == 0) ysum[(int64_t)c * gridDim.x + b] = t;
}

__global__ void __launch_bounds__(256) k_ystep_apply(int form, const float *__restrict__ U, int64_t ldu, int n,
                                                     float *__restrict__ Y, __half *__restrict__ Ypl,
                                                     int64_t pstride, const int *__restrict__ rank, StartState s,
                                                     float *__restrict__ X, int64_t ldX, int p,
                                                     const float *__restrict__ ysum, int *flags, int nflags) {
  const int b = blockIdx.x, c = blockIdx.y, nch = gridDim.x;
  zero_flags(flags, nflags);
  // (the chunk-0 CTA alone may change the status below, and only when every CTA of the start
  // returns without writing: ||u||_2 = 0)
  if (s.status[c] != ST_ACTIVE) return;
  const float *u = U + (int64_t)c * ldu;
  float *y = Y ? Y + (int64_t)c * ldu : nullptr;
  __half *yp = Ypl ? Ypl + (int64_t)(rank ? rank[c] : c) * ldu : nullptr;
  const int i1 = min(n, (b + 1) * kYChunk);
  if (b == 0 && threadIdx.x == 0) s.iters[c] += 1;
  if (is_l1_var(form)) {
    for (int i = b * kYChunk + threadIdx.x; i < i1; i += blockDim.x) {
      const float yi = (u[i] >= 0.0f) ? 1.0f : -1.0f;
      if (y) y[i] = yi;
      if (yp) yp[i] = __float2half_rn(yi * kQScale);
    }
    return;
  }
  float tot = 0.0f;
  for (int q = 0; q < nch; ++q) tot += ysum[(int64_t)c * nch + q];
  if (tot == 0.0f) {
    if (b == 0) {
      float *x = X + (int64_t)c * ldX;
      for (int j = threadIdx.x; j < p; j += blockDim.x) x[j] = 0.0f;
      if (threadIdx.x == 0) {
        s.status[c] = SPCA_ST_DEGENERATE;
        s.nnz[c] = 0;
        s.F[c] = 0.0;
      }
    }
    return;
  }
  float hi, lo, inv;
  norm_and_inverse(tot, &hi, &lo, &inv);
  for (int i = b * kYChunk + threadIdx.x; i < i1; i += blockDim.x) {
    const float yi = u[i] * inv;
    if (y) y[i] = yi;
    if (yp) {
      const float ys = yi * kQScale;
      const __half hi = __float2half_rn(ys);
      yp[i] = hi;
      yp[i + pstride] = __float2half_rn(ys - __half2float(hi));
    }
  }
}

// The y-step of long u under L2 variance straight into the packed operand of the sparse product (see
// k_pack_t), y itself not being wanted: a CTA per 128 rows and 32 listed starts, y's bits those of
// k_ystep_apply.  Bound by the launch and two round trips; with the chunk norms before it 11 us for 20 starts
// of 40000 rows, where y-step and packing were three launches of 18 us.
__global__ void __launch_bounds__(256) k_ystep_pack(const float *__restrict__ U, int64_t ldu, int n,
                                                    const int *__restrict__ list, const int *__restrict__ count,
                                                    StartState s, float *__restrict__ X, int64_t ldX, int p,
                                                    const float *__restrict__ ysum, int nch, float *__restrict__ Bt,
                                                    int ldb) {
  constexpr int SUB = 4;
  __shared__ float tile[SUB][32][33], inv[32];
  __shared__ int start[32], zero[32];
  const int cnt = *count, k0 = blockIdx.y * 32;
  const int kpad = (cnt + kSpGroup - 1) / kSpGroup * kSpGroup;
  if (k0 >= kpad) return;
  const int tx = threadIdx.x, j00 = blockIdx.x * 32 * SUB;
  if (threadIdx.y == 0) {
    const int c = k0 + tx < cnt ? list[k0 + tx] : -1;
    float tot = 0.0f, hi, lo, iv = 0.0f;
    if (c >= 0) {
      for (int q = 0; q < nch; ++q) tot += ysum[(int64_t)c * nch + q];
      if (tot != 0.0f) norm_and_inverse(tot, &hi, &lo, &iv);
    }
    start[tx] = c;
    inv[tx] = iv;
    zero[tx] = c >= 0 && tot == 0.0f;
    if (c >= 0 && blockIdx.x == 0) {
      s.iters[c] += 1;
      if (tot == 0.0f) {
        s.status[c] = SPCA_ST_DEGENERATE;
        s.nnz[c] = 0;
        s.F[c] = 0.0;
      }
    }
  }
  __syncthreads();
  if (blockIdx.x == 0) {
    for (int q = 0; q < 32; ++q) {
      if (!zero[q]) continue;
      for (int j = threadIdx.y * 32 + tx; j < p; j += 256) X[(int64_t)start[q] * ldX + j] = 0.0f;
    }
  }
  float v[SUB][4];
#pragma unroll
  for (int b = 0; b < SUB; ++b)
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const int c = start[threadIdx.y + 8 * h], j = j00 + 32 * b + tx;
      v[b][h] = c >= 0 && j < n ? U[(int64_t)c * ldu + j] : 0.0f;
    }
#pragma unroll
  for (int b = 0; b < SUB; ++b)
#pragma unroll
    for (int h = 0; h < 4; ++h) tile[b][threadIdx.y + 8 * h][tx] = v[b][h] * inv[threadIdx.y + 8 * h];
  __syncthreads();
#pragma unroll
  for (int b = 0; b < SUB; ++b)
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const int j = j00 + 32 * b + threadIdx.y + 8 * h, k = k0 + tx;
      if (j < n && k < kpad) Bt[(int64_t)j * ldb + k] = tile[b][tx][threadIdx.y + 8 * h];
    }
}

cudaError_t launch_ystep_pack(const float *U, int64_t ldu, int n, int r, const int *list, const int *count,
                              StartState s, float *X, int64_t ldX, int p, float *ysum, float *Bt, int ldb,
                              cudaStream_t st) {
  const int nch = (n + kYChunk - 1) / kYChunk;
  k_ystep_norm<<<dim3((unsigned)nch, (unsigned)r), 256, 0, st>>>(U, ldu, n, s, ysum);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_ystep_pack<<<dim3((unsigned)((n + 127) / 128), (unsigned)((r + 31) / 32)), dim3(32, 8), 0, st>>>(
      U, ldu, n, list, count, s, X, ldX, p, ysum, nch, Bt, ldb);
  return cudaGetLastError();
}

cudaError_t launch_ystep(int form, const float *U, int64_t ldu, int n, int r, float *Y, void *Ypl,
                         int64_t plane_stride, const int *rank, StartState s, float *X, int64_t ldX,
                         int p, float *ysum, const int *skip, int *flags, int nflags, cudaStream_t st) {
  const int nch = (n + kYChunk - 1) / kYChunk;
  if (ysum && nch > 2) {   // (skip: not for such u, see ystep_with_gather)
    const dim3 grid((unsigned)nch, (unsigned)r);
    if (!is_l1_var(form)) {
      k_ystep_norm<<<grid, 256, 0, st>>>(U, ldu, n, s, ysum);
      cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) return e;
    }
    k_ystep_apply<<<grid, 256, 0, st>>>(form, U, ldu, n, Y, static_cast<__half *>(Ypl), plane_stride, rank, s, X,
                                        ldX, p, ysum, flags, nflags);
    return cudaGetLastError();
  }
  k_ystep<<<r, 256, 0, st>>>(form, U, ldu, n, Y, static_cast<__half *>(Ypl), plane_stride, rank,
                             s, X, ldX, p, skip, flags, nflags);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ active-start list
__global__ void __launch_bounds__(1024) k_active_list(const int *__restrict__ status, const int *__restrict__ nnz,
                                                      int r, int *__restrict__ act, int *__restrict__ rank,
                                                      Ctrl *__restrict__ ctrl, Ctrl *__restrict__ ctrl_read) {
  active_list_body(status, nnz, r, act, rank, ctrl);
  if (ctrl_read && threadIdx.x == 0) *ctrl_read = Ctrl{};
}

cudaError_t launch_active_list(const int *status, const int *nnz, int r, int *act, int *rank, Ctrl *c,
                               Ctrl *ctrl_read, cudaStream_t st) {
  k_active_list<<<1, 1024, 0, st>>>(status, nnz, r, act, rank, c, ctrl_read);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ FP32 CUDA-core GEMM
// C[m, j] = sum_k P[m, k] Q[j, k]; P (M x K) and Q (N x K) are both K-contiguous with
// leading dimensions that are multiples of 8 and zero pads, and K is a multiple of 8.
// 128 x 128 tile, 8-deep K slices, 256 threads with an 8 x 8 register block each; the
// next slice is prefetched into registers while the current one is multiplied.
namespace {
constexpr int BM = 128, BN = 128, BK = 8;
}

__global__ void __launch_bounds__(256) k_gemm_nt_f32(const float *__restrict__ P, int64_t ldp,
                                                     const float *__restrict__ Q, int64_t ldq,
                                                     float *__restrict__ C, int64_t ldc, int M,
                                                     int N, int K, const int *__restrict__ gate) {
  if (gate && *gate == 0) return;
  __shared__ __align__(16) float As[BK][BM + 4];
  __shared__ __align__(16) float Bs[BK][BN + 4];
  const int tid = threadIdx.x;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  // loader: thread -> (row, 4 consecutive k)
  const int lrow = tid >> 1, lk = (tid & 1) * 4;
  const bool pa = (m0 + lrow) < M, qa = (n0 + lrow) < N;
  const float *pp = P + (int64_t)(pa ? m0 + lrow : 0) * ldp + lk;
  const float *qp = Q + (int64_t)(qa ? n0 + lrow : 0) * ldq + lk;
  // compute: thread -> rows {ty*4..+3, 64+ty*4..+3}, cols {tx*4..+3, 64+tx*4..+3}
  const int ty = tid >> 4, tx = tid & 15;
  float acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.0f;

  float4 ra = pa ? *reinterpret_cast<const float4 *>(pp) : make_float4(0, 0, 0, 0);
  float4 rb = qa ? *reinterpret_cast<const float4 *>(qp) : make_float4(0, 0, 0, 0);
  for (int k0 = 0; k0 < K; k0 += BK) {
    __syncthreads();
    As[lk + 0][lrow] = ra.x; As[lk + 1][lrow] = ra.y; As[lk + 2][lrow] = ra.z; As[lk + 3][lrow] = ra.w;
    Bs[lk + 0][lrow] = rb.x; Bs[lk + 1][lrow] = rb.y; Bs[lk + 2][lrow] = rb.z; Bs[lk + 3][lrow] = rb.w;
    __syncthreads();
    if (k0 + BK < K) {
      ra = pa ? *reinterpret_cast<const float4 *>(pp + k0 + BK) : make_float4(0, 0, 0, 0);
      rb = qa ? *reinterpret_cast<const float4 *>(qp + k0 + BK) : make_float4(0, 0, 0, 0);
    }
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4 *>(&As[kk][ty * 4]);
      const float4 a1 = *reinterpret_cast<const float4 *>(&As[kk][64 + ty * 4]);
      const float4 b0 = *reinterpret_cast<const float4 *>(&Bs[kk][tx * 4]);
      const float4 b1 = *reinterpret_cast<const float4 *>(&Bs[kk][64 + tx * 4]);
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int m = m0 + ((i < 4) ? ty * 4 + i : 64 + ty * 4 + (i - 4));
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int nn = n0 + ((j < 4) ? tx * 4 + j : 64 + tx * 4 + (j - 4));
      if (nn < N) C[(int64_t)m * ldc + nn] = acc[i][j];
    }
  }
}

// The same for products too small to fill the chip with 128 x 128 tiles (few starts, or one short
// side): 16 x 32 tiles, each with its K range split over `split` CTAs so that the launch has about two
// CTAs per SM.  128 threads; slices of 64 K entries of both operands in shared memory (the next one
// prefetched into registers); a thread adds 4 starts of one column, one 16-byte broadcast and one
// 4-byte read per 4 FMAs.  The CTA that finishes a tile last adds its parts in K order, so the result
// does not depend on the timing.  Bound by latency (a few L2 round trips and barriers).
// 16 starts, ncu, against 128 x 128 tiles: u, 400 x 4000, 595 -> 12 us; v, 4000 x 400, 67 -> 7 us.
namespace {
constexpr int FM = 16, FN = 32, FK = 64, FTH = 128;
}
__global__ void __launch_bounds__(FTH) k_gemm_few(const float *__restrict__ P, int64_t ldp,
                                                  const float *__restrict__ Q, int64_t ldq, float *__restrict__ C,
                                                  int64_t ldc, int M, int N, int K, int kslices,
                                                  const int *__restrict__ gate, float *parts, int *cnt) {
  if (gate && *gate == 0) return;
  __shared__ __align__(16) float Ps[FK][FM];
  __shared__ float Qs[FK][FN + 1];
  __shared__ int last;
  const int tid = threadIdx.x, n0 = blockIdx.x * FN, m0 = blockIdx.y * FM;
  const int split = gridDim.z, z = blockIdx.z;
  const int k0 = z * kslices * FK, k1 = min(K, k0 + kslices * FK);   // (K and the slices: multiples of 8)
  const int mq = (tid >> 5) * 4, nj = tid & 31;   // this thread's starts mq .. mq + 3, column nj
  float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  // loads of one slice: 16 entries of Q (4 vectors: row q, 16-byte column v) and 8 of P per thread
  float4 rq[4], rp[2];
  auto load = [&](int k) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = tid + u * FTH, row = e >> 4, kk = k + (e & 15) * 4;
      rq[u] = n0 + row < N && kk < k1 ? __ldg(reinterpret_cast<const float4 *>(Q + (int64_t)(n0 + row) * ldq + kk))
                                      : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {   // (rows fastest: the stores below meet few bank conflicts)
      const int e = tid + u * FTH, row = e & 15, kk = k + (e >> 4) * 4;
      rp[u] = m0 + row < M && kk < k1 ? __ldg(reinterpret_cast<const float4 *>(P + (int64_t)(m0 + row) * ldp + kk))
                                      : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  load(k0);
  for (int k = k0; k < k1; k += FK) {
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = tid + u * FTH, row = e >> 4, kk = (e & 15) * 4;
      Qs[kk][row] = rq[u].x; Qs[kk + 1][row] = rq[u].y; Qs[kk + 2][row] = rq[u].z; Qs[kk + 3][row] = rq[u].w;
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int e = tid + u * FTH, row = e & 15, kk = (e >> 4) * 4;
      Ps[kk][row] = rp[u].x; Ps[kk + 1][row] = rp[u].y; Ps[kk + 2][row] = rp[u].z; Ps[kk + 3][row] = rp[u].w;
    }
    __syncthreads();
    if (k + FK < k1) load(k + FK);
#pragma unroll 16
    for (int kk = 0; kk < FK; ++kk) {
      const float4 p4 = *reinterpret_cast<const float4 *>(&Ps[kk][mq]);
      const float q = Qs[kk][nj];
      acc[0] = fmaf(p4.x, q, acc[0]);
      acc[1] = fmaf(p4.y, q, acc[1]);
      acc[2] = fmaf(p4.z, q, acc[2]);
      acc[3] = fmaf(p4.w, q, acc[3]);
    }
  }
  if (split > 1) {
    const int tile = blockIdx.y * gridDim.x + blockIdx.x;
    float *mine = parts + ((int64_t)tile * split + z) * (FM * FN);
#pragma unroll
    for (int q = 0; q < 4; ++q) __stcg(mine + (mq + q) * FN + nj, acc[q]);
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      int before;
      asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(before) : "l"(cnt + tile) : "memory");
      last = before == split - 1;
      if (last) cnt[tile] = 0;
    }
    __syncthreads();
    if (!last) return;
    const float *all = parts + (int64_t)tile * split * (FM * FN) + mq * FN + nj;
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q] = 0.0f;
    for (int s = 0; s < split; ++s)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] += __ldcg(all + (int64_t)s * (FM * FN) + q * FN);
  }
  if (n0 + nj < N)
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (m0 + mq + q < M) C[(int64_t)(m0 + mq + q) * ldc + n0 + nj] = acc[q];
}

// scratch of k_gemm_few: parts only of launches with fewer than 2 CTAs per SM before the split
int64_t gemm_few_floats(int sms) { return (int64_t)4 * sms * FM * FN; }
int gemm_few_tiles(int sms) { return 2 * sms; }

// The 128 x 128 tiles run near the FP32 peak once there are enough of them; the small ones do half as
// many FMAs per shared-memory read.  So they take products below 2^27 multiply-adds (AUTO's CUDA-core
// range ends at 2^26), and larger ones while the large tiles would leave SMs idle.
cudaError_t launch_gemm_nt_f32(const float *P, int64_t ldp, const float *Q, int64_t ldq, float *C,
                               int64_t ldc, int M, int N, int K, const int *gate, float *parts, int *cnt, int sms,
                               cudaStream_t st) {
  dim3 grid((unsigned)((N + BN - 1) / BN), (unsigned)((M + BM - 1) / BM));
  const int64_t work = (int64_t)M * N * K;
  const int64_t fm = (M + FM - 1) / FM, fn = (N + FN - 1) / FN, slices = (K + FK - 1) / FK;
  if (parts && fm <= 65535 && (work < (int64_t(1) << 27) || (int64_t)grid.x * grid.y < sms)) {
    // about two CTAs per SM, at least two slices each
    int64_t split = 1;
    if (fm * fn < 2 * (int64_t)sms) split = std::max<int64_t>(1, std::min(4 * (int64_t)sms / (fm * fn), (slices + 1) / 2));
    const int64_t per = (slices + split - 1) / split;
    split = (slices + per - 1) / per;
    k_gemm_few<<<dim3((unsigned)fn, (unsigned)fm, (unsigned)split), FTH, 0, st>>>(P, ldp, Q, ldq, C, ldc, M, N, K,
                                                                                 (int)per, gate, parts, cnt);
    return cudaGetLastError();
  }
  k_gemm_nt_f32<<<grid, 256, 0, st>>>(P, ldp, Q, ldq, C, ldc, M, N, K, gate);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ u = A x over supp(x)
// U[c, i] = sum_t val[c, t] AT[idx[c, t], i] (t over the support of x, ascending index).
// Runs only when *gate != 0 (the control word chose this path for the sweep).
// Grid: x over the starts, y over row blocks of 512 (128 threads), so the CTAs in flight share a
// few row blocks: their slices of the columns in the starts' supports (512 rows x 4 bytes each;
// 37 MB per row block for 18,000 distinct columns) stay in L2, and a column used by several
// starts is read from DRAM about once.
constexpr int kGatherThreads = 128;
// rows 4 (yb kGatherThreads + t) .. + 3 of u = A x for start c (block of kGatherThreads threads)
__device__ void gather_body(const float *__restrict__ AT, int64_t ldat, int n, const int *__restrict__ sup_idx,
                            const float *__restrict__ sup_val, int cap, StartState s, float *__restrict__ U,
                            int64_t ldu, int c, int yb, int *sidx, float *sval) {
  if (s.status[c] != ST_ACTIVE) return;
  if (s.iters[c] == 0) return;   // a start not swept yet has a dense x: the dense contraction
  const int nnz = s.nnz[c];
  // four consecutive rows per thread, read as one 16-byte vector (ldat is a multiple of 8, so
  // the rows up to the padded width are in bounds); eight columns' loads are issued before
  // their FMAs, which still run in support order
  const int i4 = (yb * kGatherThreads + threadIdx.x) * 4;
  const int *gi = sup_idx + (int64_t)c * cap;
  const float *gv = sup_val + (int64_t)c * cap;
  float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  auto step = [&](float xv, float4 a) {
    acc.x = fmaf(xv, a.x, acc.x);
    acc.y = fmaf(xv, a.y, acc.y);
    acc.z = fmaf(xv, a.z, acc.z);
    acc.w = fmaf(xv, a.w, acc.w);
  };
  for (int t0 = 0; t0 < nnz; t0 += kGatherThreads) {
    __syncthreads();
    if (t0 + (int)threadIdx.x < nnz) {
      sidx[threadIdx.x] = gi[t0 + threadIdx.x];
      sval[threadIdx.x] = gv[t0 + threadIdx.x];
    }
    __syncthreads();
    const int m = min(kGatherThreads, nnz - t0);
    if (i4 < n) {
      const float *base = AT + i4;
      int t = 0;
      for (; t + 8 <= m; t += 8) {
        float4 a[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) a[q] = __ldg(reinterpret_cast<const float4 *>(base + (int64_t)sidx[t + q] * ldat));
#pragma unroll
        for (int q = 0; q < 8; ++q) step(sval[t + q], a[q]);
      }
      for (; t < m; ++t) step(sval[t], __ldg(reinterpret_cast<const float4 *>(base + (int64_t)sidx[t] * ldat)));
    }
  }
  float *u = U + (int64_t)c * ldu;
  if (i4 < n) u[i4] = acc.x;
  if (i4 + 1 < n) u[i4 + 1] = acc.y;
  if (i4 + 2 < n) u[i4 + 2] = acc.z;
  if (i4 + 3 < n) u[i4 + 3] = acc.w;
}

// gather_body over the leading FP16 plane of A^T (a resident 16-bit handle): row j of the plane
// is A[:, j] times its power-of-two scale, undone by folding at_inv[j] into x_j (exact); four rows
// per thread as one 8-byte load, products and sums in FP32 in support order
__device__ void gather_lowp_body(const __half *__restrict__ AT0, const float *__restrict__ at_inv, int64_t ldat,
                                 int n, const int *__restrict__ sup_idx, const float *__restrict__ sup_val, int cap,
                                 StartState s, float *__restrict__ U, int64_t ldu, int c, int yb, int *sidx,
                                 float *sval) {
  if (s.status[c] != ST_ACTIVE) return;
  if (s.iters[c] == 0) return;   // a start not swept yet has a dense x: the dense contraction
  const int nnz = s.nnz[c];
  const int i4 = (yb * kGatherThreads + threadIdx.x) * 4;
  const int *gi = sup_idx + (int64_t)c * cap;
  const float *gv = sup_val + (int64_t)c * cap;
  float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  auto step = [&](float xv, uint2 raw) {
    const __half2 *h2 = reinterpret_cast<const __half2 *>(&raw);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const float2 f = __half22float2(h2[q]);
      acc[2 * q] = fmaf(xv, f.x, acc[2 * q]);
      acc[2 * q + 1] = fmaf(xv, f.y, acc[2 * q + 1]);
    }
  };
  for (int t0 = 0; t0 < nnz; t0 += kGatherThreads) {
    __syncthreads();
    if (t0 + (int)threadIdx.x < nnz) {
      const int j = gi[t0 + threadIdx.x];
      sidx[threadIdx.x] = j;
      sval[threadIdx.x] = gv[t0 + threadIdx.x] * at_inv[j];
    }
    __syncthreads();
    const int m = min(kGatherThreads, nnz - t0);
    if (i4 < n) {
      const __half *base = AT0 + i4;
      int t = 0;
      for (; t + 8 <= m; t += 8) {
        uint2 a[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) a[q] = __ldg(reinterpret_cast<const uint2 *>(base + (int64_t)sidx[t + q] * ldat));
#pragma unroll
        for (int q = 0; q < 8; ++q) step(sval[t + q], a[q]);
      }
      for (; t < m; ++t) step(sval[t], __ldg(reinterpret_cast<const uint2 *>(base + (int64_t)sidx[t] * ldat)));
    }
  }
  float *u = U + (int64_t)c * ldu;
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (i4 + q < n) u[i4 + q] = acc[q];
}

// The same gather over the FP8 E4M3 copy of A^T (the low-precision sweeps of an FP8 handle): row j
// is A[:, j] times its scale, undone with at8_inv[j] folded into x_j; 16 rows per thread as one
// 16-byte load, products and sums in FP32 in support order.
__global__ void __launch_bounds__(256) k_gemm1_sparse_f8(const uint8_t *__restrict__ AT8, int64_t ldat,
                                                         const float *__restrict__ at_inv, int n,
                                                         const int *__restrict__ sup_idx,
                                                         const float *__restrict__ sup_val, int cap, StartState s,
                                                         float *__restrict__ U, int64_t ldu,
                                                         const int *__restrict__ gate) {
  if (*gate == 0) return;
  const int c = blockIdx.x;
  if (s.status[c] != ST_ACTIVE) return;
  __shared__ int sidx[256];
  __shared__ float sval[256];
  const int nnz = s.nnz[c];
  const int i16 = (blockIdx.y * blockDim.x + threadIdx.x) * 16;
  const int *gi = sup_idx + (int64_t)c * cap;
  const float *gv = sup_val + (int64_t)c * cap;
  float acc[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) acc[q] = 0.0f;
  auto step = [&](float xv, uint4 raw) {
    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const __half2_raw hr = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)(w[q] >> (16 * h)), __NV_E4M3);
        const float2 f = __half22float2(__half2(hr));
        acc[4 * q + 2 * h] = fmaf(xv, f.x, acc[4 * q + 2 * h]);
        acc[4 * q + 2 * h + 1] = fmaf(xv, f.y, acc[4 * q + 2 * h + 1]);
      }
    }
  };
  for (int t0 = 0; t0 < nnz; t0 += 256) {
    __syncthreads();
    if (t0 + (int)threadIdx.x < nnz) {
      const int j = gi[t0 + threadIdx.x];
      sidx[threadIdx.x] = j;
      sval[threadIdx.x] = gv[t0 + threadIdx.x] * at_inv[j];
    }
    __syncthreads();
    const int m = min(256, nnz - t0);
    if (i16 < n) {
      const uint8_t *base = AT8 + i16;
      int t = 0;
      for (; t + 8 <= m; t += 8) {
        uint4 a[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) a[q] = __ldg(reinterpret_cast<const uint4 *>(base + (int64_t)sidx[t + q] * ldat));
#pragma unroll
        for (int q = 0; q < 8; ++q) step(sval[t + q], a[q]);
      }
      for (; t < m; ++t) step(sval[t], __ldg(reinterpret_cast<const uint4 *>(base + (int64_t)sidx[t] * ldat)));
    }
  }
  float *u = U + (int64_t)c * ldu;
#pragma unroll
  for (int q = 0; q < 16; ++q)
    if (i16 + q < n) u[i16 + q] = acc[q];
}

cudaError_t launch_gemm1_sparse_f8(const uint8_t *AT8, int64_t ldat, const float *at_inv, int n, const int *sup_idx,
                                   const float *sup_val, int cap, StartState s, int r, float *U, int64_t ldu,
                                   const int *gate, cudaStream_t st) {
  if (ldat % 16 != 0 || (reinterpret_cast<uintptr_t>(AT8) & 15u) != 0) return cudaErrorInvalidValue;
  dim3 grid((unsigned)r, (unsigned)((n + 4095) / 4096));
  k_gemm1_sparse_f8<<<grid, 256, 0, st>>>(AT8, ldat, at_inv, n, sup_idx, sup_val, cap, s, U, ldu, gate);
  return cudaGetLastError();
}

// u = A x over the support.  T = float: A^T in FP32; __half: its leading FP16 plane, the inverse scale
// at_inv[j] folded into x_j (exact).  V rows per thread as one vector, L columns' loads in flight.
// Many starts (S = 1): a CTA per start and row block, FMAs in support order; DRAM (the distinct columns
// of all supports) and L2 bound it.
// Few starts: the round trips of a start's columns bound it, so the support is staged at once, V is small
// (more CTAs), L large, and S slices of a CTA's threads take every S-th column each (FP32 only: the FP16
// plane keeps the support order); the start's last CTA then runs the y-step on the whole of u (from L2)
// instead of a launch of its own.  cnt: r zeroed counters, left zeroed (y and ypl null: u alone).
// Gather and y-step of a sweep before and now (ncu, cold caches): one start of 5000 rows and 150 to 260 columns
// 36 -> 10 us (one row per thread, 4-column batches, y-step of its own before); 16 starts of 9001 rows in
// FP16 24 -> 16 us; 16 of 500 rows 11 -> 9 us; 1024 of 5000 rows (S = 1, y-step of its own) 72 + 11 us, as
// before: with the y-step fused 95 us (its tail runs at the gather's occupancy).
template <typename T, int V>
struct RowVec;
template <>
struct RowVec<float, 4> {
  float4 v;
  __device__ void load(const float *p) { v = __ldg(reinterpret_cast<const float4 *>(p)); }
  __device__ void fma_into(float x, float (&a)[4]) const {
    a[0] = fmaf(x, v.x, a[0]); a[1] = fmaf(x, v.y, a[1]); a[2] = fmaf(x, v.z, a[2]); a[3] = fmaf(x, v.w, a[3]);
  }
};
template <>
struct RowVec<float, 1> {
  float v;
  __device__ void load(const float *p) { v = __ldg(p); }
  __device__ void fma_into(float x, float (&a)[1]) const { a[0] = fmaf(x, v, a[0]); }
};
template <int V>
struct RowVec<__half, V> {
  uint32_t v[V / 2];
  __device__ void load(const __half *p) {
    if constexpr (V == 8) {
      const uint4 t = __ldg(reinterpret_cast<const uint4 *>(p));
      v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else {
      v[0] = __ldg(reinterpret_cast<const uint32_t *>(p));
    }
  }
  __device__ void fma_into(float x, float (&a)[V]) const {
#pragma unroll
    for (int q = 0; q < V / 2; ++q) {
      const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&v[q]));
      a[2 * q] = fmaf(x, f.x, a[2 * q]);
      a[2 * q + 1] = fmaf(x, f.y, a[2 * q + 1]);
    }
  }
};

template <typename T, int V, int L, int NT, int S>
__global__ void __launch_bounds__(NT) k_gather_y(int form, const T *__restrict__ AT, const float *__restrict__ at_inv,
                                                 int64_t ldat, int n, const int *__restrict__ sup_idx,
                                                 const float *__restrict__ sup_val, int cap, StartState s,
                                                 float *__restrict__ U, int64_t ldu, const int *__restrict__ gate,
                                                 float *Y, __half *Ypl, int64_t pstride, const int *__restrict__ rank,
                                                 float *X, int64_t ldX, int p, int *cnt) {
  constexpr int R = NT / S, kTile = V < 4 ? 1024 : NT;   // threads of a slice, columns staged at once
  static_assert(S == 1 || V == 1, "the slices' sums are added for one row per thread");
  __shared__ int sidx[kTile];
  __shared__ float sval[kTile];
  __shared__ float redf[32];
  __shared__ int last;
  if (*gate == 0) return;
  const int c = blockIdx.x;
  if (s.status[c] != ST_ACTIVE || s.iters[c] == 0) return;   // a start not swept yet has a dense x
  const int nnz = s.nnz[c], slice = threadIdx.x / R;
  const int i0 = (blockIdx.y * R + threadIdx.x % R) * V;
  const int *gi = sup_idx + (int64_t)c * cap;
  const float *gv = sup_val + (int64_t)c * cap;
  float acc[V];
#pragma unroll
  for (int q = 0; q < V; ++q) acc[q] = 0.0f;
  for (int t0 = 0; t0 < nnz; t0 += kTile) {
    __syncthreads();
    const int m = min(kTile, nnz - t0);
    for (int t = threadIdx.x; t < m; t += NT) {
      const int j = gi[t0 + t];
      sidx[t] = j;
      sval[t] = at_inv ? gv[t0 + t] * at_inv[j] : gv[t0 + t];
    }
    __syncthreads();
    if (i0 < n) {              // (the columns are padded to a multiple of 8 rows)
      const T *base = AT + i0;
      RowVec<T, V> a[L];
      int t = slice;
      for (; t + (L - 1) * S < m; t += L * S) {
#pragma unroll
        for (int q = 0; q < L; ++q) a[q].load(base + (int64_t)sidx[t + q * S] * ldat);
#pragma unroll
        for (int q = 0; q < L; ++q) a[q].fma_into(sval[t + q * S], acc);
      }
      if (t < m) {
#pragma unroll
        for (int q = 0; q < L; ++q)
          if (t + q * S < m) a[q].load(base + (int64_t)sidx[t + q * S] * ldat);
#pragma unroll
        for (int q = 0; q < L; ++q)
          if (t + q * S < m) a[q].fma_into(sval[t + q * S], acc);
      }
    }
  }
  float *u = U + (int64_t)c * ldu;
  if constexpr (S > 1) {
    __shared__ float part[S][R];
    part[slice][threadIdx.x % R] = acc[0];
    __syncthreads();
    if (slice == 0 && i0 < n) {
      float t = part[0][threadIdx.x];
#pragma unroll
      for (int q = 1; q < S; ++q) t += part[q][threadIdx.x];
      u[i0] = t;
    }
  } else if constexpr (V >= 4) {
#pragma unroll
    for (int h = 0; h < V; h += 4) {
      if (i0 + h + 4 <= n) {
        *reinterpret_cast<float4 *>(u + i0 + h) = make_float4(acc[h], acc[h + 1], acc[h + 2], acc[h + 3]);
      } else {
        for (int q = h; q < h + 4; ++q)
          if (i0 + q < n) u[i0 + q] = acc[q];
      }
    }
  } else {
#pragma unroll
    for (int q = 0; q < V; ++q)
      if (i0 + q < n) u[i0 + q] = acc[q];
  }
  if (!Y && !Ypl) return;
  __syncthreads();
  if (threadIdx.x == 0) {
    int before = 0;
    asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(before) : "l"(cnt + c) : "memory");
    last = before == (int)gridDim.y - 1;
    if (last) cnt[c] = 0;
  }
  __syncthreads();
  if (last) ystep_body<true>(form, U, ldu, n, Y, Ypl, pstride, rank, s, X, ldX, p, c, redf);
}

// The few-start variants serve while their CTAs are at most 8 per SM (256 threads of one row; FP16: 3, two
// rows): gather and y-step of n = 2000, 10 columns, in event times: 8 starts 12.7 us (wide vectors and the
// y-step of its own 16.5), 40 starts (1280 CTAs) 15.8 (17.4), 100 starts 24 (18); FP16: 100 starts (400 CTAs)
// 14.6 (16.3), 200 starts 18.6 (16.9).
bool gather_few(bool half, int r, int64_t n, int sms) {
  return half ? r * ((n + 511) / 512) <= 3 * sms : r * ((n + 63) / 64) <= 8 * sms;
}

cudaError_t launch_gather_y(int form, const float *AT, const void *AT16, const float *at_inv, int64_t ldat, int n,
                            const int *sup_idx, const float *sup_val, int cap, StartState s, int r, float *U,
                            int64_t ldu, const int *gate, float *Y, void *Ypl, int64_t pstride, const int *rank,
                            float *X, int64_t ldX, int p, int *cnt, int sms, cudaStream_t st) {
  const void *base = AT16 ? AT16 : AT;
  if (ldat % 8 != 0 || ldu % 8 != 0 || (reinterpret_cast<uintptr_t>(base) & 15u) != 0) return cudaErrorInvalidValue;
  __half *yp = static_cast<__half *>(Ypl);
  auto go = [&](auto kern, const auto *at, int rows, int nt) -> cudaError_t {
    const int64_t blocks = (n + (int64_t)rows - 1) / rows;
    if (blocks > 65535) return cudaErrorInvalidValue;   // grid y limit
    kern<<<dim3((unsigned)r, (unsigned)blocks), nt, 0, st>>>(form, at, at_inv, ldat, n, sup_idx, sup_val, cap, s, U, ldu,
                                                             gate, Y, yp, pstride, rank, X, ldX, p, cnt);
    return cudaGetLastError();
  };
  const bool few = gather_few(AT16 != nullptr, r, n, sms);
  if (AT16) {   // (256 threads: the order in which the y-step kernel adds ||u||^2)
    const __half *a = static_cast<const __half *>(AT16);
    return few ? go(k_gather_y<__half, 2, 32, 256, 1>, a, 512, 256) : go(k_gather_y<__half, 8, 8, 256, 1>, a, 2048, 256);
  }
  return few ? go(k_gather_y<float, 1, 16, 256, 4>, AT, 64, 256) : go(k_gather_y<float, 4, 8, 128, 1>, AT, 512, 128);
}

// ------------------------------------------------------------------ groups of problems
// The per-start phases for all problems of a group in one launch each: block g (or blockIdx.x for
// the per-problem active lists) looks its problem up and runs the single-problem body on that
// problem's blocks of the workspace.
__global__ void __launch_bounds__(256) k_g_start_init(const GProb *__restrict__ P, const int *__restrict__ prob,
                                                      int parity) {
  __shared__ float redf[32];
  __shared__ unsigned redu[32];
  const GProb &q = P[prob[blockIdx.x]];
  if (!q.first) return;   // only the members whose first sweep is next
  const int c = (int)blockIdx.x - q.start0;
  XPack pk;               // the two planes of x that the dense u = A x reads, row c
  pk.planes = q.Xpl;
  pk.ld = q.ldX;
  pk.stride = q.xps;
  pk.n = 2;
  pk.inv = q.x_inv;
  start_pack_body(q.x0, q.ld0, q.key, q.p, q.X, q.ldX, pk, q.st, q.gamma0, nullptr, c, redf, redu);
  last_makes_active_list(q.r, q.st.status, nullptr, q.r, q.act, q.rank, q.ctrl[parity], nullptr);
}

cudaError_t launch_g_start_init(const GProb *P, const int *prob, int R, int parity, cudaStream_t st) {
  k_g_start_init<<<R, 256, 0, st>>>(P, prob, parity);
  return cudaGetLastError();
}

__global__ void __launch_bounds__(1024) k_g_active(const GProb *__restrict__ P, int parity) {
  const GProb &q = P[blockIdx.x];
  active_list_body(q.st.status, q.st.nnz, q.r, q.act, q.rank, q.ctrl[parity]);
  // the control word that the sweep read is cleared for the next one
  if (threadIdx.x == 0) *q.ctrl[parity ^ 1] = Ctrl{};
}

cudaError_t launch_g_active(const GProb *P, int np, int parity, cudaStream_t st) {
  k_g_active<<<np, 1024, 0, st>>>(P, parity);
  return cudaGetLastError();
}

// many small device copies in one launch (block i copies list[i]): 16 bytes at a time where both
// ends are 16-byte aligned, else byte by byte
__global__ void k_copy_list(const CopyDesc *__restrict__ list) {
  const CopyDesc d = list[blockIdx.x];
  const char *src = static_cast<const char *>(d.src);
  char *dst = static_cast<char *>(d.dst);
  if (((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15u) == 0) {
    const int64_t n16 = d.bytes / 16;
    for (int64_t i = threadIdx.x; i < n16; i += blockDim.x)
      reinterpret_cast<uint4 *>(dst)[i] = reinterpret_cast<const uint4 *>(src)[i];
    for (int64_t i = 16 * n16 + threadIdx.x; i < d.bytes; i += blockDim.x) dst[i] = src[i];
  } else {
    for (int64_t i = threadIdx.x; i < d.bytes; i += blockDim.x) dst[i] = src[i];
  }
}

cudaError_t launch_copy_list(const CopyDesc *list, int count, cudaStream_t st) {
  if (count < 1) return cudaSuccess;
  k_copy_list<<<count, 256, 0, st>>>(list);
  return cudaGetLastError();
}

// the control words of one sweep parity gathered for the host: problem i's active count in out[i], the
// starts that needed the full x-step in that sweep in out[np + i]
__global__ void k_g_ctrl(const GProb *__restrict__ P, int np, int parity, int *__restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < np; i += gridDim.x * blockDim.x) {
    const Ctrl *c = P[i].ctrl[parity];
    out[i] = c->active;
    out[np + i] = c->n_full;
  }
}

cudaError_t launch_g_ctrl(const GProb *P, int np, int parity, int *out, cudaStream_t st) {
  k_g_ctrl<<<(np + 255) / 256, 256, 0, st>>>(P, np, parity, out);
  return cudaGetLastError();
}

// grid (R, row blocks of the largest n): blocks past a problem's n exit
__global__ void __launch_bounds__(kGatherThreads) k_g_gather(const GProb *__restrict__ P, const int *__restrict__ prob) {
  __shared__ int sidx[kGatherThreads];
  __shared__ float sval[kGatherThreads];
  const GProb &q = P[prob[blockIdx.x]];
  if ((int)blockIdx.y * 4 * kGatherThreads >= q.n) return;
  const int c = (int)blockIdx.x - q.start0;
  if (q.AT16)
    gather_lowp_body(q.AT16, q.at_inv, q.ldAT, q.n, q.sup_idx, q.sup_val, q.p, q.st, q.U, q.ldU, c, (int)blockIdx.y,
                     sidx, sval);
  else
    gather_body(q.AT32, q.ldAT, q.n, q.sup_idx, q.sup_val, q.p, q.st, q.U, q.ldU, c, (int)blockIdx.y, sidx, sval);
}

cudaError_t launch_g_gather(const GProb *P, const int *prob, int R, int max_n, cudaStream_t st) {
  const int blocks = (max_n + 4 * kGatherThreads - 1) / (4 * kGatherThreads);
  if (blocks > 65535 || R > 0x7fffffff) return cudaErrorInvalidValue;
  k_g_gather<<<dim3((unsigned)R, (unsigned)blocks), kGatherThreads, 0, st>>>(P, prob);
  return cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_g_ystep(const GProb *__restrict__ P, const int *__restrict__ prob) {
  __shared__ float redf[32];
  const GProb &q = P[prob[blockIdx.x]];
  const int c = (int)blockIdx.x - q.start0;
  // the member's active starts sit at its pool's Y rows *yoff + rank
  __half *ypl = q.Ypl + (q.yoff ? (int64_t)*q.yoff * q.ldU : 0);
  ystep_body(q.form, q.U, q.ldU, q.n, nullptr, ypl, q.yps, q.rank, q.st, q.X, q.ldX, q.p, c, redf);
}

__global__ void __launch_bounds__(256) k_g_pools(const GPool *__restrict__ pools, const GProb *__restrict__ P,
                                                 const int *__restrict__ members, int parity) {
  const GPool q = pools[blockIdx.x];
  if (threadIdx.x == 0) {   // Y row offsets in member order
    int acc = 0;
    for (int k = 0; k < q.nmem; ++k) {
      const GProb &m = P[members[q.first + k]];
      *m.yoff = acc;
      acc += m.ctrl[parity]->active;
    }
    *q.count = acc;
  }
  __syncthreads();   // (the offsets are this block's own global writes)
  for (int k = 0; k < q.nmem; ++k) {
    const GProb &m = P[members[q.first + k]];
    const int a = m.ctrl[parity]->active, o = *m.yoff;
    for (int t = threadIdx.x; t < a; t += blockDim.x) q.colmap[o + t] = m.vbase + m.act[t];
  }
}

cudaError_t launch_g_pools(const GPool *pools, int npool, const GProb *P, const int *members, int parity,
                           cudaStream_t st) {
  if (npool < 1) return cudaSuccess;
  k_g_pools<<<npool, 256, 0, st>>>(pools, P, members, parity);
  return cudaGetLastError();
}

cudaError_t launch_g_ystep(const GProb *P, const int *prob, int R, cudaStream_t st) {
  k_g_ystep<<<R, 256, 0, st>>>(P, prob);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ few starts: streaming GEMV
// out[orow(c)][m] = sum_k P[m, k] Q[qrow(c), k] for the first *count (<= R) starts: the Q rows in
// shared memory, a warp per row of P (two rows for R >= 4, which then share each read of Q) read
// once with 16-byte loads, each lane's R sums per row over its strided part, then the warp's
// sums in a fixed butterfly.  Q rows longer than the shared memory holds are taken in chunks of
// Kc columns (the row sums carried in registers across the chunks, in K order).
// P's rows and Q's rows are zero past K up to the next multiple of 4 (padded layouts).
// The rows are walked in steps of NR per warp over the whole grid; the last, partial step gives each
// row to as many warps of a CTA (2, 4, 8 or 16) as there are to spare, which split its columns, so that
// the chip stays busy to the end (2.06 steps took the time of three).  Bound by HBM: v = A^T y,
// 5000 x 20000 (400 MB), before and now, CUDA events (about 5 us more than the kernel): one start 74 -> 64 us,
// two 102 -> 65, eight 106 -> 86; u = A x: 92 -> 67, 109 -> 77, 405 -> 131 us (its Q rows in chunks).
template <int R, int NR>
__global__ void __launch_bounds__(512, R <= 2 ? 2 : 1) k_gemv(const float *__restrict__ P, int64_t ldp, int M, int K, int Kc,
                                                 const float *__restrict__ Q, int64_t ldq,
                                                 const int *__restrict__ rows, const int *__restrict__ count,
                                                 float *__restrict__ out, int64_t ldo, const int *__restrict__ gate) {
  extern __shared__ __align__(16) float qs[];
  __shared__ float part[R][16];
  constexpr int U = NR == 1 ? 6 : 4;   // vectors of each row in flight per lane
  if (gate && *gate == 0) return;
  const int cnt = count ? min(*count, R) : R;
  if (cnt <= 0) return;
  const int K4 = (K + 3) / 4, Kp = 4 * K4;
  const int nchunks = (Kp + Kc - 1) / Kc;
  // columns [k0, k0 + Kc) of the Q rows into shared memory (zero past K: the rows' padding), as vectors,
  // 4 in flight per thread
  auto load_q = [&](int k0) {
    const int c4 = Kc / 4, have = min(Kp - k0, Kc) / 4;
#pragma unroll 1
    for (int c = 0; c < R; ++c) {
      const float4 *q = reinterpret_cast<const float4 *>(Q + (int64_t)(c < cnt ? (rows ? rows[c] : c) : 0) * ldq + k0);
      float4 *s = reinterpret_cast<float4 *>(qs + c * Kc);
      const int n = c < cnt ? have : 0;
      for (int e = threadIdx.x; e < c4; e += 4 * blockDim.x) {
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          v[u] = e + u * (int)blockDim.x < n ? __ldg(q + e + u * blockDim.x) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (e + u * (int)blockDim.x < c4) s[e + u * blockDim.x] = v[u];
      }
    }
  };
  if (nchunks == 1) {
    load_q(0);
    __syncthreads();
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const int all = gridDim.x * warps;   // warps of the grid
  // NR rows per warp and step: every shared-memory read of Q serves all of them.  The loop count
  // is the same for every warp of the CTA (the chunked path synchronises inside it).
  for (int base = 0; base < M;) {
    int g = 1;                         // warps per row (uniform over the grid)
    const int left = M - base;
    if (left < NR * all)
      while (g < 16 && left * 2 * g <= all) g *= 2;
    const int per = g > 1 ? 1 : NR;    // rows of this warp's step
    const int m0 = base + per * ((blockIdx.x * warps + warp) / g), sub = warp & (g - 1);
    base += g > 1 ? left : NR * all;
    if (nchunks == 1 && g == 1 && m0 >= M) continue;
    const float4 *pr[NR];
#pragma unroll
    for (int t = 0; t < NR; ++t) pr[t] = reinterpret_cast<const float4 *>(P + (int64_t)min(m0 + t, M - 1) * ldp);
    float acc[NR][R];
#pragma unroll
    for (int t = 0; t < NR; ++t)
#pragma unroll
      for (int c = 0; c < R; ++c) acc[t][c] = 0.0f;
    for (int ch = 0; ch < nchunks; ++ch) {
      const int k0 = ch * Kc;
      if (nchunks > 1) {
        __syncthreads();   // the previous chunk is consumed
        load_q(k0);
        __syncthreads();
      }
      const int c4 = min(Kc, Kp - k0) / 4;   // float4 columns of this chunk
      // (the last batch of a row is predicated: a rolled remainder would wait for its loads one by one)
      for (int k4 = sub * 32 + lane; k4 < c4 && m0 < M; k4 += 32 * U * g) {
        float4 a[U][NR];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int t = 0; t < NR; ++t)
            if (k4 + 32 * u * g < c4 && t < per) a[u][t] = __ldg(pr[t] + k0 / 4 + k4 + 32 * u * g);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (k4 + 32 * u * g < c4) {
#pragma unroll
            for (int c = 0; c < R; ++c) {
              const float4 q = reinterpret_cast<const float4 *>(qs + c * Kc)[k4 + 32 * u * g];
#pragma unroll
              for (int t = 0; t < NR; ++t) {
                if (t < per) {
                  acc[t][c] = fmaf(a[u][t].x, q.x, acc[t][c]);
                  acc[t][c] = fmaf(a[u][t].y, q.y, acc[t][c]);
                  acc[t][c] = fmaf(a[u][t].z, q.z, acc[t][c]);
                  acc[t][c] = fmaf(a[u][t].w, q.w, acc[t][c]);
                }
              }
            }
          }
        }
      }
    }
#pragma unroll
    for (int t = 0; t < NR; ++t)
#pragma unroll
      for (int c = 0; c < R; ++c) acc[t][c] = warp_sum_f(acc[t][c]);
    if (g > 1) {                       // the row's warps, added in order
      __syncthreads();
#pragma unroll
      for (int c = 0; c < R; ++c)
        if (lane == 0) part[c][warp] = acc[0][c];
      __syncthreads();
      if (sub == 0) {
#pragma unroll
        for (int c = 0; c < R; ++c)
          for (int q = 1; q < g; ++q) acc[0][c] += part[c][warp + q];
      }
    }
    if (lane < cnt && sub == 0) {
      float *o = out + (int64_t)(rows ? rows[lane] : lane) * ldo;
#pragma unroll
      for (int t = 0; t < NR; ++t) {
        float v = acc[t][0];
#pragma unroll
        for (int c = 1; c < R; ++c)
          if (lane == c) v = acc[t][c];
        if (t < per && m0 + t < M) o[m0 + t] = v;
      }
    }
  }
}

// once per kernel and process (thread-safe): the largest shared memory the launcher allows
template <int R, int NR>
cudaError_t gemv_configured() {
  static const cudaError_t e =
      cudaFuncSetAttribute(k_gemv<R, NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGemvSmemMax);
  return e;
}

int gemv_width(int r) { return r <= 1 ? 1 : r <= 2 ? 2 : r <= 4 ? 4 : r <= kGemvMaxR ? kGemvMaxR : 0; }

// any K: Q rows that do not fit in shared memory are streamed in chunks
bool gemv_fits(int r, int64_t K) { return gemv_width(r) > 0 && K > 0 && K < INT32_MAX; }

cudaError_t launch_gemv(const float *P, int64_t ldp, int M, int K, const float *Q, int64_t ldq, const int *rows,
                        const int *count, int r, float *out, int64_t ldo, const int *gate, int sms, cudaStream_t st) {
  const int w = gemv_width(r);
  if (w == 0 || K < 1) return cudaErrorInvalidValue;
  const int64_t Kp = (int64_t)(K + 3) / 4 * 4;
  // chunk of the Q rows held in shared memory: all of them when they fit, else the largest
  // multiple of 128 columns that fits (whole float4 steps of every lane)
  int64_t Kc = Kp;
  if ((int64_t)w * Kp * 4 > kGemvSmemMax) Kc = (int64_t)kGemvSmemMax / (4 * w) / 128 * 128;
  const size_t smem = (size_t)w * Kc * sizeof(float);
  // CTAs resident per SM (registers: two for one or two starts, else one; shared memory), a grid of
  // that many per SM, each CTA loading the Q rows once (per row batch when they are chunked)
  const int per_sm = w <= 2 && smem <= 100 * 1024 ? 2 : 1;
  const int blocks = std::min(M, per_sm * sms);
  auto go = [&](auto kern, cudaError_t configured) -> cudaError_t {
    if (configured != cudaSuccess) return configured;
    kern<<<blocks, 512, smem, st>>>(P, ldp, M, K, (int)Kc, Q, ldq, rows, count, out, ldo, gate);
    return cudaGetLastError();
  };
  switch (w) {
    case 1: return go(k_gemv<1, 1>, gemv_configured<1, 1>());
    case 2: return go(k_gemv<2, 1>, gemv_configured<2, 1>());
    case 4: return go(k_gemv<4, 2>, gemv_configured<4, 2>());
    default: return go(k_gemv<kGemvMaxR, 2>, gemv_configured<kGemvMaxR, 2>());
  }
}

}  // namespace spca
