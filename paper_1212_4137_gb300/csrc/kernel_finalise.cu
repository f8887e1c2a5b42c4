// kernel_finalise.cu -- after the sweeps: the Table 1 objective f(x) of every start with
// u = A x accumulated as a compensated FP32-pair dot product (about twice FP32's precision) and
// the norms of u summed in FP64, the explained variance (Section 4.1), the best start (ties:
// lower index), and y(x) and the support of the best x.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "block_util.cuh"
#include "spca_internal.cuh"

namespace spca {

namespace {
constexpr int FT = 128;            // threads per CTA, four rows of A each, or one
}  // namespace
// The rows of a chunk of an n-row problem of r starts: 4 FT where those chunks fill the chip, four on each of
// about 150 SMs, and their threads (n > 2 FT), else FT.  A start's columns are one chain of loads and dependent
// sums, twice as long for four rows of a thread as for one.  Supports of 9000 columns, four rows and one: n = 100, one
// start 1044 and 342 us (524 before there were four); n = 2000, 16 starts 2621 and 801, 150 starts (600 chunks)
// 2469 and 2010; n = 9000, 64 starts (1152) 2834 and 3645; n = 500, 1024 starts 2448 and 3163.
// (By the problem's own starts and rows: in a group a problem has the same chunks alone and in any mix.)
static __host__ __device__ inline int finalise_rows(int64_t n, int64_t r) {
  return r * ((n + 4 * FT - 1) / (4 * FT)) >= 608 && n > 2 * FT ? 4 * FT : FT;
}
int finalise_chunks(int64_t n, int64_t r) {
  const int rows = finalise_rows(n, r);
  return (int)((n + rows - 1) / rows);
}

// argmax over r starts of f (or of the explained variance), ties to the lower index; written by other
// CTAs of the same launch, so read from L2
__device__ __forceinline__ void best_body(const double *val, int r, int *best) {
  __shared__ double sv[32];
  __shared__ int si[32];
  double bv = -INFINITY;
  int bi = 0x7fffffff;
  for (int c = threadIdx.x; c < r; c += blockDim.x) {
    const double v = __ldcg(val + c);
    if (v > bv) { bv = v; bi = c; }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double ov = __shfl_xor_sync(0xffffffffu, bv, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) { sv[w] = bv; si[w] = bi; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < (int)(blockDim.x >> 5); ++k)
      if (sv[k] > bv || (sv[k] == bv && si[k] < bi)) { bv = sv[k]; bi = si[k]; }
    *best = (bi == 0x7fffffff) ? 0 : bi;
  }
}

// R consecutive entries of a column of A (a row of A^T): FP32, or FP16 times the column's
// power-of-two inverse scale (the 16-bit copy of a resident handle; exact in FP32)
template <int R>
struct ColVec {
  float v[R];
};
__device__ __forceinline__ void col_load(ColVec<4> &a, const float *p) {
  const float4 t = __ldg(reinterpret_cast<const float4 *>(p));
  a.v[0] = t.x; a.v[1] = t.y; a.v[2] = t.z; a.v[3] = t.w;
}
__device__ __forceinline__ void col_load(ColVec<4> &a, const __half *p) {
  const uint2 raw = __ldg(reinterpret_cast<const uint2 *>(p));
  const __half2 *h = reinterpret_cast<const __half2 *>(&raw);
  const float2 lo = __half22float2(h[0]), hi = __half22float2(h[1]);
  a.v[0] = lo.x; a.v[1] = lo.y; a.v[2] = hi.x; a.v[3] = hi.y;
}
__device__ __forceinline__ void col_load(ColVec<1> &a, const float *p) { a.v[0] = __ldg(p); }
__device__ __forceinline__ void col_load(ColVec<1> &a, const __half *p) { a.v[0] = __half2float(__ldg(p)); }

// Chunk b (of nch) of start c: u_i = sum_t x_{j_t} A[i, j_t] over the support (compensated FP32 pairs),
// R rows per thread as one vector with eight columns' loads in flight, and the chunk's FP64 sum of
// |u_i| or u_i^2, whichever the formulation's variance takes.  The start's last chunk then adds the
// partial sums in a fixed order and gives f (Table 1) and the explained variance; the last start finds
// the best one.  cnt: r + 1 zeroed counters, left zeroed.
// Starts on grid x, chunks on y: the CTAs in flight share row chunks, so a column slice used by several
// starts' supports is read from DRAM about once.  The pairs' FP32 arithmetic (about 12 operations per
// entry) and the gather through L2 bound it.
// 1024 starts of 50 nonzeros, n = 5000: 156 us (a row per thread, one load in flight, both norms, and
// three launches: 353 us); 12 members of a group: 42 us (342 us as launches of their own).
template <int R, typename T>
__device__ __forceinline__ void finalise_body(int form, const T *__restrict__ AT, const float *__restrict__ row_inv,
                                              int64_t ldat, int n, const int *__restrict__ sup_idx,
                                              const float *__restrict__ sup_val, int cap, const StartState &st, int r,
                                              float *__restrict__ U, int64_t ldu, double *partials, int *cnt,
                                              int use_ev, int *best, int c, int b, int nch) {
  __shared__ int sidx[FT];
  __shared__ float sval[FT];
  __shared__ float sinv[FT];
  __shared__ double red[32];
  __shared__ int state;
  const int i0 = (b * FT + threadIdx.x) * R;
  const int nnz = st.nnz[c];
  const int *gi = sup_idx + (int64_t)c * cap;
  const float *gv = sup_val + (int64_t)c * cap;
  F32Pair acc[R];
  auto step = [&](float x, float inv, const ColVec<R> &a) {
#pragma unroll
    for (int q = 0; q < R; ++q) f32pair_fma(acc[q], x, a.v[q] * inv);
  };
  for (int t0 = 0; t0 < nnz; t0 += FT) {
    __syncthreads();
    if (t0 + (int)threadIdx.x < nnz) {
      const int j = gi[t0 + threadIdx.x];
      sidx[threadIdx.x] = j;
      sval[threadIdx.x] = gv[t0 + threadIdx.x];
      sinv[threadIdx.x] = row_inv ? row_inv[j] : 1.0f;
    }
    __syncthreads();
    const int m = min(FT, nnz - t0);
    if (i0 < n) {              // (the columns are padded to a multiple of 8 rows)
      const T *base = AT + i0;
      ColVec<R> a[8];
      int t = 0;
      for (; t + 8 <= m; t += 8) {
#pragma unroll
        for (int q = 0; q < 8; ++q) col_load(a[q], base + (int64_t)sidx[t + q] * ldat);
#pragma unroll
        for (int q = 0; q < 8; ++q) step(sval[t + q], sinv[t + q], a[q]);
      }
      for (; t < m; ++t) {
        col_load(a[0], base + (int64_t)sidx[t] * ldat);
        step(sval[t], sinv[t], a[0]);
      }
    }
  }
  const bool l1 = is_l1_var(form);
  double part = 0.0;
#pragma unroll
  for (int q = 0; q < R; ++q) {
    if (i0 + q < n) {
      const double u = f32pair_value(acc[q]);
      U[(int64_t)c * ldu + i0 + q] = (float)u;
      part = l1 ? part + fabs(u) : fma(u, u, part);
    }
  }
  part = block_sum_d(part, red);
  if (threadIdx.x == 0) {
    partials[(int64_t)c * nch + b] = part;
    int before;
    asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(before) : "l"(cnt + c) : "memory");
    state = before == nch - 1;
  }
  __syncthreads();
  if (!state) return;
  // the start's last chunk
  double sum = 0.0, x1 = 0.0;
  for (int q = threadIdx.x; q < nch; q += FT) sum += __ldcg(partials + (int64_t)c * nch + q);
  sum = block_sum_d(sum, red);
  if (uses_V(form)) {          // ||x||_1 (Table 1's L1 penalty alone needs it)
    for (int t = threadIdx.x; t < nnz; t += FT) x1 += fabs((double)gv[t]);
    x1 = block_sum_d(x1, red);
  }
  if (threadIdx.x == 0) {
    const double norm = l1 ? sum : sqrt(sum), g = st.gamma[c];
    double f = norm;
    if (uses_U(form)) f = norm * norm - g * (double)nnz;
    if (form == 5) f = sum - g * (double)nnz;
    if (uses_V(form)) f = norm - g * x1;
    st.f[c] = f;
    st.ev[c] = sum;
    cnt[c] = 0;
    int before;
    asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(before) : "l"(cnt + r) : "memory");
    state = before == r - 1;
    if (state) cnt[r] = 0;
  }
  __syncthreads();
  if (state) best_body(use_ev ? st.ev : st.f, r, best);
}

template <int R, typename T>
__global__ void __launch_bounds__(FT) k_finalise(int form, const T *__restrict__ AT, const float *__restrict__ row_inv,
                                                 int64_t ldat, int n, const int *__restrict__ sup_idx,
                                                 const float *__restrict__ sup_val, int cap, StartState st,
                                                 float *__restrict__ U, int64_t ldu, double *partials, int *cnt,
                                                 int use_ev, int *best) {
  finalise_body<R>(form, AT, row_inv, ldat, n, sup_idx, sup_val, cap, st, (int)gridDim.x, U, ldu, partials, cnt,
                   use_ev, best, (int)blockIdx.x, (int)blockIdx.y, (int)gridDim.y);
}

cudaError_t launch_finalise(int form, const float *AT, const __half *AT16, const float *at_inv, int64_t ldat, int n,
                            StartState s, int r, float *U, int64_t ldu, const int *sup_idx, const float *sup_val,
                            int cap, double *partials, int *cnt, int use_ev, int *best, cudaStream_t st) {
  const int rows = finalise_rows(n, r), nch = finalise_chunks(n, r);
  if (nch > 65535) return cudaErrorInvalidValue;   // grid y limit
  const dim3 grid((unsigned)r, (unsigned)nch);
  auto go = [&](auto kern, const auto *at, const float *inv) {
    kern<<<grid, FT, 0, st>>>(form, at, inv, ldat, n, sup_idx, sup_val, cap, s, U, ldu, partials, cnt, use_ev, best);
    return cudaGetLastError();
  };
  if (AT16)
    return rows == FT ? go(k_finalise<1, __half>, AT16, at_inv) : go(k_finalise<4, __half>, AT16, at_inv);
  return rows == FT ? go(k_finalise<1, float>, AT, nullptr) : go(k_finalise<4, float>, AT, nullptr);
}

// the same for the finishing members of a group (done[i] != 0; all when null), one launch
__global__ void __launch_bounds__(FT) k_g_finalise(const GProb *__restrict__ P, const int *__restrict__ prob,
                                                   const int *__restrict__ done) {
  const int i = prob[blockIdx.x];
  if (done && !done[i]) return;
  const GProb &q = P[i];
  const int rows = finalise_rows(q.n, q.r), nch = (q.n + rows - 1) / rows, c = (int)blockIdx.x - q.start0;
  if ((int)blockIdx.y >= nch) return;
  auto go = [&](auto rows_each, const auto *at, const float *inv) {
    finalise_body<decltype(rows_each)::value>(q.form, at, inv, q.ldAT, q.n, q.sup_idx, q.sup_val, q.p, q.st, q.r, q.U,
                                              q.ldU, q.partials, q.fin_cnt, q.use_ev, q.best, c, (int)blockIdx.y, nch);
  };
  using One = std::integral_constant<int, 1>;
  using Four = std::integral_constant<int, 4>;
  if (q.AT16) {
    if (rows == FT) go(One{}, q.AT16, q.at_inv);
    else go(Four{}, q.AT16, q.at_inv);
  } else {
    const float *none = nullptr;
    if (rows == FT) go(One{}, q.AT32, none);
    else go(Four{}, q.AT32, none);
  }
}

// argmax over starts of f (or of the explained variance), ties to the lower index
__global__ void __launch_bounds__(1024) k_best(int use_ev, StartState st, int r, int *best) {
  best_body(use_ev ? st.ev : st.f, r, best);
}

cudaError_t launch_best(int form, int use_ev, StartState s, int r, int *best, cudaStream_t st) {
  (void)form;
  k_best<<<1, 1024, 0, st>>>(use_ev, s, r, best);
  return cudaGetLastError();
}

// y = y(x) (S2: sgn(u), S1: u / ||u||_2, with ||u||_2^2 = the explained variance), x and the support of
// the best start.  CTA 0 compacts the support, from the start's list (sup_idx / sup_val, nnz entries) or,
// without lists, from all of x: each warp counts a contiguous range, one exchange over the warps, then
// each writes its part.  The other CTAs copy x and write y.  One CTA did all of it before, 1024 entries of
// x per barrier pair: p = 100000 158 us, p = 20000 53 us; now 5 and 6 us.
constexpr int OT_ = 512;
__device__ __forceinline__ void best_outputs_body(int form, int c, const float *__restrict__ U, int64_t ldu, int n,
                                                  const double *__restrict__ ev, const float *__restrict__ X,
                                                  int64_t ldX, int p, const int *sup_idx, const float *sup_val,
                                                  int cap, const int *nnz_of, float *y_out, float *x_out,
                                                  int64_t *support_out, int64_t *nnz_out, int b, int nb) {
  __shared__ int wcnt[OT_ / 32];
  __shared__ float inv_s;
  const float *u = U + (int64_t)c * ldu;
  const float *x = X + (int64_t)c * ldX;
  if (b == 0) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int m = sup_idx ? nnz_of[c] : p;
    const int *ix = sup_idx ? sup_idx + (int64_t)c * cap : nullptr;
    const float *v = sup_idx ? sup_val + (int64_t)c * cap : x;
    const int per = ((m + OT_ / 32 - 1) / (OT_ / 32) + 31) / 32 * 32, lo = min(m, w * per), hi = min(m, lo + per);
    int cnt = 0;
#pragma unroll 8
    for (int i = lo + lane; i < hi; i += 32) cnt += v[i] != 0.0f;
    cnt = warp_sum_i(cnt);
    if (lane == 0) wcnt[w] = cnt;
    __syncthreads();
    int pos = 0, tot = 0;
    for (int k = 0; k < OT_ / 32; ++k) {
      pos += k < w ? wcnt[k] : 0;
      tot += wcnt[k];
    }
#pragma unroll 4
    for (int base = lo; base < hi; base += 32) {
      const int i = base + lane;
      const bool on = i < hi && v[i] != 0.0f;
      const unsigned ball = __ballot_sync(0xffffffffu, on);
      if (on) support_out[pos + __popc(ball & ((1u << lane) - 1u))] = ix ? ix[i] : i;
      pos += __popc(ball);
    }
    if (threadIdx.x == 0) *nnz_out = tot;
    return;
  }
  const int t0 = (b - 1) * OT_ + threadIdx.x, step = (nb - 1) * OT_;
  if (!is_l1_var(form)) {
    if (threadIdx.x == 0) {
      const double nrm = sqrt(ev[c]);
      inv_s = nrm > 0.0 ? (float)(1.0 / nrm) : 0.0f;
    }
    __syncthreads();
  }
  const float inv = inv_s;
  for (int i = t0; i < n; i += step) y_out[i] = is_l1_var(form) ? (u[i] >= 0.0f ? 1.0f : -1.0f) : u[i] * inv;
  for (int j = t0; j < p; j += step) x_out[j] = x[j];
}
// CTAs for the outputs of an n x p problem: about four entries per thread
static int output_ctas(int64_t n, int64_t p) {
  const int64_t b = (std::max(n, p) + 4 * OT_ - 1) / (4 * OT_);
  return 1 + (int)std::min<int64_t>(b, 64);
}

__global__ void __launch_bounds__(OT_) k_best_outputs(int form, const int *__restrict__ best,
                                                      const float *__restrict__ U, int64_t ldu, int n,
                                                      const double *__restrict__ ev, const float *__restrict__ X,
                                                      int64_t ldX, int p, const int *sup_idx, const float *sup_val,
                                                      int cap, const int *nnz_of, float *__restrict__ y_out,
                                                      float *__restrict__ x_out, int64_t *__restrict__ support_out,
                                                      int64_t *__restrict__ nnz_out) {
  best_outputs_body(form, *best, U, ldu, n, ev, X, ldX, p, sup_idx, sup_val, cap, nnz_of, y_out, x_out, support_out,
                    nnz_out, (int)blockIdx.x, (int)gridDim.x);
}

cudaError_t launch_best_outputs(int form, const int *best, const float *U, int64_t ldu, int n, const double *ev,
                                const float *X, int64_t ldX, int p, const int *sup_idx, const float *sup_val, int cap,
                                const int *nnz_of, float *y_out, float *x_out, int64_t *support_out, int64_t *nnz_out,
                                cudaStream_t st) {
  k_best_outputs<<<output_ctas(n, p), OT_, 0, st>>>(form, best, U, ldu, n, ev, X, ldX, p, sup_idx, sup_val, cap,
                                                    nnz_of, y_out, x_out, support_out, nnz_out);
  return cudaGetLastError();
}

// the same for the finishing members of a group: grid (CTAs of the largest member, members)
__global__ void __launch_bounds__(OT_) k_g_best_outputs(const GProb *__restrict__ P, const int *__restrict__ done) {
  if (done && !done[blockIdx.y]) return;
  const GProb &q = P[blockIdx.y];
  best_outputs_body(q.form, *q.best, q.U, q.ldU, q.n, q.st.ev, q.X, q.ldX, q.p, q.sup_idx, q.sup_val, q.p, q.st.nnz,
                    q.y_out, q.x_out, q.support_out, q.nnz_out, (int)blockIdx.x, (int)gridDim.x);
}

cudaError_t launch_g_finish(const GProb *P, const int *prob, int R, int np, int max_n, int max_p, int max_chunks,
                            const int *done, cudaStream_t st) {
  if (max_chunks > 65535) return cudaErrorInvalidValue;
  k_g_finalise<<<dim3((unsigned)R, (unsigned)max_chunks), FT, 0, st>>>(P, prob, done);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_g_best_outputs<<<dim3((unsigned)output_ctas(max_n, max_p), (unsigned)np), OT_, 0, st>>>(P, done);
  return cudaGetLastError();
}

}  // namespace spca
