// sweep_bodies.cuh -- the per-start bodies of the start initialisation (Algorithm 2, "select
// initial point") and of the y-step (Table 3, S1 and S2), and the active list, shared by the kernels that run them one
// start per CTA: the single-problem kernels, the grouped kernels and the one-launch solve of small
// problems.
#pragma once

#include <cuda_fp16.h>

#include <cstdint>

#include "block_util.cuh"
#include "spca_internal.cuh"

namespace spca {

// ------------------------------------------------------------------ a1: start initialisation
// SplitMix64 (Steele, Lea, Flood 2014) finaliser with the published constants, used as a
// counter-based generator: word(key, i) = mix(key + (i + 1) * golden).
static __device__ __forceinline__ uint64_t sm64_mix(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
static __device__ __forceinline__ double sm64_uniform(uint64_t key, uint64_t i) {
  return (double)(sm64_mix(key + (i + 1ull) * 0x9E3779B97F4A7C15ull) >> 11) * 0x1.0p-53;
}
// normal number i of the stream (Box-Muller over the pair i/2)
static __device__ __forceinline__ double bm_normal(uint64_t key, uint64_t i) {
  const uint64_t j = i >> 1;
  const double u1 = 1.0 - sm64_uniform(key, 2 * j), u2 = sm64_uniform(key, 2 * j + 1);
  const double rad = sqrt(-2.0 * log(u1)), ang = 6.283185307179586 * u2;
  return (i & 1) ? rad * sin(ang) : rad * cos(ang);
}

// Algorithm 2, "select initial point": x^(0) = g / ||g||_2 for the start in row c of X, taking
// start `start` (its row of x0, or normal numbers start * p + j of the seeded stream).
static __device__ void start_init_body(const float *__restrict__ x0, int64_t ld0, uint64_t key, int p,
                                       float *__restrict__ X, int64_t ldX, StartState s, double gamma0, int c,
                                       int64_t start, float *redf) {
  float *x = X + (int64_t)c * ldX;
  const float *g = x0 ? x0 + start * ld0 : nullptr;
  float part = 0.0f;
  for (int j = threadIdx.x; j < p; j += blockDim.x) {
    const float gj = g ? g[j] : (float)bm_normal(key, (uint64_t)start * (uint64_t)p + (uint64_t)j);
    x[j] = gj;
    part = fmaf(gj, gj, part);
  }
  float nrm, lo, inv;
  norm_and_inverse(block_sum_f(part, redf), &nrm, &lo, &inv);
  for (int j = threadIdx.x; j < p; j += blockDim.x) x[j] = x[j] * inv;
  if (threadIdx.x == 0) {
    s.status[c] = (nrm > 0.0f) ? ST_ACTIVE : SPCA_ST_DEGENERATE;
    s.iters[c] = 0;
    s.nnz[c] = (nrm > 0.0f) ? p : 0;
    s.F[c] = 0.0;
    s.F_prev[c] = 0.0;
    s.gamma[c] = gamma0;
    s.thr[c] = 0.0f;
    if (s.tprev) s.tprev[c] = 0.0f;
  }
}

// The same for a solve's first sweep, which reads x^(0) as FP32 (pk.x32) or as FP16 planes of the
// row-scaled x (pk.planes, row c, with 1 / scale in pk.inv[c]) and never as both.  x0 (checked: a
// non-finite entry sets *flag and ends the start) is read twice, the second time mostly from L2; a
// seeded start's raw normals are kept in X between the passes.  ||g||^2 is added as in start_init_body.
static __device__ void start_pack_body(const float *x0, int64_t ld0, uint64_t key, int p, float *X, int64_t ldX,
                                       const XPack &pk, StartState s, double gamma0, int *flag, int c, float *redf,
                                       unsigned *redu) {
  float *x = X + (int64_t)c * ldX;
  const float *g = x0 ? x0 + (int64_t)c * ld0 : nullptr;
  float part = 0.0f;
  unsigned mk = 0u;
  const int nt = (int)blockDim.x;
  constexpr int U = 8, U1 = 16;                // loads in flight per thread
  // (the first 256 threads, whatever the CTA's size: the sum's order)
  constexpr int N1 = 256;
  if (threadIdx.x >= N1) {
    if (!g) g = x;
  } else if (g) {
    for (int j0 = threadIdx.x; j0 < p; j0 += U1 * N1) {
      float v[U1];
#pragma unroll
      for (int k = 0; k < U1; ++k) v[k] = j0 + k * N1 < p ? g[j0 + k * N1] : 0.0f;
#pragma unroll
      for (int k = 0; k < U1; ++k) {
        part = fmaf(v[k], v[k], part);
        mk = max(mk, abs_key(v[k]));
      }
    }
  } else {
    for (int j = threadIdx.x; j < p; j += N1) {
      const float v = (float)bm_normal(key, (uint64_t)c * (uint64_t)p + (uint64_t)j);
      x[j] = v;
      part = fmaf(v, v, part);
      mk = max(mk, abs_key(v));
    }
    g = x;
  }
  float nrm, lo, inv;
  norm_and_inverse(block_sum_f(part, redf), &nrm, &lo, &inv);
  const unsigned top = block_max_u(mk, redu);  // (its barriers also order a seeded start's x)
  const bool bad = top >= 0x7f800000u;         // a non-finite entry
  if (bad) inv = 0.0f;
  const bool alive = nrm > 0.0f && !bad;
  // the planes' scale puts max |x_j| = max |g_j| / ||g|| in [2^13, 2^14) (rounding is monotone)
  const float mx = __uint_as_float(bad ? 0u : top) * inv;
  int e = 0;
  if (mx > 0.0f) e = max(-120, min(120, 13 - ilogbf(mx)));
  const float sc = ldexpf(1.0f, e);
  auto norm = [&](int j) { return alive ? g[j] * inv : 0.0f; };
  if (pk.x32 || !alive) {                      // (a start that never sweeps keeps x = 0)
    for (int j0 = threadIdx.x; j0 < p; j0 += U * nt) {
      float v[U];
#pragma unroll
      for (int k = 0; k < U; ++k) v[k] = j0 + k * nt < p ? norm(j0 + k * nt) : 0.0f;
#pragma unroll
      for (int k = 0; k < U; ++k)
        if (j0 + k * nt < p) x[j0 + k * nt] = v[k];
    }
  }
  if (pk.planes) {
    __half *hi = pk.planes + (int64_t)c * pk.ld;
    constexpr int W = 4;                       // pairs of entries in flight per thread
    for (int j0 = 2 * threadIdx.x; j0 < p; j0 += 2 * W * nt) {
      float v[W][2];
#pragma unroll
      for (int k = 0; k < W; ++k) {
        const int j = j0 + 2 * k * nt;
        v[k][0] = j < p ? norm(j) * sc : 0.0f;
        v[k][1] = j + 1 < p ? norm(j + 1) * sc : 0.0f;
      }
#pragma unroll
      for (int k = 0; k < W; ++k) {
        const int j = j0 + 2 * k * nt;
        if (j >= p) break;
        // (the entry past an odd p is a zero of the row's padding)
        const __half2 h = __floats2half2_rn(v[k][0], v[k][1]);
        *reinterpret_cast<__half2 *>(hi + j) = h;
        if (pk.n > 1) {
          const float2 f = __half22float2(h);
          *reinterpret_cast<__half2 *>(hi + pk.stride + j) = __floats2half2_rn(v[k][0] - f.x, v[k][1] - f.y);
        }
      }
    }
    if (threadIdx.x == 0) pk.inv[c] = ldexpf(1.0f, -e);
  }
  if (threadIdx.x == 0) {
    if (bad && flag) atomicOr(flag, 1);
    s.status[c] = alive ? ST_ACTIVE : SPCA_ST_DEGENERATE;
    s.iters[c] = 0;
    s.nnz[c] = alive ? p : 0;
    s.F[c] = 0.0;
    s.F_prev[c] = 0.0;
    s.gamma[c] = gamma0;
    s.thr[c] = 0.0f;
    if (s.tprev) s.tprev[c] = 0.0f;
  }
}

// ------------------------------------------------------------------ y-step (Table 3 S1, S2)
// Counts the sweep for every active start; L1 variance: y = sgn(u) with sgn(0) = +1;
// L2 variance: y = u / ||u||_2, and ||u||_2 = 0 ends the start as degenerate (x = 0).
// y goes to Y (FP32) and/or to the FP16 planes of kQScale y (hi, lo; one exact plane for +-1).
// (kCg: u was written by other CTAs of the same launch, and is read from L2)
template <bool kCg = false>
static __device__ void ystep_body(int form, const float *__restrict__ U, int64_t ldu, int n,
                                  float *__restrict__ Y, __half *__restrict__ Ypl, int64_t pstride,
                                  const int *__restrict__ rank, StartState s, float *__restrict__ X, int64_t ldX,
                                  int p, int c, float *redf) {
  if (s.status[c] != ST_ACTIVE) return;
  const float *u = U + (int64_t)c * ldu;
  float *y = Y ? Y + (int64_t)c * ldu : nullptr;
  __half *yp = Ypl ? Ypl + (int64_t)(rank ? rank[c] : c) * ldu : nullptr;
  if (threadIdx.x == 0) s.iters[c] += 1;
  // four consecutive entries per thread and step (rows are 16-byte aligned: ldu is a multiple of 8)
  const int n4 = n & ~3;
  if (is_l1_var(form)) {
    for (int i = 4 * threadIdx.x; i < n4; i += 4 * blockDim.x) {
      const float4 uv = kCg ? __ldcg(reinterpret_cast<const float4 *>(u + i)) : *reinterpret_cast<const float4 *>(u + i);
      const float4 yv = make_float4(uv.x >= 0.0f ? 1.0f : -1.0f, uv.y >= 0.0f ? 1.0f : -1.0f,
                                    uv.z >= 0.0f ? 1.0f : -1.0f, uv.w >= 0.0f ? 1.0f : -1.0f);
      if (y) *reinterpret_cast<float4 *>(y + i) = yv;
      if (yp) {
        // +-2^14, exact
        __half2 *h2 = reinterpret_cast<__half2 *>(yp + i);
        h2[0] = __floats2half2_rn(yv.x * kQScale, yv.y * kQScale);
        h2[1] = __floats2half2_rn(yv.z * kQScale, yv.w * kQScale);
      }
    }
    for (int i = n4 + threadIdx.x; i < n; i += blockDim.x) {
      const float yi = ((kCg ? __ldcg(u + i) : u[i]) >= 0.0f) ? 1.0f : -1.0f;
      if (y) y[i] = yi;
      if (yp) yp[i] = __float2half_rn(yi * kQScale);
    }
    return;
  }
  float part = 0.0f;
  for (int i = 4 * threadIdx.x; i < n4; i += 4 * blockDim.x) {
    const float4 uv = kCg ? __ldcg(reinterpret_cast<const float4 *>(u + i)) : *reinterpret_cast<const float4 *>(u + i);
    part = fmaf(uv.x, uv.x, part);
    part = fmaf(uv.y, uv.y, part);
    part = fmaf(uv.z, uv.z, part);
    part = fmaf(uv.w, uv.w, part);
  }
  for (int i = n4 + threadIdx.x; i < n; i += blockDim.x) {
    const float ui = kCg ? __ldcg(u + i) : u[i];
    part = fmaf(ui, ui, part);
  }
  const float sumsq = block_sum_f(part, redf);
  if (sumsq == 0.0f) {
    float *x = X + (int64_t)c * ldX;
    for (int j = threadIdx.x; j < p; j += blockDim.x) x[j] = 0.0f;
    if (threadIdx.x == 0) {
      s.status[c] = SPCA_ST_DEGENERATE;
      s.nnz[c] = 0;
      s.F[c] = 0.0;
    }
    return;
  }
  float hi, lo, inv;
  norm_and_inverse(sumsq, &hi, &lo, &inv);
  // y = u / ||u||_2, and its planes: kQScale y is exact (a power of two), |kQScale y| <= 2^14
  auto planes = [&](float yi, __half &hi, __half &lo) {
    const float ys = yi * kQScale;
    hi = __float2half_rn(ys);
    lo = __float2half_rn(ys - __half2float(hi));
  };
  for (int i = 4 * threadIdx.x; i < n4; i += 4 * blockDim.x) {
    const float4 uv = kCg ? __ldcg(reinterpret_cast<const float4 *>(u + i)) : *reinterpret_cast<const float4 *>(u + i);
    const float4 yv = make_float4(uv.x * inv, uv.y * inv, uv.z * inv, uv.w * inv);
    if (y) *reinterpret_cast<float4 *>(y + i) = yv;
    if (yp) {
      __half h[4], l[4];
      planes(yv.x, h[0], l[0]);
      planes(yv.y, h[1], l[1]);
      planes(yv.z, h[2], l[2]);
      planes(yv.w, h[3], l[3]);
      __half2 *ph = reinterpret_cast<__half2 *>(yp + i);
      __half2 *pl = reinterpret_cast<__half2 *>(yp + pstride + i);
      ph[0] = __halves2half2(h[0], h[1]);
      ph[1] = __halves2half2(h[2], h[3]);
      pl[0] = __halves2half2(l[0], l[1]);
      pl[1] = __halves2half2(l[2], l[3]);
    }
  }
  for (int i = n4 + threadIdx.x; i < n; i += blockDim.x) {
    const float yi = (kCg ? __ldcg(u + i) : u[i]) * inv;
    if (y) y[i] = yi;
    if (yp) {
      __half hi, lo;
      planes(yi, hi, lo);
      yp[i] = hi;
      yp[i + pstride] = lo;
    }
  }
}

// ------------------------------------------------------------------ active-start list
// one CTA: ordered compaction of the flags status[c] == ST_ACTIVE over r starts (read from L2: other
// CTAs of the same launch may have written them), 4 consecutive starts per thread and round, their
// loads in flight together
static __device__ void active_list_body(const int *status, const int *nnz, int r, int *act, int *rank, Ctrl *ctrl) {
  __shared__ int warp_n[32];
  __shared__ long long red_l[32];
  __shared__ int red_m[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
  int base_pos = 0;
  long long nz = 0;
  int mz = 0;
  for (int base = 0; base < r; base += 4 * blockDim.x) {
    const int c0 = base + 4 * threadIdx.x;
    int s[4], k[4], mine = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      s[q] = c0 + q < r ? __ldcg(status + c0 + q) : ST_ACTIVE + 1;
      k[q] = nnz && c0 + q < r ? __ldcg(nnz + c0 + q) : 0;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (s[q] == ST_ACTIVE) {
        ++mine;
        nz += k[q];
        mz = max(mz, k[q]);
      }
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (base > 0) __syncthreads();   // (the last round's counts are read)
    if (lane == 31) warp_n[w] = incl;
    __syncthreads();
    const int n = lane < nw ? warp_n[lane] : 0;
    int pos = base_pos + incl - mine + __reduce_add_sync(0xffffffffu, lane < w ? n : 0);
    base_pos += __reduce_add_sync(0xffffffffu, n);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (s[q] == ST_ACTIVE) {
        act[pos] = c0 + q;
        rank[c0 + q] = pos++;
      }
  }
  // sum of the active support sizes (a bound on the size of their union)
  for (int o = 16; o > 0; o >>= 1) nz += __shfl_xor_sync(0xffffffffu, nz, o);
  mz = __reduce_max_sync(0xffffffffu, mz);
  if (lane == 0) {
    red_l[w] = nz;
    red_m[w] = mz;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    long long t = 0;
    int m = 0;
    for (int k = 0; k < nw; ++k) {
      t += red_l[k];
      m = max(m, red_m[k]);
    }
    ctrl->max_nnz = m;
    ctrl->active = base_pos;
    ctrl->use_gather = (nnz && __ldcg(&ctrl->need_dense) == 0 && base_pos > 0) ? 1 : 0;
    ctrl->sum_nnz = (int)(t < 0x7fffffffLL ? t : 0x7fffffffLL);
  }
}

// the last CTA of `total` to get here makes the active list of the next sweep (every CTA's thread 0 has
// written its start's status and counts: it releases them) and clears the control word that this sweep
// read (the next x-step writes it); a null nnz: the first list of a solve, whose x are dense
static __device__ __forceinline__ void last_makes_active_list(int total, const int *status, const int *nnz, int r,
                                                              int *act, int *rank, Ctrl *ctrl, Ctrl *ctrl_read) {
  __shared__ int last;
  if (threadIdx.x == 0) {
    int before;
    asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(before) : "l"(&ctrl->done) : "memory");
    last = before == total - 1;
    if (last && !nnz) ctrl->need_dense = 1;
  }
  __syncthreads();
  if (!last) return;
  active_list_body(status, nnz, r, act, rank, ctrl);
  if (threadIdx.x == 0) {
    if (ctrl_read) *ctrl_read = Ctrl{};
    if (!nnz) ctrl->done = 0;
  }
}

}  // namespace spca
