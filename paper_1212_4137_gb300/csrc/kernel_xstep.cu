// kernel_xstep.cu -- the x-step of Algorithm 2 for every active start (one CTA per start):
//   forms 1, 2   S3: T_s(v), the s largest |v_i| (ties: lower index)
//   forms 3, 4   S4: V_lambda(v) with lambda = lambda_s(v), the root of
//                    phi(lambda) = s ||V_lambda||_2^2 - ||V_lambda||_1^2
//   forms 5, 6   S5: U_gamma(v), keep v_i^2 > gamma  (eq. 5)
//   forms 7, 8   S6: V_gamma(v), soft threshold       (eq. 6)
// then normalisation (Section 2.2), the Table 3 value F(x^(k+1), y^(k)), the stopping rule,
// and the support list (ascending indices) used by the sparse u = A x and the FP64 objective.
// Section 4.1's gamma rule (penalty forms) picks gamma so that exactly s entries survive.
//
// Two paths: the threshold x-step (a short list of the entries above a lower bound of the operator's
// threshold, then the operator on the list), and the full pass for the starts it cannot serve: radix
// select, or bisection of phi, over all of v, staged in shared memory (p * 4 bytes up to
// XSTEP_SMEM_MAX, else read from global memory on every pass).  Reductions are in a fixed order that
// does not depend on the CTA's size: a start's result does not depend on the other starts or on
// scheduling.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "block_util.cuh"
#include "spca_internal.cuh"
#include "sweep_bodies.cuh"

namespace spca {

namespace {
constexpr int XT = 512;                        // threads per CTA of the full-pass kernels
constexpr int XW = 16;                         // index segments; a CTA's warps share them out
constexpr int XSTEP_SMEM_MAX = 200 * 1024;     // largest v staged in shared memory (bytes)
static_assert(kXstepSmemMaxP * 4 == XSTEP_SMEM_MAX, "the grouped x-step's split");

struct XShared {
  unsigned hist[256];
  double red_d[XW][2];
  float red_f[XW][2];
  int red_i[XW][2];
  int wcnt[32];                                // per-segment (or per-warp) counts of one pass
  int woff[XW];                                // their exclusive prefix over the segments
  int eoff[XW];                                // the same of the tied keys
  int digit, rem, cnt_bin;
  unsigned red_u[32];
};

struct Seg {
  int lo, hi;
};
// index segment w: 16 contiguous ranges, each a multiple of 32 long (the last shorter).  A pass takes
// them warp by warp (for_segments), and every sum is made per segment and then over the segments in
// order, so that its bits do not depend on the CTA's size.
__device__ __forceinline__ Seg index_seg(int p, int w) {
  const int seg = (((p + XW - 1) / XW) + 31) / 32 * 32;
  Seg s;
  s.lo = min(p, w * seg);
  s.hi = min(p, s.lo + seg);
  return s;
}
// (kOne: the CTA has XT threads, a warp per segment, and writes x.  Loops over segments and a test of x inside
// the passes keep them from being unrolled: 1024 starts of p = 20011, T_s, whole call 268 us for 212.)
template <bool kOne, typename Fn>
__device__ __forceinline__ void for_segments(int p, Fn &&fn) {
  if constexpr (kOne) {
    const int w = threadIdx.x >> 5;
    fn(w, index_seg(p, w));
  } else {
    for (int w = threadIdx.x >> 5; w < XW; w += blockDim.x >> 5) fn(w, index_seg(p, w));
  }
}

// sums of (f0, f1, i0, i1) over segment w, published by its warp ...
__device__ __forceinline__ void put_sum2f(int w, float f0, float f1, int i0, int i1, XShared &sh) {
  f0 = warp_sum_f(f0); f1 = warp_sum_f(f1); i0 = warp_sum_i(i0); i1 = warp_sum_i(i1);
  if ((threadIdx.x & 31) == 0) {
    sh.red_f[w][0] = f0; sh.red_f[w][1] = f1; sh.red_i[w][0] = i0; sh.red_i[w][1] = i1;
  }
}
// ... and added over the segments, FP32 in a fixed order; every thread gets them.
// (GB300's FP64 pipe is ~1/64 of FP32: FP64 stays out of the per-pass reductions.)
__device__ __forceinline__ void get_sum2f(float &f0, float &f1, int &i0, int &i1, XShared &sh) {
  __syncthreads();
  f0 = f1 = 0.0f; i0 = i1 = 0;
  for (int k = 0; k < XW; ++k) { f0 += sh.red_f[k][0]; f1 += sh.red_f[k][1]; i0 += sh.red_i[k][0]; i1 += sh.red_i[k][1]; }
  __syncthreads();
}

// the same for two FP64 values (each thread's value already accurate); the segments' partials are
// combined by one thread, so the FP64 work is ~5 adds per thread
__device__ __forceinline__ void put_sum2d(int w, double d0, double d1, XShared &sh) {
  d0 = warp_sum_d(d0); d1 = warp_sum_d(d1);
  if ((threadIdx.x & 31) == 0) { sh.red_d[w][0] = d0; sh.red_d[w][1] = d1; }
}
__device__ __forceinline__ void get_sum2d(double &d0, double &d1, XShared &sh) {
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0;
    for (int k = 0; k < XW; ++k) { a += sh.red_d[k][0]; b += sh.red_d[k][1]; }
    sh.red_d[0][0] = a; sh.red_d[0][1] = b;
  }
  __syncthreads();
  d0 = sh.red_d[0][0]; d1 = sh.red_d[0][1];
  __syncthreads();
}

// compensated (Neumaier) FP32 accumulation: s + c carries the sum to ~2^-40 relative
__device__ __forceinline__ void kahan_add(float &s, float &c, float x) {
  const float t = s + x;
  c += (fabsf(s) >= fabsf(x)) ? ((s - t) + x) : ((x - t) + s);
  s = t;
}

// the segments' counts (sh.wcnt) -> exclusive offsets over the segments (sh.woff) and the total
__device__ __forceinline__ int segment_offsets(XShared &sh) {
  __syncthreads();
  if (threadIdx.x == 0) {
    int acc = 0;
    for (int k = 0; k < XW; ++k) { sh.woff[k] = acc; acc += sh.wcnt[k]; }
    sh.cnt_bin = acc;
  }
  __syncthreads();
  return sh.cnt_bin;
}

// The j-th largest (1 <= j <= p) of the keys |v_i| by MSB-first radix select over the digits
// bits 30..23 (the exponent), 22..15, 14..7, 6..0.  Histogram updates are aggregated per warp.
// If the chosen bin is exactly the remainder of the top j before the last digit, the search
// stops: every element of the bin is in the top j.  Then, with exact == false, *K is the bin's
// lower bound and *whole = true; with exact == true one more pass finds the bin's minimum,
// which is the j-th largest key.  Otherwise *need_eq / *eq_total describe ties at *K.
template <bool kOne>
__device__ void radix_select(const float *vv, int p, int j, bool exact, XShared &sh, uint32_t *K,
                             bool *whole, int *need_eq, int *eq_total) {
  const int shifts[4] = {23, 15, 7, 0};
  const uint32_t wmask[4] = {0xFFu, 0xFFu, 0xFFu, 0x7Fu};
  const int lane = threadIdx.x & 31;
  uint32_t prefix = 0u, mask = 0u;
  int rem = j;
  *whole = false;
  for (int t = 0; t < 4; ++t) {
    const int sh_ = shifts[t];
    for (int b = threadIdx.x; b < 256; b += blockDim.x) sh.hist[b] = 0u;
    __syncthreads();
    for_segments<kOne>(p, [&](int, Seg sg) {
      for (int base = sg.lo; base < sg.hi; base += 32) {
        const int i = base + lane;
        const uint32_t key = (i < sg.hi) ? abs_key(vv[i]) : 0xFFFFFFFFu;
        const bool m = (i < sg.hi) && (key & mask) == prefix;
        const uint32_t bin = m ? (key >> sh_) & wmask[t] : 0xFFFFFFFFu;
        const unsigned peers = __match_any_sync(0xffffffffu, bin);
        if (m && lane == __ffs(peers) - 1) atomicAdd(&sh.hist[bin], (unsigned)__popc(peers));
      }
    });
    __syncthreads();
    if (threadIdx.x < 32) {
      // warp 0 finds the bin holding the rem-th largest: lane l owns the bins
      // [top - l*per, top - l*per - per + 1] (descending), scans the lane sums from the top,
      // and the owning lane walks its own bins
      const int nb = (int)wmask[t] + 1, per = nb / 32, top = nb - 1 - lane * per;
      int lsum = 0;
      for (int q = 0; q < per; ++q) lsum += (int)sh.hist[top - q];
      int incl = lsum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      const int excl = incl - lsum;
      const bool mine = excl < rem && rem <= incl;
      const unsigned who = __ballot_sync(0xffffffffu, mine);
      if (mine && lane == __ffs(who) - 1) {
        int acc = excl, d = top;
        for (int q = 0; q < per - 1; ++q, --d) {
          if (acc + (int)sh.hist[d] >= rem) break;
          acc += (int)sh.hist[d];
        }
        sh.digit = d;
        sh.rem = rem - acc;
        sh.cnt_bin = (int)sh.hist[d];
      }
    }
    __syncthreads();
    prefix |= (uint32_t)sh.digit << sh_;
    mask |= wmask[t] << sh_;
    rem = sh.rem;
    const int cnt = sh.cnt_bin;
    __syncthreads();
    if (t == 3) {
      *K = prefix;
      *need_eq = rem;
      *eq_total = cnt;
      return;
    }
    if (cnt == rem) {  // the whole bin belongs to the top j
      if (!exact) {
        *K = prefix;
        *whole = true;
        return;
      }
      unsigned mn = 0xFFFFFFFFu;
      for (int i = threadIdx.x; i < p; i += blockDim.x) {
        const uint32_t key = abs_key(vv[i]);
        if ((key & mask) == prefix) mn = min(mn, key);
      }
      // block minimum
      mn = __reduce_min_sync(0xffffffffu, mn);
      if (lane == 0) sh.red_u[threadIdx.x >> 5] = mn;
      __syncthreads();
      unsigned m2 = 0xFFFFFFFFu;
      for (int k = 0; k < (int)(blockDim.x >> 5); ++k) m2 = min(m2, sh.red_u[k]);
      __syncthreads();
      *K = m2;
      *whole = true;
      return;
    }
  }
}

// lambda_s(v) (Section 2.1) when phi(0) < 0.  Bisection over the float keys of lambda in
// [lo0, max|v|] (phi(lo0) < 0 is known: lo0 = 0, or a lower bound checked by the caller) on
// the sign of phi, stopping as soon as no |v_i| lies strictly inside the bracket (the active
// set is then fixed); then the root of phi on that piece in FP64.
// *lo_out: the active set is {key_i > *lo_out}.
template <bool kOne>
__device__ double lambda_s_bisect(const float *vv, int p, double s, uint32_t lo0, uint32_t maxkey, XShared &sh,
                                  uint32_t *lo_out) {
  const int lane = threadIdx.x & 31;
  uint32_t lo = lo0, hi = maxkey;  // phi(key lo) < 0 <= phi(key hi)
  while (hi - lo > 1u) {
    const uint32_t mid = lo + (hi - lo) / 2u;
    const float lam = __uint_as_float(mid);
    float sw, sw2;
    int in_lo, in_hi;          // elements strictly inside (lo, mid) and (mid, hi)
    for_segments<kOne>(p, [&](int seg, Seg sg) {
      sw = sw2 = 0.0f;
      in_lo = in_hi = 0;
      for (int i = sg.lo + lane; i < sg.hi; i += 32) {
        const float a = fabsf(vv[i]);
        const uint32_t key = __float_as_uint(a);
        if (a > lam) {
          const float w = a - lam;
          sw += w;
          sw2 = fmaf(w, w, sw2);
        }
        in_lo += (key > lo && key < mid);
        in_hi += (key > mid && key < hi);
      }
      put_sum2f(seg, sw, sw2, in_lo, in_hi, sh);
    });
    get_sum2f(sw, sw2, in_lo, in_hi, sh);
    const float phi = (float)s * sw2 - sw * sw;
    if (phi < 0.0f) {
      lo = mid;
      if (in_hi == 0) break;  // no magnitude strictly inside (mid, hi): active set fixed
    } else {
      hi = mid;
      if (in_lo == 0) break;
    }
  }
  // active set {key > lo}: k, S1, S2 (compensated per thread, FP64 across threads), then the
  // root of phi on this piece in FP64
  double s1, s2;
  float f_unused, f_unused2;
  int kc, i_unused;
  for_segments<kOne>(p, [&](int seg, Seg sg) {
    float a1 = 0.0f, c1 = 0.0f, a2 = 0.0f, c2 = 0.0f;
    kc = 0;
    for (int i = sg.lo + lane; i < sg.hi; i += 32) {
      const float a = fabsf(vv[i]);
      if (__float_as_uint(a) > lo) {
        ++kc;
        kahan_add(a1, c1, a);
        const float aa = a * a;
        kahan_add(a2, c2, aa);
        kahan_add(a2, c2, fmaf(a, a, -aa));   // exact square: aa + the FMA residual
      }
    }
    put_sum2d(seg, (double)a1 + (double)c1, (double)a2 + (double)c2, sh);
    put_sum2f(seg, 0.0f, 0.0f, kc, 0, sh);
  });
  get_sum2d(s1, s2, sh);
  get_sum2f(f_unused, f_unused2, kc, i_unused, sh);
  const double k = (double)kc;
  const double flo = (double)__uint_as_float(lo), fhi = (double)__uint_as_float(hi);
  double lam;
  if (k <= s) {
    lam = flo;
  } else {
    double disc = s * (k * s2 - s1 * s1) / (k - s);
    if (disc < 0.0) disc = 0.0;
    lam = (s1 - sqrt(disc)) / k;
    lam = fmin(fmax(lam, flo), fhi);
  }
  *lo_out = lo;
  return lam;
}

// ---------------------------------------------------------------- the operator, then x
// mode 0: T_s with ties: keep key > K, plus the first need_eq of key == K in index order
// mode 1: hard threshold: keep key > tkey, value v            (U_gamma; T_s otherwise)
// mode 2: soft threshold: keep key > tkey, value sgn(v)(|v|-t)  (V_gamma, V_lambda)
struct XOp {
  int mode = 1;
  uint32_t K = 0u, tkey = 0u;
  int need_eq = 0;
  float tval = 0.0f;    // threshold value subtracted in mode 2
  double gam = 0.0;     // gamma in Table 1 units (penalties) or lambda_s (S4)
  float tnext = 0.0f;   // the threshold (|v| units) that seeds the next sweep's candidate filter
};

// Pass A (||w||_2^2 and nnz of the unnormalised result w), the Table 3 value, pass B (x = w /
// ||w||_2 and the support list in index order) and the per-start outputs, over vv[0 .. len).
template <bool kOne>
__device__ void xstep_finish(const XstepArgs &a, int c, const float *vv, int len, const XOp &op, float *x,
                             StartState st, int *sup_idx, float *sup_val, Ctrl *ctrl, XShared &sh) {
  const int lane = threadIdx.x & 31;
  const int form = a.form;

  // ---- ties (mode 0): offsets of each segment's equal keys in index order
  if (op.mode == 0) {
    for_segments<kOne>(len, [&](int seg, Seg sg) {
      int eq = 0;
      for (int i = sg.lo + lane; i < sg.hi; i += 32) eq += abs_key(vv[i]) == op.K;
      eq = warp_sum_i(eq);
      if (lane == 0) sh.wcnt[seg] = eq;
    });
    segment_offsets(sh);
  }
  if (threadIdx.x < XW) sh.eoff[threadIdx.x] = op.mode == 0 ? sh.woff[threadIdx.x] : 0;
  __syncthreads();
  const unsigned lt_mask = (1u << lane) - 1u;

  auto wval = [&](float vi, uint32_t key, bool tie_keep) -> float {
    if (op.mode == 0) return (key > op.K || (key == op.K && tie_keep)) ? vi : 0.0f;
    if (key <= op.tkey) return 0.0f;
    if (op.mode == 1) return vi;
    return copysignf(fabsf(vi) - op.tval, vi);
  };
  for_segments<kOne>(len, [&](int seg, Seg sg) {
    float part = 0.0f;
    int wnnz = 0;
    int eq_run = sh.eoff[seg];
    for (int base = sg.lo; base < sg.hi; base += 32) {
      const int i = base + lane;
      const float vi = (i < sg.hi) ? vv[i] : 0.0f;
      const uint32_t key = abs_key(vi);
      bool tie_keep = false;
      if (op.mode == 0) {
        const unsigned b = __ballot_sync(0xffffffffu, i < sg.hi && key == op.K);
        tie_keep = (eq_run + __popc(b & lt_mask)) < op.need_eq;
        eq_run += __popc(b);
      }
      const float w = (i < sg.hi) ? wval(vi, key, tie_keep) : 0.0f;
      part = fmaf(w, w, part);
      wnnz += __popc(__ballot_sync(0xffffffffu, w != 0.0f));
    }
    if (lane == 0) sh.wcnt[seg] = wnnz;
    put_sum2f(seg, part, 0.0f, 0, 0, sh);
  });
  float part, fz;
  int zz, zz2;
  get_sum2f(part, fz, zz, zz2, sh);
  const int nnz = segment_offsets(sh);   // sh.woff: each segment's first slot in the support list
  float nrm_hi, nrm_lo, inv;
  norm_and_inverse(part, &nrm_hi, &nrm_lo, &inv);

  // ---- Table 3 value of the subproblem
  // (by the thread that uses it, below: FP64 is slow)
  auto value = [&]() -> double {
    const double nrm = norm_fp64(part, nrm_hi, nrm_lo);
    if (uses_lam(form)) return op.gam * a.sqrt_s + nrm;       // S4: lambda sqrt(s) + ||V||_2
    if (uses_U(form)) return (double)part - op.gam * (double)nnz;     // S5: ||U||^2 - gamma ||U||_0
    return nrm;                                                // S3: ||T_s(v)||_2, S6: ||V_gamma(v)||_2
  };

  // ---- pass B
  int *gi = sup_idx ? sup_idx + (int64_t)c * a.cap : nullptr;
  float *gv = sup_val ? sup_val + (int64_t)c * a.cap : nullptr;
  for_segments<kOne>(len, [&](int seg, Seg sg) {
    int eq_run = sh.eoff[seg];
    int pos = sh.woff[seg];
    for (int base = sg.lo; base < sg.hi; base += 32) {
      const int i = base + lane;
      const float vi = (i < sg.hi) ? vv[i] : 0.0f;
      const uint32_t key = abs_key(vi);
      bool tie_keep = false;
      if (op.mode == 0) {
        const unsigned b = __ballot_sync(0xffffffffu, i < sg.hi && key == op.K);
        tie_keep = (eq_run + __popc(b & lt_mask)) < op.need_eq;
        eq_run += __popc(b);
      }
      const float w = (i < sg.hi) ? wval(vi, key, tie_keep) : 0.0f;
      const float xi = w * inv;
      if ((kOne || x) && i < sg.hi) x[i] = xi;
      // (listed by w, as nnz counts: x may underflow to 0 where w does not, and the list has nnz entries)
      const unsigned nzb = __ballot_sync(0xffffffffu, w != 0.0f);
      if (gi && w != 0.0f) {
        const int q = pos + __popc(nzb & lt_mask);
        if (q < a.cap) {
          gi[q] = i;
          gv[q] = xi;
        }
      }
      pos += __popc(nzb);
    }
  });

  // ---- outputs, stopping rule (Section 2.2), control words for the next sweep
  if (threadIdx.x == 0) {
    const double F = value();
    if (st.F) st.F[c] = F;
    if (st.nnz) st.nnz[c] = nnz;
    if (st.gamma) st.gamma[c] = op.gam;
    if (st.tprev) st.tprev[c] = op.tnext;
    if (st.status) {
      int status = ST_ACTIVE;
      if (part == 0.0f) {
        status = SPCA_ST_DEGENERATE;
      } else if (a.stop_test && F <= (1.0 + a.tol) * st.F_prev[c]) {
        status = SPCA_ST_CONVERGED;
      } else if (st.iters[c] >= a.max_iter) {
        status = SPCA_ST_MAXITER;
      }
      st.F_prev[c] = F;
      st.status[c] = status;
      // (the active count and list for the next sweep are built after this kernel)
      if (status == ST_ACTIVE && ctrl && nnz > a.sparse_cap) atomicOr(&ctrl->need_dense, 1);
    }
  }
}

// ---------------------------------------------------------------- full x-step
// the full x-step of start c (block-wide; kSmem: by XT threads, with v staged in vsm, p floats of shared
// memory; kOne: see for_segments)
template <bool kSmem, bool kOne>
__device__ void xstep_full_one(const XstepArgs &a_in, int c, const float *__restrict__ V, int64_t ldv,
                               float *__restrict__ X, int64_t ldx, StartState &st, int *__restrict__ sup_idx,
                               float *__restrict__ sup_val, Ctrl *ctrl, float *vsm, XShared &sh) {
  const XstepArgs a = xstep_switches(a_in, st.iters ? st.iters[c] : 0);
  const int p = a.p;
  const int lane = threadIdx.x & 31;
  const float *vg = V + (int64_t)c * ldv;
  float *x = X ? X + (int64_t)c * ldx : nullptr;   // (null: the support list is all that is wanted)
  const int form = a.form;
  if (kSmem) {
    for (int i = threadIdx.x; i < p; i += XT) vsm[i] = vg[i];
    __syncthreads();
  }
  const float *vv = kSmem ? vsm : vg;

  XOp op;
  const int s_int = (int)a.s;
  if (uses_T(form)) {
    op.mode = 1;
    if (s_int < p) {
      bool whole;
      int eq_total;
      radix_select<kOne>(vv, p, s_int, false, sh, &op.K, &whole, &op.need_eq, &eq_total);
      op.tnext = __uint_as_float(op.K);
      if (whole) {
        op.tkey = op.K == 0u ? 0u : op.K - 1u;   // keep every key >= the bin's lower bound
      } else if (op.K == 0u || op.need_eq >= eq_total) {
        op.tkey = op.K == 0u ? 0u : op.K - 1u;   // no ties to break: keep key >= K
      } else {
        op.mode = 0;
      }
    }
  } else if (uses_lam(form)) {
    // phi(0) = s ||v||_2^2 - ||v||_1^2 >= 0: the L1 ball is not binding, lambda = 0
    float f1, f2;
    unsigned mk = 0u;
    for_segments<kOne>(p, [&](int seg, Seg sg) {
      f1 = f2 = 0.0f;
      for (int i = sg.lo + lane; i < sg.hi; i += 32) {
        const float av = fabsf(vv[i]);
        f1 += av;
        f2 = fmaf(av, av, f2);
        mk = max(mk, __float_as_uint(av));
      }
      put_sum2f(seg, f1, f2, 0, 0, sh);
    });
    int d0 = 0, d1 = 0;
    get_sum2f(f1, f2, d0, d1, sh);
    const uint32_t maxkey = block_max_u(mk, sh.red_u);
    op.mode = 2;
    if ((float)a.s * f2 - f1 * f1 < 0.0f) {
      uint32_t lo;
      op.gam = lambda_s_bisect<kOne>(vv, p, a.s, 0u, maxkey, sh, &lo);
      op.tkey = lo;
      op.tval = (float)op.gam;
      op.tnext = op.tval;
    }
  } else {  // penalties
    op.mode = uses_U(form) ? 1 : 2;
    if (a.calibrate) {
      const int j = s_int + 1;
      uint32_t tk = 0u;
      if (j <= p) {
        int ne, et;
        bool whole;
        radix_select<kOne>(vv, p, j, true, sh, &tk, &whole, &ne, &et);
      }
      op.tkey = tk;
      op.tval = __uint_as_float(tk);
      op.gam = uses_U(form) ? (double)op.tval * (double)op.tval : (double)op.tval;
      op.tnext = op.tval;
      if (threadIdx.x == 0 && st.thr) st.thr[c] = op.tval;
    } else if (a.per_start_thr) {
      op.tval = st.thr[c];
      op.gam = st.gamma[c];
      op.tkey = __float_as_uint(op.tval);
    } else {
      op.tval = a.thr_fixed;
      op.gam = a.gamma_fixed;
      op.tkey = __float_as_uint(op.tval);
    }
  }
  xstep_finish<kOne>(a, c, vv, p, op, x, st, sup_idx, sup_val, ctrl, sh);
}

// Every pass over all p entries of v (staged in shared memory when it fits), persistent CTAs over
// the starts that the threshold x-step below left (xfast = 0, or nnz = -1 without xfast), or over every
// active start.
template <bool kSmem>
__global__ void __launch_bounds__(XT) k_xstep(XstepArgs a_in, const float *__restrict__ V, int64_t ldv, int r,
                                              float *__restrict__ X, int64_t ldx, StartState st,
                                              int *__restrict__ sup_idx, float *__restrict__ sup_val,
                                              Ctrl *ctrl, int every) {
  extern __shared__ float vsm[];
  __shared__ XShared sh;
  for (int c = blockIdx.x; c < r; c += gridDim.x) {
    if (st.status && st.status[c] != ST_ACTIVE) continue;
    if (!every && (st.xfast ? st.xfast[c] != 0 : st.nnz[c] != -1)) continue;
    __syncthreads();   // (every thread has read the mark; shared memory is reused from start to start)
    xstep_full_one<kSmem, true>(a_in, c, V, ldv, X, ldx, st, sup_idx, sup_val, ctrl, vsm, sh);
    if (threadIdx.x == 0 && st.xfast) st.xfast[c] = 2;
    __syncthreads();
  }
}


// ---------------------------------------------------------------- threshold x-step
// Every operator keeps only entries above a threshold (the s-th or (s+1)-th largest |v_i|, lambda_s,
// or the penalty's threshold), so a lower bound G of it turns the x-step into one coalesced pass that
// lists the entries above G (in index order, a short list) and the operator on that list in shared
// memory.  The bound comes from
//   - a fixed threshold itself (exact);
//   - last sweep's threshold t: G = kGuess t (kGuessSteady t while t holds steady);
//   - the maxima of 512 or 2048 disjoint subsets of v (one more pass), the same ones whatever the CTA's size: at
//     least j entries lie at or above the j-th largest of them, and for j well below their number not many more;
//   - 0 for a very short v: the list holds every nonzero entry.
// A bound is checked before it is used: at least s (or s + 1) listed entries for the selections,
// phi(G) < 0 for lambda_s (phi increases through its root); then the list holds every surviving
// entry and the result is that of a pass over all of v.  A start that no bound serves (more than
// kFastSegCap entries above it in one of the 16 segments, lambda_s = 0, s beyond the list) takes the full
// pass.  Bound, list and these choices do not depend on the CTA's size, so neither does the path that a
// start takes nor any bit of its result: in a group, whose starts and longest v choose the size, a member
// has the same bits alone and in any mix.
//
// One CTA does all of it for a start, in one launch per sweep, and the CTA that finishes last makes
// the active list of the next sweep.  What bounds it is each start's chain of dependent steps (reads
// of v from L2 or HBM, then about ten block barriers), so the chain is short: ranks are counted by
// all threads at once instead of selected bit by bit by one warp, lambda_s takes a few monotone
// steps instead of a bisection, and FP64 (1/64 of the FP32 rate) is left to single threads.
// 1024 starts, p = 20011, lambda_s (spca_xstep, the whole call): 119 us, 390 us for the full pass in
// shared memory.  A solve's x-step and active list per sweep, before (filter, one-warp operator, full
// pass and list: four launches) and now: p = 20000, T_s, 1024 starts 90 -> 46 us; p = 100000, V_gamma,
// 16 starts 57 -> 23 us; p = 20000, lambda_s, one start 44 -> 25 us (CUDA events, a few us included).
constexpr int kFastCand = 1024;                // listed entries per start
constexpr int kFastBins = 2048, kFastShift = 17;   // bins of 2^-6 octave below the largest |v_i|
constexpr int kFastSubsets = 2048;             // disjoint subsets of v whose maxima bound the threshold (or 512)
constexpr int kCoarseJ = 170, kCoarseMaxJ = 200;   // j of the maxima of 512 subsets
constexpr int kFastAllP = 64;                  // v up to this long: list every nonzero entry
// j of the subset maxima: some 570 entries lie above the bound for 500, 36 in a segment, and rarely more than
// the 64 that a segment may list (for 600 more than that in every other start)
constexpr int kFastMaxJ = 500;
constexpr int kFastMaxNeed = 600;              // selected entries, above last sweep's bound
// Entries of v per selected one below which the full pass is the faster one: ranks are counted against the
// whole list, so their cost grows with its square (20 sweeps of 16 starts by T_s, list and full pass:
// p = 1000, s = 333 1.7 times the time, s = 166 as long; p = 1500, s = 300 1.08, s = 187 0.97; p = 3000,
// s = 600 1.24, s = 500 1.14, s = 375 0.99)
constexpr int kFastPerNeed = 6;
constexpr float kGuess = 0.85f;
constexpr float kGuessSteady = 0.95f;          // while t holds steady
constexpr float kGuessLo = 0.6f;
constexpr float kHint = 0.98f;
constexpr float kSteady = 0.05f;               // |t_new / t - 1| below this: t holds steady
constexpr int kSegOrderP = 4096;               // see xstep_fast_one, "the order of ||w||^2"
constexpr int kFastSegCap = kFastCand / XW;    // ... and per index segment (a sixteenth of v)

template <int T>
struct FastShared {
  static constexpr int W = T / 32;
  // a warp lists 16 / W segments, or half of one
  static constexpr int kSegs = W < XW ? XW / W : 1, kWarpCap = kSegs * kFastSegCap;
  union {
    struct {
      float wv[W * kWarpCap];                  // per-warp lists
      int wi[W * kWarpCap];
    } w;
    int rank[kFastCand];
    uint32_t maxima[kFastSubsets];
    struct {
      float val[kFastCand];                    // the surviving entries, in index order
      int idx[kFastCand];
    } s;
  } a;
  union {
    struct {
      float cv[kFastCand];                     // the list, in index order
      int ci[kFastCand];
    } l;
    float by_index[2 * kFastCand];
    unsigned hist[kFastBins];
  } u;
  float4 red[2][W];                            // (used alternately: one barrier per exchange)
  int cnt[kFastCand / 32];
  double lam;                                  // lambda_s, or < 0: the bound is too high
  XShared sh;
};

// A row of v read as aligned 16-byte vectors wherever it starts: entry i is at q = i + sh of the aligned
// base b.  The vectors at lo4 .. hi4 - 4 lie inside the row; the one at 0 (sh > 0) and the one at hi4 (end no
// multiple of 4) cross an end.  Those are read entry by entry, once a pass and not at every load: an
// x-step's warps stall for instructions more than for anything else, and that code at every load was a third of
// a pass.
struct Row {
  const float *b;
  int sh, end;                                 // valid q: sh .. end - 1
  int lo4, hi4;
};
__device__ __forceinline__ Row row_of(const float *v, int p) {
  Row r;
  r.sh = (int)((reinterpret_cast<uintptr_t>(v) >> 2) & 3u);
  r.b = v - r.sh;
  r.end = p + r.sh;
  r.lo4 = r.sh > 0 ? 4 : 0;
  r.hi4 = r.end & ~3;
  return r;
}
// entries q .. q + 3 (q a multiple of 4) of a vector inside the row and below hi, else 0
__device__ __forceinline__ float4 row_load(const Row &r, int q, int hi) {
  return q >= r.lo4 && q < min(hi, r.hi4) ? *reinterpret_cast<const float4 *>(r.b + q)
                                          : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
}
// entry q of the row, 0 outside
__device__ __forceinline__ float row_entry(const Row &r, int q) { return q >= r.sh && q < r.end ? r.b[q] : 0.0f; }
__device__ __forceinline__ float4 row_vector(const Row &r, int q) {
  return make_float4(row_entry(r, q), row_entry(r, q + 1), row_entry(r, q + 2), row_entry(r, q + 3));
}
// where the vector over the row's end begins (-1: none, or it is the one over its beginning)
__device__ __forceinline__ int row_last(const Row &r) { return r.hi4 < r.end && r.hi4 >= r.lo4 ? r.hi4 : -1; }
// the entries of the vectors that cross an end, one for each of the first eight threads: its place, or -1
__device__ __forceinline__ int edge_entry(const Row &r, int t) {
  const int q = t < 4 ? t : row_last(r) + t - 4;
  const bool is = t < 4 ? r.sh > 0 : t < 8 && row_last(r) >= 0;
  return is && q >= r.sh && q < r.end ? q : -1;
}

// a lower bound of the j-th largest |v_i| from the maxima of 512 or 2048 subsets: the lower edge of the
// histogram bin of the j-th largest maximum.  0 when the bins do not resolve it.
// lam_s > 0, for lambda_s: the maxima are a sample of v's largest entries, so phi over them tells, but for a
// few percent, whether lambda_s lies above the bound.  If not for j, a larger one is taken (j becomes it), half as
// much again each time; if not for kFastMaxJ either, kNoBound: the start's active set is longer than the list, as
// one pass has shown.  (Sums over whole counts in a fixed order: not a matter of T.)
constexpr uint32_t kNoBound = 0xFFFFFFFFu;
__device__ __forceinline__ int bin_of_rank(const unsigned *hist, int j) {
  // one warp: the first bin, from the largest down, whose running count reaches j (64 bins a step: the
  // largest maxima lie within a few octaves)
  const int lane = threadIdx.x & 31;
  int acc = 0;
  for (int base = 0; base < kFastBins; base += 64) {
    const int h0 = (int)hist[base + 2 * lane], h1 = (int)hist[base + 2 * lane + 1];
    int incl = h0 + h1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    const int before = acc + incl - h0 - h1;
    const unsigned here = __ballot_sync(0xffffffffu, before < j && j <= acc + incl);
    if (here) return __shfl_sync(0xffffffffu, base + 2 * lane + (before + h0 >= j ? 0 : 1), __ffs(here) - 1);
    acc += __shfl_sync(0xffffffffu, incl, 31);
  }
  return kFastBins - 1;
}
// keys of bins 0 .. bin are above this one; 0 for the last bin (it holds all smaller keys)
__device__ __forceinline__ uint32_t bin_edge(uint32_t top, int bin) {
  const uint32_t down = (uint32_t)(bin + 1) << kFastShift;
  return bin >= kFastBins - 1 || down >= top ? 0u : top - down;
}
// (n_sub: the subsets that v's p entries are spread over)
__device__ __forceinline__ bool root_above(const unsigned *hist, uint32_t top, int bin, float s, int p, int n_sub) {
  const uint32_t Gk = bin_edge(top, bin);
  if (Gk == 0u) return true;
  const int lane = threadIdx.x & 31;
  const float G = __uint_as_float(Gk);
  float w1 = 0.0f, w2 = 0.0f;
  int n = 0;
  for (int b = lane; b <= bin; b += 32) {
    const int h = (int)hist[b];
    const float w = __uint_as_float(top - ((uint32_t)b << kFastShift) - (1u << (kFastShift - 1))) - G;
    w1 = fmaf((float)h, w, w1);
    w2 = fmaf((float)h * w, w, w2);
    n += h;
  }
  w1 = warp_sum_f(w1);
  w2 = warp_sum_f(w2);
  n = warp_sum_i(n);
  // of m entries above G, spread over subsets of q entries each, n are their subset's maximum
  const float sub = (float)n_sub, q = fmaxf(1.0f, (float)p / sub);
  const float m = sub * q * (1.0f - powf(1.0f - (float)n / sub, 1.0f / q));
  return s * w2 < 1.02f * (m / (float)n) * (w1 * w1);
}
// The histogram of the subset maxima (fs.u.hist; the return value: the largest of them, bin 0): 2048 subsets
// (kFine) or 512, the entries at q, q + 2048 or 512, ... of the row.  A thread has G groups of four subsets, load k
// belonging to group k mod G; threads that share subsets meet in shared memory.
template <int T, bool kFine>
__device__ __forceinline__ uint32_t subset_maxima(const Row &row, FastShared<T> &fs) {
  constexpr int CH = T > 256 ? 4 : 8;          // loads in flight per thread
  constexpr int N = kFine ? kFastSubsets : kFastSubsets / 4, G = N > 4 * T ? N / (4 * T) : 1;
  static_assert(CH % G == 0, "a step covers whole rounds of the subsets");
  uint32_t *sub = fs.a.maxima;
  for (int b = threadIdx.x; b < kFastBins; b += T) {
    fs.u.hist[b] = 0u;
    if (b < N) sub[b] = 0u;
  }
  uint32_t m[G][4];
#pragma unroll
  for (int k = 0; k < G; ++k) m[k][0] = m[k][1] = m[k][2] = m[k][3] = 0u;
  for (int q0 = 4 * threadIdx.x; q0 < row.end; q0 += 4 * T * CH) {
    float4 t[CH];
#pragma unroll
    for (int k = 0; k < CH; ++k) t[k] = row_load(row, q0 + 4 * T * k, row.end);
#pragma unroll
    for (int k = 0; k < CH; ++k) {
      m[k % G][0] = max(m[k % G][0], abs_key(t[k].x));
      m[k % G][1] = max(m[k % G][1], abs_key(t[k].y));
      m[k % G][2] = max(m[k % G][2], abs_key(t[k].z));
      m[k % G][3] = max(m[k % G][3], abs_key(t[k].w));
    }
  }
  __syncthreads();                             // (the zeros)
#pragma unroll
  for (int k = 0; k < G; ++k)
#pragma unroll
    for (int e = 0; e < 4; ++e) atomicMax(&sub[(4 * (threadIdx.x + T * k) + e) & (N - 1)], m[k][e]);
  const int q = edge_entry(row, (int)threadIdx.x);
  if (q >= 0) atomicMax(&sub[q & (N - 1)], abs_key(row.b[q]));
  __syncthreads();
  uint32_t all = 0u;
  for (int b = threadIdx.x; b < N; b += T) all = max(all, sub[b]);
  const uint32_t top = block_max_u(all, fs.sh.red_u);
  for (int b = threadIdx.x; b < N; b += T)
    atomicAdd(&fs.u.hist[min((top - sub[b]) >> kFastShift, (uint32_t)kFastBins - 1u)], 1u);
  __syncthreads();
  return top;
}
template <int T>
__device__ __noinline__ uint32_t subset_maxima_fine(const Row &row, FastShared<T> &fs) {
  return subset_maxima<T, true>(row, fs);
}

template <int T>
__device__ __forceinline__ uint32_t subset_bound(const Row &row, int &j, float lam_s, FastShared<T> &fs) {
  // up to kCoarseJ the maxima of 512 subsets do (a list of 200 entries for j = 166, 173 with 2048), and the CTA
  // saves three quarters of the updates of the histogram (1024 starts of p = 20011: 19 us); a lambda_s that lies
  // lower than their limit takes the pass again with 2048
  bool fine = j > kCoarseJ;
  for (;;) {
    const uint32_t top = fine ? subset_maxima_fine<T>(row, fs) : subset_maxima<T, false>(row, fs);
    const int limit = fine ? kFastMaxJ : kCoarseMaxJ, n_sub = fine ? kFastSubsets : kFastSubsets / 4;
    if (threadIdx.x < 32) {
      int jn = j, bin = bin_of_rank(fs.u.hist, jn);
      while (lam_s > 0.0f && bin >= 0 && !root_above(fs.u.hist, top, bin, lam_s, row.end - row.sh, n_sub)) {
        const bool longer = jn < limit;
        jn = min(limit, jn + jn / 2);
        bin = longer ? bin_of_rank(fs.u.hist, jn) : -1;
      }
      if (threadIdx.x == 0) {
        fs.sh.digit = bin;
        fs.sh.rem = jn;
      }
    }
    __syncthreads();
    const int bin = fs.sh.digit;
    j = fs.sh.rem;
    if (bin >= 0 || fine) return bin < 0 ? kNoBound : bin_edge(top, bin);
    fine = true;
    __syncthreads();                 // (the result is read, and the histogram)
  }
}

// An index segment of more than 1024 entries of v (a sixteenth, as list_above cuts it)
__device__ __forceinline__ int list_seg(const Row &row) { return ((row.end + XW - 1) / XW + 127) / 128 * 128; }

// Whether the first segment alone holds more entries above a fixed threshold than the list takes: any number
// of entries may survive one, and a start with too many should go to the full pass without a pass over v
// (1024 starts of p = 20011, half of v above: 172 us for a whole call of 109 us before).
template <int T>
__device__ __forceinline__ bool first_segment_full(const Row &row, uint32_t Gk, FastShared<T> &fs) {
  if (row.end <= kFastCand) return false;
  const int hi = min(row.end, list_seg(row));
  int n = 0;
  for (int q = 4 * threadIdx.x; q < hi; q += 4 * T) {
    const float4 e = row_load(row, q, hi);
    n += (abs_key(e.x) > Gk) + (abs_key(e.y) > Gk) + (abs_key(e.z) > Gk) + (abs_key(e.w) > Gk);
  }
  const int qe = edge_entry(row, (int)threadIdx.x);
  if (qe >= 0 && qe < hi) n += abs_key(row.b[qe]) > Gk;
  return block_sum_i(n, reinterpret_cast<int *>(fs.sh.red_u)) > kFastSegCap;
}

// Lists the entries with key > Gk in index order (fs.u.l.cv / ci, *ncand of them) and, for the
// lambda forms, the block sums of |v| and v^2; false when a segment (a sixteenth of v) holds more than
// kFastSegCap of them, whatever the number of warps.
template <int T>
__device__ __forceinline__ bool list_above(const Row &row, uint32_t Gk, bool sums, FastShared<T> &fs, int &buf,
                                           int *ncand, float *f1_out, float *f2_out) {
  using FS = FastShared<T>;
  constexpr int W = FS::W;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  // this warp's range: its segments (a sixteenth each, a multiple of 128 entries), or half of one; a v
  // no longer than the list is shared out evenly, and any part of it fits
  int lo, hi, seg_chunks = 1 << 30;            // 128-entry chunks per segment
  if (row.end <= kFastCand) {
    const int per = ((row.end + W - 1) / W + 3) / 4 * 4;
    lo = min(row.end, w * per);
    hi = min(row.end, lo + per);
  } else {
    const int seg = list_seg(row);
    if (W <= XW) {
      lo = min(row.end, w * FS::kSegs * seg);
      hi = min(row.end, lo + FS::kSegs * seg);
      seg_chunks = seg / 128;
    } else {
      lo = min(row.end, (w >> 1) * seg + (w & 1) * (seg / 2));
      hi = min(row.end, (w >> 1) * seg + (w & 1 ? seg : seg / 2));
    }
  }
  float *wv = fs.a.w.wv + w * FS::kWarpCap;
  int *wi = fs.a.w.wi + w * FS::kWarpCap;
  int wc = 0, wc0 = 0, chunk = 0;              // wc0: the list's length where the segment began
  bool over = false;
  float f1 = 0.0f, f2 = 0.0f;
  // CH 128-entry chunks per step, the next step's loads in flight while this one is used
  constexpr int CH = T == 1024 ? 3 : 4;
  float4 e[CH], nx[CH];
#pragma unroll
  for (int h = 0; h < CH; ++h) e[h] = row_load(row, lo + h * 128 + 4 * lane, hi);
  if (lo == 0 && hi > 0 && row.sh > 0 && lane == 0) e[0] = row_vector(row, 0);
  int at_end = row_last(row);                  // the vector over the row's end, if it is this lane's
  float4 end_v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  if (at_end < lo || at_end >= hi || ((at_end - lo) & 127) != 4 * lane) at_end = -1;
  if (at_end >= 0) end_v = row_vector(row, at_end);
  for (int base = lo; base < hi && !over; base += 128 * CH) {
#pragma unroll
    for (int h = 0; h < CH; ++h) nx[h] = row_load(row, base + (CH + h) * 128 + 4 * lane, hi);
#pragma unroll
    for (int h = 0; h < CH; ++h) {
      if (chunk == seg_chunks) {
        chunk = 0;
        wc0 = wc;
      }
      ++chunk;
      if (base + h * 128 + 4 * lane == at_end) e[h] = end_v;
      const float ev[4] = {e[h].x, e[h].y, e[h].z, e[h].w};
      if (sums) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float av = fabsf(ev[k]);
          f1 += av;
          f2 = fmaf(av, av, f2);
        }
      }
      int cnt = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) cnt += abs_key(ev[k]) > Gk ? 1 : 0;   // (the 0s past an end are never above)
      if (!__any_sync(0xffffffffu, cnt != 0)) continue;   // the common case: nothing above the bound
      // the warp's exclusive prefix of cnt (0..4) from the ballots of its three bits
      const unsigned b0 = __ballot_sync(0xffffffffu, cnt & 1), b1 = __ballot_sync(0xffffffffu, cnt & 2),
                     b2 = __ballot_sync(0xffffffffu, cnt & 4);
      const int tot = __popc(b0) + 2 * __popc(b1) + 4 * __popc(b2);
      if (wc + tot > FS::kWarpCap || (seg_chunks < (1 << 30) && wc - wc0 + tot > kFastSegCap)) {
        over = true;
        break;
      }
      int q = wc + __popc(b0 & lt) + 2 * __popc(b1 & lt) + 4 * __popc(b2 & lt);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (abs_key(ev[k]) > Gk) {
          wv[q] = ev[k];
          wi[q] = base + h * 128 + 4 * lane + k - row.sh;
          ++q;
        }
      }
      wc += tot;
    }
#pragma unroll
    for (int h = 0; h < CH; ++h) e[h] = nx[h];
  }
  if (sums) {
    f1 = warp_sum_f(f1);
    f2 = warp_sum_f(f2);
  }
  if (lane == 0) fs.red[buf][w] = make_float4(f1, f2, __int_as_float(wc), __int_as_float(over ? 1 : 0));
  __syncthreads();   // (also: the histogram's readers are done before the list overwrites it)
  // lane q looks at warp q
  const float4 t = lane < W ? fs.red[buf][lane] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  buf ^= 1;
  const int n = __float_as_int(t.z);
  bool too_many = __float_as_int(t.w) != 0;
  if (W > XW) {      // two warps to a segment
    const int both = n + __shfl_xor_sync(0xffffffffu, n, 1);
    too_many = too_many || (row.end > kFastCand && both > kFastSegCap);
  }
  int incl = n;
#pragma unroll
  for (int o = 1; o < W; o <<= 1) {
    const int up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  const int off = __shfl_sync(0xffffffffu, incl - n, w);
  *ncand = __shfl_sync(0xffffffffu, incl, W - 1);
  if (sums) {
    *f1_out = warp_sum_f(t.x);
    *f2_out = warp_sum_f(t.y);
  }
  if (__any_sync(0xffffffffu, too_many)) return false;
  __syncwarp();
  for (int t = lane; t < wc; t += 32) {
    fs.u.l.cv[off + t] = wv[t];
    fs.u.l.ci[off + t] = wi[t];
  }
  __syncthreads();
  return true;
}

// lambda_s over the list, by one warp; < 0 when phi(G) >= 0 (the bound is too high).
// For the set S of entries above a lower bound of the root, the root of phi restricted to S is a lower
// bound again (an entry below the root adds to phi), so raising the bound to it and dropping the
// entries below converges monotonically to the active set.  The steps run in FP32, on w = |v| - lo and
// lowered by their rounding error, from `hint` when phi(hint) < 0 and from G otherwise; the last ones,
// on compensated sums, end when no entry lies between the bound and the root: the result is the root
// of phi on its own active set, by two FP64 Newton steps from its FP32 value (FP64's division and
// square root took longer than all of the steps).
__device__ __forceinline__ double list_lambda(const float *cv, int ncand, float s, double s_d, float G, float hint) {
  const int lane = threadIdx.x & 31;
  float lo = hint > G ? hint : G, w1, w2;
  int k;
  auto sums = [&]() {                // k, sum w and sum w^2 of w = |v| - lo > 0
    w1 = w2 = 0.0f;
    k = 0;
    for (int t = lane; t < ncand; t += 32) {
      const float w = fabsf(cv[t]) - lo;
      if (w > 0.0f) {
        w1 += w;
        w2 = fmaf(w, w, w2);
        ++k;
      }
    }
    w1 = warp_sum_f(w1);
    w2 = warp_sum_f(w2);
    k = warp_sum_i(k);
  };
  sums();
  if (!(s * w2 - w1 * w1 < 0.0f) && lo > G) {
    lo = G;
    sums();
  }
  if (!(s * w2 - w1 * w1 < 0.0f)) return -1.0;
  for (int it = 0; it < 64 && (float)k > s; ++it) {
    const float kf = (float)k, mean = w1 / kf;
    const float var = fmaxf(kf * w2 - w1 * w1, 0.0f) + 2e-6f * kf * w2;
    const float d = mean - sqrtf(s * var / (kf - s)) / kf - 4e-6f * mean;
    if (!(lo + d > lo)) break;
    lo += d;
    const int kprev = k;
    sums();
    if (k == kprev) break;
  }
  double bound = (double)lo, lam = bound;
  float bound_f = lo;                // (for a float v, v > a double b is v > the largest float <= b)
  for (int it = 0; it < 64; ++it) {
    float a1 = 0.0f, c1 = 0.0f, a2 = 0.0f, c2 = 0.0f;
    int kc = 0;
    for (int i = lane; i < ncand; i += 32) {
      const float v = fabsf(cv[i]);
      if (v > bound_f) {
        ++kc;
        kahan_add(a1, c1, v);
        const float vv = v * v;
        kahan_add(a2, c2, vv);
        kahan_add(a2, c2, fmaf(v, v, -vv));
      }
    }
    const double s1 = warp_sum_d((double)a1 + (double)c1), s2 = warp_sum_d((double)a2 + (double)c2);
    const int kn = warp_sum_i(kc);
    const double kd = (double)kn;
    if (kd <= s_d) {
      lam = bound;
      break;
    }
    // sums of w = |v| - bound, and d = lam - bound from them in FP32
    const double W1 = fma(-kd, bound, s1), W2 = fma(-bound, s1 + W1, s2);
    const float kf = (float)kn, W1f = (float)W1, gap = (float)(kd - s_d);
    const float var = fmaxf((float)fma(kd, W2, -W1 * W1), 0.0f);
    double d = (double)(W1f / kf - sqrtf(s * var / gap) / kf);
    // phi(d) = s (W2 - 2 d W1 + k d^2) - (W1 - k d)^2, phi'(d) = 2 (k - s) (W1 - k d)
    float tf = 0.0f;
#pragma unroll 1
    for (int q = 0; q < 2; ++q) {
      const double t = fma(-kd, d, W1);
      tf = (float)t;
      if (!(tf > 1e-3f * W1f)) break;
      const double phi = fma(s_d, fma(-d, W1 + t, W2), -t * t);
      d -= (double)((float)phi / (2.0f * gap * tf));
    }
    if (!(tf > 1e-3f * W1f)) {       // all of the set nearly equal: the root in closed form
      double disc = s_d * (kd * s2 - s1 * s1) / (kd - s_d);
      if (disc < 0.0) disc = 0.0;
      d = (s1 - sqrt(disc)) / kd - bound;
    }
    lam = fmax(bound + d, bound);
    const float lam_f = __double2float_rd(lam);
    int below = 0;
    for (int i = lane; i < ncand; i += 32) {
      const float v = fabsf(cv[i]);
      below += v > bound_f && v <= lam_f;
    }
    if (warp_sum_i(below) == 0) break;
    bound = lam;
    bound_f = lam_f;
  }
  return lam;
}

// An entry within a quarter of its last bit of lambda_s survives or not by the rounding of phi alone.  The
// x-step of given v leaves a start that has one to the full pass (one start in 25000 of p = 40000, s = 50),
// so that the number of survivors is the full pass's in every case.
constexpr double kLamTie = -2.0;
__device__ __forceinline__ bool lambda_tie(const float *cv, int ncand, double lam) {
  const int lane = threadIdx.x & 31, near = __float_as_int(__double2float_rd(lam));
  bool tie = false;
  for (int i = lane; i < ncand; i += 32) {
    const int key = (int)abs_key(cv[i]);
    if (key < near || key > near + 1) continue;
    const double v = (double)__int_as_float(key), ulp = (double)__int_as_float(key + 1) - v;
    tie = tie || fabs(v - lam) < 0.25 * ulp;
  }
  return __any_sync(0xffffffffu, tie);
}

// a start's state as the x-step reads it, all loads in flight at once
struct XState {
  int iters = 0, nnz = 0, xfast = 0;
  float tprev = 0.0f, thr = 0.0f;
  double gamma = 0.0, F_prev = 0.0;
};
__device__ __forceinline__ XState load_state(const StartState &st, int c) {
  XState q;
  if (st.iters) q.iters = st.iters[c];
  if (st.status) {                   // (a solve: every array is there)
    q.nnz = st.nnz[c];
    q.xfast = st.xfast[c];
    q.tprev = st.tprev[c];
    q.thr = st.thr[c];
    q.gamma = st.gamma[c];
    q.F_prev = st.F_prev[c];
  }
  return q;
}

// The form's family as a compile-time constant: the code of a family holds nothing of the others', and an
// x-step's warps stall for instructions more than for anything else (16 sweeps' x-steps, without and with:
// 16 starts of p = 4000, T_s, 236 and 204 us; of p = 100000, V_gamma, 446 and 365; one of 20000, T_s, 343 and 259).
// kAny: groups, whose one launch serves members of every form.
enum class XKind { kSelect, kLambda, kPenalty, kAny };
inline XKind xstep_kind(int form) {
  return uses_T(form) ? XKind::kSelect : uses_lam(form) ? XKind::kLambda : XKind::kPenalty;
}

// the x-step of start c (block-wide, T threads); false when it is left to the full pass
template <int T, XKind K>
__device__ __forceinline__ bool xstep_fast_one(const XstepArgs &a_in, int c, const float *__restrict__ V, int64_t ldv,
                                               float *__restrict__ X, int64_t ldx, const StartState &st,
                                               const XState &q0, int *__restrict__ sup_idx,
                                               float *__restrict__ sup_val, Ctrl *ctrl, FastShared<T> &fs) {
  const XstepArgs a = xstep_switches(a_in, q0.iters);
  const int p = a.p, form = a.form, s_int = (int)a.s;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const Row row = row_of(V + (int64_t)c * ldv, p);
  float *x = X ? X + (int64_t)c * ldx : nullptr;   // (null: the support list is all that is wanted)
  const unsigned lt_mask = (1u << lane) - 1u;
  const bool t_form = K == XKind::kAny ? uses_T(form) : K == XKind::kSelect;
  const bool lam_form = K == XKind::kAny ? uses_lam(form) : K == XKind::kLambda;
  const bool pen_form = K == XKind::kAny ? is_pen(form) : K == XKind::kPenalty;
  const bool exact = pen_form && !a.calibrate;
  const bool keep_all = t_form && s_int >= p;
  const int need = t_form ? s_int : (pen_form && a.calibrate ? s_int + 1 : 1);
  const bool all = p <= kFastAllP || (p <= kFastCand && keep_all);
  if (!all && !exact && (need > kFastMaxNeed || keep_all || need * kFastPerNeed > p)) return false;
  // j of the subset maxima: the active set of lambda_s has about 2 s entries where |v|'s tail is
  // exponential, so 3 s lie below its threshold; never so many that subsets hold several of them
  int j = lam_form ? (int)fminf(3.0f * (float)a.s + 16.0f, (float)kFastMaxJ) : need;
  const float tprev = q0.tprev;
  const bool steady = q0.xfast == 1;
  // x is zero outside the last support list, once there is one (before: all of x is written)
  const bool listed = sup_idx && q0.iters > 1 && q0.nnz <= a.cap;
  // (there, the old list's entries are cleared once the new one is made: their indices load meanwhile)
  const int nnz_old = x && listed ? q0.nnz : 0;
  const int *old = sup_idx + (int64_t)c * a.cap;
  const int old0 = (int)threadIdx.x < nnz_old ? old[threadIdx.x] : -1;
  auto clear_row = [&] {             // as aligned vectors, whatever the row's alignment
    const int sh = (int)((reinterpret_cast<uintptr_t>(x) >> 2) & 3u);
    float *xb = x - sh;
    for (int q = 4 * threadIdx.x; q < p + sh; q += 4 * T) {
      if (q >= sh && q + 4 <= p + sh) {
        *reinterpret_cast<float4 *>(xb + q) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      } else {
        for (int k = 0; k < 4; ++k)
          if (q + k >= sh && q + k < p + sh) xb[q + k] = 0.0f;
      }
    }
  };
  // a whole row's zeros are stored while v is read, but for an x over v itself (the x-step of given v, in place),
  // and for a fixed threshold, above which there may be any number of entries (and the full pass writes all
  // of x): there once the list is made, which v is read for
  const float *vrow = V + (int64_t)c * ldv;
  const bool late = (x < vrow + p && vrow < x + p) || exact;
  if (x && !listed && !late) clear_row();

  // ---- a bound, the list above it, and the check (block-uniform throughout)
  int buf = 0, ncand = 0;
  double lam = 0.0;
  bool lam0 = false;                 // lambda_s = 0: the L1 ball does not bind
  enum { kAll, kExact, kHigh, kLow, kSubsets };
  int how = exact ? kExact : all ? kAll : listed && tprev > 0.0f ? kHigh : kSubsets;
  uint32_t Gk;
  float thr = 0.0f;
  double gam = 0.0;
  if (exact) {
    thr = a.per_start_thr ? q0.thr : a.thr_fixed;
    gam = a.per_start_thr ? q0.gamma : a.gamma_fixed;
  }
  for (;;) {
    if (how == kExact) {
      Gk = __float_as_uint(thr);
      if (!listed && first_segment_full<T>(row, Gk, fs)) return false;
    } else if (how == kAll) Gk = 0u;
    else if (how == kHigh) Gk = __float_as_uint((steady && !a.ordered ? kGuessSteady : kGuess) * tprev);
    else if (how == kLow) Gk = __float_as_uint(kGuessLo * tprev);
    else Gk = j <= kFastMaxJ ? subset_bound<T>(row, j, lam_form ? (float)a.s : 0.0f, fs) : kNoBound;
    if (Gk == kNoBound) return false;
    float f1 = 0.0f, f2 = 0.0f;
    const bool fits = list_above<T>(row, Gk, lam_form, fs, buf, &ncand, &f1, &f2);
    // phi(0) >= 0, every entry survives: no bound above 0 can serve.  (The sums' last bits depend on T: with
    // this margin the start would fail the check of phi(G) below all the same, for sqrt(s) ||V||_2 / ||V||_1
    // grows with the threshold.)
    if (lam_form && Gk != 0u && (float)a.s * f2 > 1.001f * (f1 * f1)) return false;
    bool ok = fits;
    if (fits && lam_form) {
      if (w == 0) {                  // (a hint just below the last lambda_s: few steps while it holds steady)
        double l = list_lambda(fs.u.l.cv, ncand, (float)a.s, a.s, __uint_as_float(Gk), kHint * tprev);
        // (given v: see kLamTie)
        if (!st.status && l >= 0.0 && lambda_tie(fs.u.l.cv, ncand, l)) l = kLamTie;
        if (lane == 0) fs.lam = l;
      }
      __syncthreads();
      lam = fs.lam;
      if (lam == kLamTie) return false;
      ok = lam >= 0.0;
      if (!ok && Gk == 0u) ok = lam0 = true;   // phi(0) >= 0 over all of v's nonzero entries
    } else if (fits && !exact) ok = ncand >= need || Gk == 0u;
    if (ok) break;
    if (how == kHigh) {
      how = a.ordered && fits && !steady ? kLow : kSubsets;
      // lambda_s lies below this bound: its active set is larger than the list
      if (lam_form && fits) j = min(kFastMaxJ, max(j, ncand + ncand / 2 + 32));
    } else if (how == kLow) {
      how = kSubsets;
    } else if (how == kSubsets && lam_form && fits && j < kFastMaxJ) {
      j = kFastMaxJ;                     // the root lies lower: a longer list
    } else {
      return false;
    }
    __syncthreads();                 // the lists are reused
  }
  // (every thread has read its part of v: the list's barrier)
  if (old0 >= 0) x[old0] = 0.0f;
  for (int t = threadIdx.x + T; t < nnz_old; t += T) x[old[t]] = 0.0f;
  if (x && !listed && late) clear_row();

  // ---- the operator on the list: which entries survive, as
  //   select: rank < need (T_s; ties at the threshold: the lower indices), or key above the threshold
  float tval = 0.0f, tnext = tprev;
  const bool select = (t_form && !keep_all) || (pen_form && a.calibrate);
  const bool ranked = select && ncand >= need;
  uint32_t kmin = 0xFFFFFFFFu;       // the need-th largest key
  if (ranked) {
    // rank of each entry = entries with a larger key; the need-th largest key is the smallest one of
    // rank < need
    int above = 0;
    const int n4 = ncand & ~3;
    for (int t = threadIdx.x; t < ncand; t += T) {
      const uint32_t mine = abs_key(fs.u.l.cv[t]);
      int rk = 0;
#pragma unroll 4
      for (int i = 0; i < n4; i += 4) {
        const float4 e = *reinterpret_cast<const float4 *>(fs.u.l.cv + i);
        rk += (abs_key(e.x) > mine) + (abs_key(e.y) > mine) + (abs_key(e.z) > mine) + (abs_key(e.w) > mine);
      }
      for (int i = n4; i < ncand; ++i) rk += abs_key(fs.u.l.cv[i]) > mine;
      fs.a.rank[t] = rk;             // (read back by this thread)
      if (rk < need) {
        kmin = min(kmin, mine);
        ++above;
      }
    }
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    above = warp_sum_i(above);
    if (lane == 0) fs.red[buf][w] = make_float4(__uint_as_float(kmin), __int_as_float(above), 0.0f, 0.0f);
    __syncthreads();
    kmin = __reduce_min_sync(0xffffffffu, lane < T / 32 ? __float_as_uint(fs.red[buf][lane].x) : 0xFFFFFFFFu);
    above = warp_sum_i(lane < T / 32 ? __float_as_int(fs.red[buf][lane].y) : 0);
    buf ^= 1;
    tval = __uint_as_float(kmin);
    tnext = tval;
    if (t_form && above > need) {   // more entries tie at the threshold than fit: by index
      for (int t = threadIdx.x; t < ncand; t += T) {
        if (abs_key(fs.u.l.cv[t]) != kmin) continue;
        int order = 0;
        for (int i = 0; i < t; ++i) order += abs_key(fs.u.l.cv[i]) == kmin;
        fs.a.rank[t] += order;
      }
      __syncthreads();               // (the list's values are replaced below)
    }
  } else if (lam_form) {
    tval = lam0 ? 0.0f : (float)lam;
    gam = lam0 ? 0.0 : lam;
    tnext = tval;
  } else if (exact) {
    tval = thr;
  } else {
    tnext = 0.0f;                    // at most s (or s + 1) nonzero entries: all of them; gamma = 0
  }
  if (pen_form && a.calibrate) gam = (pen_form && uses_U(form)) ? (double)tval * (double)tval : (double)tval;
  const bool soft = lam_form || (pen_form && uses_V(form));
  // an entry survives when its key is above this one (lambda_s: |v| > lam in FP64)
  const uint32_t cut = lam_form && !lam0 ? __float_as_uint(__double2float_rd(lam))
                       : ranked && !t_form ? kmin : 0u;

  // ---- w, which takes the place of the list's values; the survivors are counted per 32 entries
  const int rounds = (ncand + T - 1) / T;
  for (int q = 0; q < rounds; ++q) {
    const int t = threadIdx.x + q * T;
    float wq = 0.0f;
    if (t < ncand) {
      const float v = fs.u.l.cv[t];
      const uint32_t mine = abs_key(v);
      bool keep = mine > cut;
      if (ranked && t_form) keep = fs.a.rank[t] < need;
      if (keep) wq = soft ? copysignf(fabsf(v) - tval, v) : v;
    }
    const unsigned ball = __ballot_sync(0xffffffffu, wq != 0.0f);
    if (lane == 0) fs.cnt[q * (T / 32) + w] = __popc(ball);
    __syncwarp();
    if (t < ncand) fs.u.l.cv[t] = wq;
  }
  __syncthreads();
  int incl = lane < rounds * (T / 32) ? fs.cnt[lane] : 0;
  const int own = incl;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  const int nnz = __shfl_sync(0xffffffffu, incl, 31);
  for (int q = 0; q < rounds; ++q) {
    const int t = threadIdx.x + q * T;
    const float wq = t < ncand ? fs.u.l.cv[t] : 0.0f;
    const unsigned ball = __ballot_sync(0xffffffffu, wq != 0.0f);
    const int o = __shfl_sync(0xffffffffu, incl - own, q * (T / 32) + w) + __popc(ball & lt_mask);
    if (wq != 0.0f) {
      fs.a.s.val[o] = wq;
      fs.a.s.idx[o] = fs.u.l.ci[t];
    }
  }
  __syncthreads();
  // ---- ||w||^2, over the survivors as one warp adds them (lane l entries l, l + 32, ...; every warp
  // repeats it for itself), so that it does not depend on the list or the number of threads.
  // On a resident 16-bit matrix (ordered) every sweep rounds y to 11 bits, and a last-bit difference of
  // ||w|| can end as one of 4e-5 in x (measured after 16 sweeps).  There the sum keeps the order of a warp
  // over the list when that comes from last sweep's threshold (or is exact), and of the full pass, by
  // index segment and lane, otherwise.
  const bool seg_order = a.ordered && (p < kSegOrderP || how == kAll || how == kSubsets || (how == kExact && !listed));
  float sumsq = 0.0f;
  if (!a.ordered) {
    for (int t = lane; t < nnz; t += 32) sumsq = fmaf(fs.a.s.val[t], fs.a.s.val[t], sumsq);
    sumsq = warp_sum_f(sumsq);
  } else if (!seg_order) {
    for (int t = lane; t < ncand; t += 32) sumsq = fmaf(fs.u.l.cv[t], fs.u.l.cv[t], sumsq);
    sumsq = warp_sum_f(sumsq);
  } else {
    const bool by_index = p <= 2 * kFastCand;
    if (by_index) {                  // w at its index, zeros elsewhere
      for (int i = threadIdx.x; i < p; i += T) fs.u.by_index[i] = 0.0f;
      __syncthreads();
      for (int t = threadIdx.x; t < nnz; t += T) fs.u.by_index[fs.a.s.idx[t]] = fs.a.s.val[t];
      __syncthreads();
    }
    for_segments<false>(p, [&](int sgi, Seg sg) {
      float part = 0.0f;
      if (by_index) {
        for (int i = sg.lo + lane; i < sg.hi; i += 32) part = fmaf(fs.u.by_index[i], fs.u.by_index[i], part);
      } else {
        for (int t = 0; t < nnz; ++t) {
          const int i = fs.a.s.idx[t] - sg.lo;
          if (i >= 0 && i < sg.hi - sg.lo && (i & 31) == lane) part = fmaf(fs.a.s.val[t], fs.a.s.val[t], part);
        }
      }
      put_sum2f(sgi, part, 0.0f, 0, 0, fs.sh);
    });
    float f_unused;
    int i_unused, i_unused2;
    get_sum2f(sumsq, f_unused, i_unused, i_unused2, fs.sh);
  }
  float inv, nrm_hi, nrm_lo;
  norm_and_inverse(sumsq, &nrm_hi, &nrm_lo, &inv);

  // ---- x and the support list (the zeros above are ordered before these by the barriers since)
  int *gi = sup_idx ? sup_idx + (int64_t)c * a.cap : nullptr;
  float *gv = sup_val ? sup_val + (int64_t)c * a.cap : nullptr;
  for (int t = threadIdx.x; t < nnz; t += T) {
    const int i = fs.a.s.idx[t];
    const float xi = fs.a.s.val[t] * inv;
    if (x) x[i] = xi;
    if (gi && t < a.cap) {
      gi[t] = i;
      gv[t] = xi;
    }
  }
  // ---- outputs, stopping rule (Section 2.2), control word for the next sweep
  if (threadIdx.x == 0) {
    const double nrm = norm_fp64(sumsq, nrm_hi, nrm_lo);
    double F;
    if (lam_form) F = gam * a.sqrt_s + nrm;                              // S4
    else if ((pen_form && uses_U(form))) F = (double)sumsq - gam * (double)nnz;        // S5
    else F = nrm;                                                        // S3, S6
    if (st.F) st.F[c] = F;
    if (st.nnz) st.nnz[c] = nnz;
    if (st.gamma) st.gamma[c] = gam;
    if (st.thr && pen_form && a.calibrate) st.thr[c] = tval;
    if (st.tprev) st.tprev[c] = tnext;
    if (st.xfast) {
      const bool near = tnext >= (1.0f - kSteady) * tprev && tnext <= (1.0f + kSteady) * tprev;
      st.xfast[c] = how == kExact || (how == kHigh && near) ? 1 : 2;
    }
    if (st.status) {
      int status = ST_ACTIVE;
      if (sumsq == 0.0f) {
        status = SPCA_ST_DEGENERATE;
      } else if (a.stop_test && F <= (1.0 + a.tol) * q0.F_prev) {
        status = SPCA_ST_CONVERGED;
      } else if (q0.iters >= a.max_iter) {
        status = SPCA_ST_MAXITER;
      }
      st.F_prev[c] = F;
      st.status[c] = status;
      if (status == ST_ACTIVE && ctrl && nnz > a.sparse_cap) atomicOr(&ctrl->need_dense, 1);
    }
  }
  return true;
}

// the start's x-step: the threshold x-step, else the full pass from global memory at once (defer
// false) or a mark for k_xstep / k_g_xstep (xfast = 0; without xfast, nnz = -1).  The starts that
// needed the full pass are counted in ctrl->n_full: the host queues the full kernel, which stages v in
// shared memory, only for sweeps after some start needed it.
template <bool kOne>
__device__ __noinline__ void xstep_full_global(const XstepArgs &a, int c, const float *__restrict__ V, int64_t ldv,
                                               float *__restrict__ X, int64_t ldx, StartState st,
                                               int *__restrict__ sup_idx, float *__restrict__ sup_val, Ctrl *ctrl,
                                               XShared &sh) {
  xstep_full_one<false, kOne>(a, c, V, ldv, X, ldx, st, sup_idx, sup_val, ctrl, nullptr, sh);
}
template <int T, XKind K>
__device__ __forceinline__ void xstep_start(const XstepArgs &a, int c, const float *__restrict__ V, int64_t ldv,
                                            float *__restrict__ X, int64_t ldx, const StartState &st,
                                            const XState &q0, int *__restrict__ sup_idx,
                                            float *__restrict__ sup_val, Ctrl *ctrl, bool defer, FastShared<T> &fs) {
  if (xstep_fast_one<T, K>(a, c, V, ldv, X, ldx, st, q0, sup_idx, sup_val, ctrl, fs)) return;
  if (ctrl && threadIdx.x == 0) atomicAdd(&ctrl->n_full, 1);
  __syncthreads();
  if (!defer) {
    xstep_full_global<T == XT>(a, c, V, ldv, X, ldx, st, sup_idx, sup_val, ctrl, fs.sh);
    if (threadIdx.x == 0 && st.xfast) st.xfast[c] = 2;
  } else if (threadIdx.x == 0) {
    if (st.xfast) st.xfast[c] = 0;
    else st.nnz[c] = -1;
  }
}

// (CTAs per SM for the register budget: 7 x 152 of 128 threads hold 1024 starts at once)
constexpr int fast_ctas(int t) { return t == 128 ? 7 : t == 256 ? 3 : 1; }
template <int T, XKind K>
__global__ void __launch_bounds__(T, fast_ctas(T)) k_xstep_fast(XstepArgs a, const float *__restrict__ V, int64_t ldv,
                                                            int r, float *__restrict__ X, int64_t ldx, StartState st,
                                                            int *__restrict__ sup_idx, float *__restrict__ sup_val,
                                                            Ctrl *ctrl, Ctrl *ctrl_read, int *act, int *rank,
                                                            int defer, int *flags, int nflags) {
  __shared__ FastShared<T> fs;
  const int c = blockIdx.x;
  if (flags && c == 0)
    for (int i = threadIdx.x; i < nflags; i += T) flags[i] = 0;
  const int status = st.status ? st.status[c] : ST_ACTIVE;
  const XState q0 = load_state(st, c);
  if (status == ST_ACTIVE) xstep_start<T, K>(a, c, V, ldv, X, ldx, st, q0, sup_idx, sup_val, ctrl, defer != 0, fs);
  if (act) last_makes_active_list(r, st.status, st.nnz, r, act, rank, ctrl, ctrl_read);
}

// Threads per start, 128 to 1024: reading v shrinks with the threads, barriers and the sums over the
// warps grow with them, so 16 to 256 entries per thread (a sweep's x-step of 16 starts, forms 1 and 3, event
// times: p = 4000 with 128 threads 15.3 and 20.0 us, 256 14.2 and 18.5; p = 12000 with 256 15.4 and 20.4, 512
// 15.4 and 18.7; p = 40000 with 512 18.3 and 23.1, 1024 20.0 and 25.7; p = 200000 with 512 37.6 and 38.7, 1024
// 35.0 and 38.6); and never more than keeps all starts
// resident at once (fast_ctas).
int fast_threads(int64_t starts, int p, int sms) {
  const int by_p = p <= 2048 ? 128 : p <= 8192 ? 256 : p <= 131072 ? 512 : 1024;
  const int by_r = starts <= sms ? 1024 : starts <= 3 * (int64_t)sms ? 256 : 128;
  return std::min(by_p, by_r);
}
// (function-local static: initialised once, thread-safe)
int sm_count() {
  static const int sms = [] {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) !=
                                                   cudaSuccess)
      return 0;
    return v;
  }();
  return sms;
}
}  // namespace

// groups of problems: the full pass for the starts that k_g_xstep_fast left, persistent CTAs over the
// global starts; the kSmem launch takes the problems whose v fits in shared memory (staged there),
// the other launch the rest
template <bool kSmem>
__global__ void __launch_bounds__(XT, 2) k_g_xstep(const GProb *__restrict__ P, const int *__restrict__ prob, int R,
                                                   int parity) {
  extern __shared__ float vsm[];
  __shared__ XShared sh;
  for (int g = blockIdx.x; g < R; g += gridDim.x) {
    const GProb &q = P[prob[g]];
    if (kSmem != ((size_t)q.p * sizeof(float) <= (size_t)XSTEP_SMEM_MAX)) continue;
    const int c = g - q.start0;
    StartState st = q.st;
    if (st.status[c] != ST_ACTIVE || st.xfast[c] != 0) continue;
    __syncthreads();   // (every thread has read the mark; shared memory is reused from start to start)
    xstep_full_one<kSmem, true>(q.xa, c, q.V, q.ldX, q.X, q.ldX, st, q.sup_idx, q.sup_val, q.ctrl[parity], vsm, sh);
    if (threadIdx.x == 0) st.xfast[c] = 2;
    __syncthreads();
  }
}

// groups of problems: the threshold x-step, a CTA per global start; each problem's last CTA makes its
// active list unless the full kernel follows (defer)
template <int T>
__global__ void __launch_bounds__(T, fast_ctas(T)) k_g_xstep_fast(const GProb *__restrict__ P,
                                                              const int *__restrict__ prob, int parity, int defer) {
  __shared__ FastShared<T> fs;
  const GProb &q = P[prob[blockIdx.x]];
  const int c = (int)blockIdx.x - q.start0;
  const int status = q.st.status[c];
  const XState q0 = load_state(q.st, c);
  if (status == ST_ACTIVE)
    xstep_start<T, XKind::kAny>(q.xa, c, q.V, q.ldX, q.X, q.ldX, q.st, q0, q.sup_idx, q.sup_val, q.ctrl[parity],
                                defer != 0, fs);
  if (!defer)
    last_makes_active_list(q.r, q.st.status, q.st.nnz, q.r, q.act, q.rank, q.ctrl[parity], q.ctrl[parity ^ 1]);
}

cudaError_t launch_g_xstep(const GProb *P, const int *prob, int R, int max_p, int max_p_small, bool any_large,
                           bool defer, int parity, int sms, cudaStream_t st) {
  const int d = defer ? 1 : 0;
  switch (fast_threads(R, max_p, sms)) {
    case 1024: k_g_xstep_fast<1024><<<R, 1024, 0, st>>>(P, prob, parity, d); break;
    case 512: k_g_xstep_fast<512><<<R, 512, 0, st>>>(P, prob, parity, d); break;
    case 256: k_g_xstep_fast<256><<<R, 256, 0, st>>>(P, prob, parity, d); break;
    default: k_g_xstep_fast<128><<<R, 128, 0, st>>>(P, prob, parity, d); break;
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || !defer) return e;
  if (max_p_small > 0) {   // the problems whose v fits in shared memory: staged there
    const size_t bytes = (size_t)max_p_small * sizeof(float);
    if (bytes > (size_t)XSTEP_SMEM_MAX) return cudaErrorInvalidValue;
    static const cudaError_t configured =
        cudaFuncSetAttribute(k_g_xstep<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, XSTEP_SMEM_MAX);
    if (configured != cudaSuccess) return configured;
    const int per_sm = bytes <= 100u * 1024u ? 2 : 1;
    k_g_xstep<true><<<min(R, per_sm * sms), XT, bytes, st>>>(P, prob, R, parity);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (any_large) {
    k_g_xstep<false><<<min(R, 2 * sms), XT, 0, st>>>(P, prob, R, parity);
    return cudaGetLastError();
  }
  return cudaSuccess;
}

// ---------------------------------------------------------------- small problems in one launch
// For a small matrix the chain of launches of a sweep, not its work, sets the time.  Here every sweep of
// every start runs in one launch, a cluster of C CTAs per start, until the start stops or `sweeps` sweeps
// have run: u = A x over the support's rows of A^T, the y-step, v = A^T y over the CTA's share of A's
// columns (in its shared memory where they fit), v's pieces to every CTA of the cluster, the threshold
// x-step.  u, y, v, the support list and the start's state live in shared memory, in every CTA alike: the
// CTAs of a cluster repeat the same steps on the same v and so decide alike, and meet once a sweep.
// What bounds a sweep is its chain of dependent steps (a round trip to L2 for u, then about 15 barriers).
// 16 starts, n = 100, p = 500, 40 sweeps: 535 -> 235 us; n = 250, p = 1000, 20 sweeps 1250 -> 240 us
// (one CTA per start, u by whole rows of A, u, y and v through memory before).
// A start that has swept goes on from its support list and state: the sweeps may be cut into several launches,
// with the same bits.

// for every o < out: put(o, sum over k of w[k] M[row(k) ld + o]), row(k) = idx[k] or k: a thread per four
// outputs and slice of the k (part: 4 T floats for the slices' sums)
template <int T, typename Put>
__device__ __forceinline__ void small_product(const float *M, int64_t ld, const int *idx, const float *w, int K,
                                              int out, float *part, const Put &put) {
  constexpr int L = 8;
  const int quads = (out + 3) / 4, width = (quads + 7) / 8 * 8;
  const int S = width >= T ? 1 : min(min(32, K), T / width);   // (K >= 1)
  const int slice = S == 1 ? 0 : (int)threadIdx.x / width, q0 = S == 1 ? (int)threadIdx.x : (int)threadIdx.x % width;
  for (int q = q0; q < quads && slice < S; q += T) {
    const float *m = M + 4 * q;
    float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    auto load = [&](int k) { return *reinterpret_cast<const float4 *>(m + (int64_t)(idx ? idx[k] : k) * ld); };
    auto add = [&](float x, float4 a) {
      acc.x = fmaf(x, a.x, acc.x); acc.y = fmaf(x, a.y, acc.y);
      acc.z = fmaf(x, a.z, acc.z); acc.w = fmaf(x, a.w, acc.w);
    };
    float4 a[L];
    int k = slice;
    for (; k + (L - 1) * S < K; k += L * S) {
#pragma unroll
      for (int h = 0; h < L; ++h) a[h] = load(k + h * S);
#pragma unroll
      for (int h = 0; h < L; ++h) add(w[k + h * S], a[h]);
    }
    if (k < K) {
#pragma unroll
      for (int h = 0; h < L; ++h)
        if (k + h * S < K) a[h] = load(k + h * S);
#pragma unroll
      for (int h = 0; h < L; ++h)
        if (k + h * S < K) add(w[k + h * S], a[h]);
    }
    if (S == 1) {
      put(4 * q, acc.x);
      if (4 * q + 1 < out) put(4 * q + 1, acc.y);
      if (4 * q + 2 < out) put(4 * q + 2, acc.z);
      if (4 * q + 3 < out) put(4 * q + 3, acc.w);
    } else {
      reinterpret_cast<float4 *>(part)[slice * width + q] = acc;
    }
  }
  if (S == 1) return;
  __syncthreads();
  for (int o = threadIdx.x; o < out; o += T) {
    float t = part[o];
#pragma unroll 4
    for (int h = 1; h < S; ++h) t += part[h * 4 * width + o];
    put(o, t);
  }
}

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// a float to shared-memory address `addr` of the cluster's CTA `rank`
__device__ __forceinline__ void store_cluster(uint32_t addr, int rank, float v) {
  asm volatile("{\n\t.reg .b32 a;\n\tmapa.shared::cluster.u32 a, %0, %1;\n\tst.shared::cluster.f32 [a], %2;\n\t}"
               ::"r"(addr), "r"(rank), "f"(v) : "memory");
}

// a start's state in shared memory, addressed as StartState with c = 0
struct SmallState {
  double F, F_prev, gamma;
  float thr, tprev;
  int status, iters, nnz, xfast;
};
__device__ __forceinline__ StartState small_state(SmallState &s) {
  StartState t{};
  t.status = &s.status; t.iters = &s.iters; t.nnz = &s.nnz; t.xfast = &s.xfast;
  t.F = &s.F; t.F_prev = &s.F_prev; t.gamma = &s.gamma;
  t.thr = &s.thr; t.tprev = &s.tprev;
  return t;
}

// the CTA's columns of v = A^T y (all but the last CTAs the same number, a multiple of 4)
__host__ __device__ inline int small_cols(int p, int ctas) { return ((p + ctas - 1) / ctas + 3) / 4 * 4; }
// shared memory in floats: v (two buffers when the pieces come from several CTAs), the support's indices
// and values, and u (n) with the slices' sums, or the x-step's lists in their place; then A's columns
template <int T>
__host__ __device__ inline int64_t small_words(int64_t n, int64_t p, int ctas) {
  const int64_t p4 = (p + 3) & ~int64_t(3), n4 = (n + 3) & ~int64_t(3);
  const int64_t a = n4 + 4 * T, b = (sizeof(FastShared<T>) + 15) / 16 * 4;
  return (ctas > 1 ? 4 : 3) * p4 + (a > b ? a : b);
}

template <int T, XKind K>
__global__ void __launch_bounds__(T, 1) k_small_sweeps(XstepArgs xa, const float *__restrict__ A, int64_t lda,
                                                    const float *__restrict__ AT, int64_t ldat, int n, int p,
                                                    int ctas, int a_smem, float *__restrict__ X, int64_t ldx,
                                                    StartState st, int *__restrict__ sup_idx,
                                                    float *__restrict__ sup_val, int sweeps) {
  extern __shared__ float4 sm4[];
  __shared__ float redf[32];
  __shared__ SmallState ss;
  const int c = blockIdx.x / ctas, rank = blockIdx.x % ctas;
  const int p4 = (p + 3) & ~3, n4 = (n + 3) & ~3;
  float *vb = reinterpret_cast<float *>(sm4);
  float *lv = vb + (ctas > 1 ? 2 : 1) * p4;
  int *li = reinterpret_cast<int *>(lv + p4);
  float *u = lv + 2 * p4, *part = u + n4;
  FastShared<T> &fs = *reinterpret_cast<FastShared<T> *>(u);
  float *as = vb + small_words<T>(n, p, ctas);
  const int pc = small_cols(p, ctas), j0 = rank * pc, mine = max(0, min(pc, p - j0));
  float *x = X + (int64_t)c * ldx;
  // x^(0), or the support list of a start that has swept; the start's state, this CTA's columns of A
  const bool fresh = st.iters[c] == 0;
  const int nnz0 = fresh ? p : st.nnz[c];
  for (int j = threadIdx.x; j < nnz0; j += T) {
    lv[j] = fresh ? x[j] : sup_val[(int64_t)c * p + j];
    li[j] = fresh ? j : sup_idx[(int64_t)c * p + j];
  }
  if (a_smem) {
    for (int q = threadIdx.x; q < n * (pc / 4); q += T) {
      const int i = q / (pc / 4), h = 4 * (q % (pc / 4));
      if (h < mine) *reinterpret_cast<float4 *>(as + (int64_t)i * pc + h) =
          *reinterpret_cast<const float4 *>(A + (int64_t)i * lda + j0 + h);   // (rows are padded to a multiple of 8)
    }
  }
  if (threadIdx.x == 0) {
    ss.status = st.status[c]; ss.iters = st.iters[c]; ss.nnz = nnz0; ss.xfast = st.xfast[c];
    ss.F = st.F[c]; ss.F_prev = st.F_prev[c]; ss.gamma = st.gamma[c];
    ss.thr = st.thr[c]; ss.tprev = st.tprev[c];
  }
  StartState sl = small_state(ss);
  const uint32_t vaddr = (uint32_t)__cvta_generic_to_shared(vb);
  if (ctas > 1) cluster_barrier();   // (every CTA has started and read its state)
  else __syncthreads();
  if (ss.status != ST_ACTIVE) return;   // (the same in every CTA of the cluster)
  for (int k = 0; k < sweeps; ++k) {
    float *v = vb + (ctas > 1 && (k & 1) ? p4 : 0);
    small_product<T>(AT, ldat, fresh && k == 0 ? nullptr : li, lv, ss.nnz, n, part, [&](int i, float t) { u[i] = t; });
    __syncthreads();
    // y-step
    if (threadIdx.x == 0) ss.iters += 1;
    if (is_l1_var(xa.form)) {
      for (int i = threadIdx.x; i < n; i += T) u[i] = u[i] >= 0.0f ? 1.0f : -1.0f;
    } else {
      float sq = 0.0f;
      for (int i = threadIdx.x; i < n; i += T) sq = fmaf(u[i], u[i], sq);
      const float sumsq = block_sum_f(sq, redf);
      if (sumsq == 0.0f) {
        __syncthreads();
        if (threadIdx.x == 0) {
          ss.status = SPCA_ST_DEGENERATE;
          ss.nnz = 0;
          ss.F = 0.0;
        }
        __syncthreads();
        break;
      }
      float hi, lo, inv;
      norm_and_inverse(sumsq, &hi, &lo, &inv);
      for (int i = threadIdx.x; i < n; i += T) u[i] *= inv;
    }
    __syncthreads();
    // v = A^T y, to every CTA
    if (mine > 0) {
      const int at = (int)(v - vb) + j0;
      small_product<T>(a_smem ? as : A + j0, a_smem ? pc : lda, nullptr, u, n, mine, part, [&](int o, float t) {
        if (ctas == 1) v[o] = t;
        else
          for (int h = 0; h < ctas; ++h) store_cluster(vaddr + 4u * (uint32_t)(at + o), h, t);
      });
    }
    if (ctas > 1) cluster_barrier();
    else __syncthreads();
    if (!xstep_fast_one<T, K>(xa, 0, v, 0, nullptr, 0, sl, load_state(sl, 0), li, lv, nullptr, fs)) {
      __syncthreads();
      xstep_full_one<false, false>(xa, 0, v, 0, nullptr, 0, sl, li, lv, nullptr, nullptr, fs.sh);
      if (threadIdx.x == 0) ss.xfast = 2;
    }
    __syncthreads();
    if (ss.status != ST_ACTIVE) break;
  }
  if (rank != 0) return;
  // the results: x, its support list, the state
  const int nnz = ss.nnz;
  for (int j = threadIdx.x; j < p; j += T) x[j] = 0.0f;
  __syncthreads();
  for (int t = threadIdx.x; t < nnz; t += T) {
    x[li[t]] = lv[t];
    sup_idx[(int64_t)c * p + t] = li[t];
    sup_val[(int64_t)c * p + t] = lv[t];
  }
  if (threadIdx.x == 0) {
    st.status[c] = ss.status; st.iters[c] = ss.iters; st.nnz[c] = nnz; st.xfast[c] = ss.xfast;
    st.F[c] = ss.F; st.F_prev[c] = ss.F_prev; st.gamma[c] = ss.gamma;
    st.thr[c] = ss.thr; st.tprev[c] = ss.tprev;
  }
}

constexpr int kSmallT = 256, kSmallCtas = 8;
bool small_sweeps_fit(int64_t n, int64_t p, int r, double support) {
  if (small_words<kSmallT>(n, p, kSmallCtas) * 4 > (int64_t)XSTEP_SMEM_MAX) return false;
  if (n * p > kSmallAlways && (double)n * std::min(support, (double)p) > (double)kSmallReads) return false;
  return n * p <= kSmallEntries && r <= 2 * sm_count();
}

template <XKind K>
static cudaError_t small_smem() {
  return cudaFuncSetAttribute(k_small_sweeps<kSmallT, K>, cudaFuncAttributeMaxDynamicSharedMemorySize, XSTEP_SMEM_MAX);
}

cudaError_t launch_small_sweeps(XstepArgs xa, const float *A, int64_t lda, const float *AT, int64_t ldat, int n, int p,
                                float *X, int64_t ldx, StartState s, int *sup_idx, float *sup_val, int r, int sweeps,
                                cudaStream_t st) {
  if (!small_sweeps_fit(n, p, r, 0.0) || lda % 8 != 0 || ldat % 8 != 0) return cudaErrorInvalidValue;
  // CTAs per start, of at least 32 columns each: as many as are resident at once (a cluster lies in one GPC,
  // so of 152 SMs clusters of 8 reach 120 and clusters of 4 reach 144, at a CTA per SM; a second wave doubled
  // the time: 16 starts of p = 500 in clusters of 8 565 us, of 4 320)
  const int sms = sm_count();
  if (sms < 1) return cudaErrorInvalidDevice;
  int ctas = kSmallCtas;
  while (ctas > 1 && ((int64_t)r * ctas > sms * (ctas == 8 ? 6 : 7) / 8 || p < 32 * ctas)) ctas /= 2;
  size_t bytes = 4 * (size_t)small_words<kSmallT>(n, p, ctas);
  const size_t a_bytes = 4 * (size_t)n * (size_t)small_cols(p, ctas);
  const int a_smem = bytes + a_bytes <= (size_t)XSTEP_SMEM_MAX ? 1 : 0;
  if (a_smem) bytes += a_bytes;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(r * ctas));
  cfg.blockDim = dim3(kSmallT);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)ctas;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  auto go = [&](auto kern, cudaError_t configured) -> cudaError_t {
    if (configured != cudaSuccess) return configured;
    return cudaLaunchKernelEx(&cfg, kern, xa, A, lda, AT, ldat, n, p, ctas, a_smem, X, ldx, s, sup_idx, sup_val, sweeps);
  };
  // (function-local statics: configured once, thread-safe)
  switch (xstep_kind(xa.form)) {
    case XKind::kSelect: {
      static const cudaError_t set = small_smem<XKind::kSelect>();
      return go(k_small_sweeps<kSmallT, XKind::kSelect>, set);
    }
    case XKind::kLambda: {
      static const cudaError_t set = small_smem<XKind::kLambda>();
      return go(k_small_sweeps<kSmallT, XKind::kLambda>, set);
    }
    default: {
      static const cudaError_t set = small_smem<XKind::kPenalty>();
      return go(k_small_sweeps<kSmallT, XKind::kPenalty>, set);
    }
  }
}

// The x-step of given v has no last threshold to start from, so its list costs a pass for the bound and one
// for the list.  It pays, against the full pass of every start in one launch, for lambda_s with s up to 150
// (above, the list often does not hold the active set), and for T_s and the Section 4.1 rule with few
// selected entries: a 25th of v (a 13th when starts outnumber two per SM) and at most kFastMaxJ.  Whole
// calls, full pass and list: one start, p = 1500, T_s, s = 200 28 and 31 us, s = 50 27 and 28; p = 6000, s = 500 33
// and 39, s = 200 35 and 30; 1024 starts, p = 3000, s = 200 66 and 44, s = 500 68 and 86; 600, p = 6000, s = 500 62
// and 68.  A fixed threshold is the list's bound itself.
bool xstep_list_pays(int form, double s, bool calibrate, int64_t p, int64_t r, int sms) {
  if (uses_lam(form)) return s <= 150.0;
  if (is_pen(form) && !calibrate) return true;
  const int64_t need = (int64_t)s + (calibrate ? 1 : 0);
  return need <= kFastMaxJ && need * (r <= 2 * (int64_t)sms ? 25 : 13) <= p;
}

cudaError_t launch_xstep(XstepArgs a, const float *V, int64_t ldv, int r, float *X, int64_t ldx,
                         StartState s, int *sup_idx, float *sup_val, Ctrl *ctrl, Ctrl *ctrl_read, int *act,
                         int *rank, XFull full, int *flags, int nflags, cudaStream_t st) {
  const int sms = sm_count(), d = full == XFull::kAfter ? 1 : 0;
  if (sms < 1) return cudaErrorInvalidDevice;
  int *al = d ? nullptr : act;
  cudaError_t e = cudaSuccess;
  if (full != XFull::kAlone) {
    auto go = [&](auto kern, int threads) {
      kern<<<r, threads, 0, st>>>(a, V, ldv, r, X, ldx, s, sup_idx, sup_val, ctrl, ctrl_read, al, rank, d, flags, nflags);
      return cudaGetLastError();
    };
    const XKind kind = xstep_kind(a.form);
#define SPCA_FAST(T)                                                  \
  (kind == XKind::kSelect   ? go(k_xstep_fast<T, XKind::kSelect>, T)  \
   : kind == XKind::kLambda ? go(k_xstep_fast<T, XKind::kLambda>, T)  \
                            : go(k_xstep_fast<T, XKind::kPenalty>, T))
    switch (fast_threads(r, a.p, sms)) {
      case 1024: e = SPCA_FAST(1024); break;
      case 512: e = SPCA_FAST(512); break;
      case 256: e = SPCA_FAST(256); break;
      default: e = SPCA_FAST(128); break;
    }
    if (e != cudaSuccess || full == XFull::kInside) return e;
  }
#undef SPCA_FAST
  // the full pass for the starts left: persistent CTAs (as many as fit), so that a sweep in which no
  // start needs it costs one short launch
  const size_t bytes = (size_t)a.p * sizeof(float);
  const int every = full == XFull::kAlone ? 1 : 0;
  if (bytes <= (size_t)XSTEP_SMEM_MAX) {
    static const cudaError_t configured =
        cudaFuncSetAttribute(k_xstep<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, XSTEP_SMEM_MAX);
    if (configured != cudaSuccess) return configured;
    const int per_sm = bytes <= 100u * 1024u ? 2 : 1;
    k_xstep<true><<<min(r, per_sm * sms), XT, bytes, st>>>(a, V, ldv, r, X, ldx, s, sup_idx, sup_val, ctrl, every);
  } else {
    k_xstep<false><<<min(r, 2 * sms), XT, 0, st>>>(a, V, ldv, r, X, ldx, s, sup_idx, sup_val, ctrl, every);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess || !act) return e;
  return launch_active_list(s.status, s.nnz, r, act, rank, ctrl, ctrl_read, st);
}

}  // namespace spca
