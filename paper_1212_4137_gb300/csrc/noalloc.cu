// noalloc.cu -- spca_objective_noalloc: the Table 1 objective and explained variance of given
// vectors x, for callers that must not allocate device memory.
//
// Who needs it: code that runs where cudaMalloc is off limits -- inside a captured CUDA graph
// being recorded by someone else's framework, under a memory pool or allocator that owns the
// whole device, or in a real-time loop where an allocation's implicit synchronisation and
// latency are not acceptable.  Such a caller already holds A, the x's and the result arrays in
// device memory; this entry point adds nothing to the device heap.
//
// The computation is the one spca_solve reports per start (u = A x with FP64 products and sums,
// then the objective of the formulation and ||Ax||_2^2 or ||Ax||_1), done by a variant of the
// finalisation kernels whose per-(start, row chunk) partial sums live in a file-scope
// __device__ array instead of handle memory.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <mutex>

#include "block_util.cuh"
#include "spca_internal.cuh"

namespace spca {
namespace {

constexpr int NT = 512;                 // threads per CTA
constexpr int NW = NT / 32;             // warps per CTA
constexpr int NROWS = 256;              // rows of A per CTA (a chunk)
constexpr int RPW = NROWS / NW;         // consecutive rows per warp (16)
constexpr int LPR = 8;                  // lanes per row: a warp works on 32 / LPR rows at once
constexpr int RPL = RPW / (32 / LPR);   // rows per lane (4)
constexpr int XPIECE = 8 * NT;          // entries of x scanned between two barriers
constexpr int XSTAGE = XPIECE + 512;    // nonzeros of x staged in shared memory before they are used

// the scratch: (r * ceil(n / 256)) pairs of doubles, at most SPCA_NOALLOC_MAX_PARTIALS pairs.
// Every GPU that loads the library holds these 4 MiB until the process exits.
__device__ __align__(256) double g_partials[2 * SPCA_NOALLOC_MAX_PARTIALS];

// Sum of acc[0 .. RPL) over the LPR = 8 lanes of a row group, as a reduce-scatter: each exchange
// halves the sums a lane still carries, so 4 rows cost 4 FP64 adds per lane instead of 12 (FP64 runs
// at 1/64 of the FP32 rate and bounds this kernel).  Lane l of the group ends with row l >> 1.
__device__ __forceinline__ double group_reduce(const double (&acc)[RPL], int lane) {
  static_assert(RPL == 4 && LPR == 8, "the exchange pattern");
  const bool h2 = lane & 4, h1 = lane & 2;
  double a0 = h2 ? acc[2] : acc[0], a1 = h2 ? acc[3] : acc[1];
  const double g0 = h2 ? acc[0] : acc[2], g1 = h2 ? acc[1] : acc[3];
  a0 += __shfl_xor_sync(0xffffffffu, g0, 4);
  a1 += __shfl_xor_sync(0xffffffffu, g1, 4);
  double v = h1 ? a1 : a0;
  v += __shfl_xor_sync(0xffffffffu, h1 ? a0 : a1, 2);
  return v + __shfl_xor_sync(0xffffffffu, v, 1);
}

// grid nchunks x r, the starts fastest: u_i = sum_j x_j A[i, j] over the nonzeros of x, products and sums in FP64,
// for the 256 rows of chunk b; this CTA's sums of |u_i| and u_i^2 go to
// partials[(c * nchunks + b) * 2].
// Bound by finding the nonzeros (each CTA scans the p entries of its x from L2) and by the FP64 pipe.
// The scan takes 4096 entries per barrier pair, a warp 256 consecutive ones with its 8 loads in
// flight (256 entries per barrier pair before).  Then 8 lanes share a row and a warp works on 4 rows
// at a time, 4 times: with few nonzeros most lanes have work, a lane has 4 rows' loads in flight,
// and the lane sums end in the reduce-scatter above.  The staged columns ascend, so 8 lanes read one
// 32-byte sector of a row when x is dense.
// All starts of a row chunk run side by side, so that a 32-byte sector of A that several starts need comes
// from memory once (A is larger than L2).
// 64 starts with 50 nonzeros each, n = 5000, p = 20000: 168 us (659 with a scan of 256 entries per barrier
// pair, 252 with the row chunks of a start side by side).
__global__ void __launch_bounds__(NT) k_obj_partial(const float *__restrict__ A, int64_t lda, int n, int p,
                                                    const float *__restrict__ X, int64_t ldx, int r, int nchunks,
                                                    double *__restrict__ partials) {
  __shared__ int sj[XSTAGE];
  __shared__ float sx[XSTAGE];
  __shared__ int wcnt[NW];
  __shared__ double red[32];
  const int c = blockIdx.x % r, chunk = blockIdx.x / r;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int sub = lane / LPR, l8 = lane % LPR;
  const int row0 = chunk * NROWS + w * RPW + sub;   // this lane's rows: row0 + k (32 / LPR)
  const float *x = X + (int64_t)c * ldx;
  const float *arow[RPL];
#pragma unroll
  for (int k = 0; k < RPL; ++k) arow[k] = A + (int64_t)min(row0 + k * (32 / LPR), n - 1) * lda;
  double acc[RPL] = {0.0, 0.0, 0.0, 0.0};
  const unsigned lt = (1u << lane) - 1u;
  int staged = 0;
  const unsigned up = (unsigned)p;   // (base may pass 2^31 in its last step)
  for (unsigned base = 0; base < up; base += XPIECE) {
    // this warp's 256 entries of the piece, in index order
    float xv[8];
    unsigned b[8];
    int cnt = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const unsigned j = base + w * 256 + k * 32 + lane;
      xv[k] = j < up ? x[j] : 0.0f;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      b[k] = __ballot_sync(0xffffffffu, xv[k] != 0.0f);
      cnt += __popc(b[k]);
    }
    if (lane == 0) wcnt[w] = cnt;
    __syncthreads();
    int pos = staged;
#pragma unroll
    for (int q = 0; q < NW; ++q) {
      const int t = wcnt[q];
      pos += q < w ? t : 0;
      staged += t;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (xv[k] != 0.0f) {
        const int q = pos + __popc(b[k] & lt);
        sj[q] = (int)(base + w * 256 + k * 32 + lane);
        sx[q] = xv[k];
      }
      pos += __popc(b[k]);
    }
    __syncthreads();
    // use the staged nonzeros when the next piece might not fit, and at the end
    if (staged > XSTAGE - XPIECE || base + XPIECE >= up) {
      for (int t = l8; t < staged; t += LPR) {
        const int j = sj[t];
        float a[RPL];
#pragma unroll
        for (int k = 0; k < RPL; ++k) a[k] = __ldg(arow[k] + j);
        const double xd = (double)sx[t];
#pragma unroll
        for (int k = 0; k < RPL; ++k) acc[k] = fma(xd, (double)a[k], acc[k]);
      }
      __syncthreads();
      staged = 0;
    }
  }
  // |u_i| and u_i^2 of the row this lane ends with (the odd lanes hold copies)
  const double u = group_reduce(acc, lane);
  const int i = row0 + (l8 >> 1) * (32 / LPR);
  const bool mine = (l8 & 1) == 0 && i < n;
  const double l1 = block_sum_d(mine ? fabs(u) : 0.0, red);
  const double l2 = block_sum_d(mine ? u * u : 0.0, red);
  if (threadIdx.x == 0) {
    double *o = partials + ((int64_t)c * nchunks + chunk) * 2;
    o[0] = l1;
    o[1] = l2;
  }
}

// a CTA per start: the partials, ||x||_0 and ||x||_1 (coalesced, 8 loads in flight per thread; one
// thread per start walked x alone before: 25 us, 2552 us before, at the size above), then the objective
__global__ void __launch_bounds__(NT) k_obj_reduce(int form, double gamma, const double *__restrict__ partials,
                                                   int nchunks, const float *__restrict__ X, int64_t ldx, int p,
                                                   double *__restrict__ f, double *__restrict__ ev) {
  __shared__ double red[32];
  __shared__ int red_i[32];
  const int c = blockIdx.x;
  double l1 = 0.0, l2sq = 0.0, x1 = 0.0;
  int nz = 0;
  for (int b = threadIdx.x; b < nchunks; b += NT) {
    l1 += partials[((int64_t)c * nchunks + b) * 2 + 0];
    l2sq += partials[((int64_t)c * nchunks + b) * 2 + 1];
  }
  const float *x = X + (int64_t)c * ldx;
  const unsigned up = (unsigned)p;
  for (unsigned base = threadIdx.x; base < up; base += 8 * NT) {
    float xv[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) xv[k] = base + k * NT < up ? x[base + k * NT] : 0.0f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (xv[k] != 0.0f) {   // (a zero adds nothing: the FP64 adds are the slow part)
        ++nz;
        x1 += fabs((double)xv[k]);
      }
    }
  }
  l1 = block_sum_d(l1, red);
  l2sq = block_sum_d(l2sq, red);
  x1 = block_sum_d(x1, red);
  const double x0 = (double)block_sum_i(nz, red_i);
  if (threadIdx.x != 0) return;
  const double l2 = sqrt(l2sq);
  double val;
  switch (form) {
    case 1: case 3: val = l2; break;
    case 2: case 4: val = l1; break;
    case 5: val = l2sq - gamma * x0; break;
    case 6: val = l1 * l1 - gamma * x0; break;
    case 7: val = l2 - gamma * x1; break;
    default: val = l1 - gamma * x1; break;
  }
  f[c] = val;
  ev[c] = is_l1_var(form) ? l1 : l2sq;
}

// set-up once per device (with that device current): the device address of the scratch
std::mutex g_mu;
double *g_addr[64] = {nullptr};

cudaError_t scratch_for_current_device(double **out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_addr[dev]) {
    void *ptr = nullptr;
    e = cudaGetSymbolAddress(&ptr, g_partials);
    if (e != cudaSuccess) return e;
    g_addr[dev] = static_cast<double *>(ptr);
  }
  *out = g_addr[dev];
  return cudaSuccess;
}

}  // namespace
}  // namespace spca

using namespace spca;

extern "C" int spca_objective_noalloc(int form, double gamma, const float *A, int64_t n, int64_t p, int64_t lda,
                                      const float *X, int64_t ldx, int r, double *f, double *ev,
                                      void *cuda_stream) {
  if (form < 1 || form > 8 || !A || !X || !f || !ev) return SPCA_E_INVALID;
  if (n < 1 || p < 1 || r < 1 || lda < p || ldx < p || n > INT32_MAX || p > INT32_MAX) return SPCA_E_INVALID;
  if (!std::isfinite(gamma) || gamma < 0.0) return SPCA_E_INVALID;
  if (r > spca::kMaxStarts) return SPCA_E_UNSUPPORTED;   // the limit of every call on starts
  const int64_t nchunks = (n + NROWS - 1) / NROWS;
  if ((int64_t)r * nchunks > (int64_t)SPCA_NOALLOC_MAX_PARTIALS) return SPCA_E_INVALID;   // beyond the scratch
  double *partials = nullptr;
  if (scratch_for_current_device(&partials) != cudaSuccess) return SPCA_E_CUDA;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  // every partial the reduction reads is written by this call's first kernel (no zeroing needed)
  k_obj_partial<<<(unsigned)(nchunks * r), NT, 0, st>>>(A, lda, (int)n, (int)p, X, ldx, r, (int)nchunks, partials);
  if (cudaGetLastError() != cudaSuccess) return SPCA_E_CUDA;
  k_obj_reduce<<<r, NT, 0, st>>>(form, gamma, partials, (int)nchunks, X, ldx, (int)p, f, ev);
  if (cudaGetLastError() != cudaSuccess) return SPCA_E_CUDA;
  return SPCA_OK;
}
