// Allocation-free scenario operator: u = A^T diag(w) A v + (rho/2) v for one
// scenario whose CSR matrix the caller already holds in device memory.
//
// For callers that must not allocate device memory: code running where
// cudaMalloc is not available or not allowed (inside a memory pool that owns all
// device memory, in a real-time loop that may not block on the allocator, or in
// a process whose allocations are accounted by someone else).  Such a caller
// passes its own device inputs and output; the only working memory is a
// file-scope device array of fixed size, the per-CTA partial sums.
//
// The scratch array lives in every device that loads the library, for the life
// of the process.  In host code its name is only a host-side stand-in, so the
// device address is looked up once per device (cudaGetSymbolAddress) and passed
// to the kernels.  Every call overwrites each scratch slot it later reads, so
// nothing has to be cleared between calls; calls that overlap on the GPU share
// the array and race.
#include <algorithm>
#include <mutex>
#include <string>

#include "plan.h"

namespace rpt {
namespace {

constexpr int kNaThreads = 1024;
constexpr int kNaMaxCtas = 128;            // CTAs whose partial sums fit the scratch at kNaMaxCols
constexpr int kNaMaxCols = 8192;           // largest n (columns padded to a multiple of 32)

// Per-CTA partial accumulators, one row of n_pad floats per CTA (4 MiB in all).
static __device__ __align__(256) float g_noalloc_scratch[kNaMaxCtas * kNaMaxCols];

// CTAs that get a partial row: what the scratch holds at this width (at least
// kNaMaxCtas).
constexpr int na_ctas(int n_pad) { return kNaMaxCtas * kNaMaxCols / n_pad; }

constexpr int kNaLanes = 8;                // lanes per row
constexpr int kNaKeep = 16;                // entries per lane kept between the dot and the scatter
constexpr int kNaApart = 1024;             // the 4 rows of a warp step lie up to this far apart
constexpr int kNaBatch = 8;                // steps whose row offsets are loaded together
constexpr int kNaTail = 8;                 // entries of a longer row, per lane, loaded together (few rows)
constexpr int kNaFew = 8192;               // up to so many rows each is a step of its own, for a whole warp

// One row by L lanes (this lane is sl), or nothing when lo == hi: the row's
// entries, the first KEEP L of them kept in registers between the dot and the
// scatter, and TAIL of the further ones loaded at a time.  Entries outside [0, n) are
// ignored.  Every lane of the warp calls it.
template <int L, int KEEP, int TAIL>
__device__ __forceinline__ void na_row(unsigned lo, unsigned hi, unsigned sl, float wi, int n, const int32_t* __restrict__ col,
                                       const float* __restrict__ val, const float* sv, float* acc) {
  float a[KEEP];
  int c[KEEP];
#pragma unroll
  for (int k = 0; k < KEEP; ++k) {
    const unsigned e = lo + sl + L * k;
    a[k] = e < hi ? __ldg(val + e) : 0.f;
    c[k] = e < hi ? __ldg(col + e) : -1;
  }
  float t = 0.f;
#pragma unroll
  for (int k = 0; k < KEEP; ++k)
    if ((unsigned)c[k] < (unsigned)n) t = fmaf(a[k], sv[c[k]], t);
  if constexpr (TAIL == 1) {
    for (unsigned e = lo + sl + L * KEEP; e < hi; e += L) {
      const int q = __ldg(col + e);
      if ((unsigned)q < (unsigned)n) t = fmaf(__ldg(val + e), sv[q], t);
    }
  } else {
    for (unsigned e = lo + sl + L * KEEP; e < hi; e += L * TAIL) {
      float b[TAIL];
      int q[TAIL];
#pragma unroll
      for (int k = 0; k < TAIL; ++k) {
        b[k] = e + L * k < hi ? __ldg(val + e + L * k) : 0.f;
        q[k] = e + L * k < hi ? __ldg(col + e + L * k) : -1;
      }
#pragma unroll
      for (int k = 0; k < TAIL; ++k)
        if ((unsigned)q[k] < (unsigned)n) t = fmaf(b[k], sv[q[k]], t);
    }
  }
#pragma unroll
  for (int o = L / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  const float coef = wi * t;
#pragma unroll
  for (int k = 0; k < KEEP; ++k)
    if ((unsigned)c[k] < (unsigned)n) atomicAdd(&acc[c[k]], coef * a[k]);
  if constexpr (TAIL == 1) {
    for (unsigned e = lo + sl + L * KEEP; e < hi; e += L) {
      const int q = __ldg(col + e);
      if ((unsigned)q < (unsigned)n) atomicAdd(&acc[q], coef * __ldg(val + e));
    }
  } else {
    for (unsigned e = lo + sl + L * KEEP; e < hi; e += L * TAIL) {
      float b[TAIL];
      int q[TAIL];
#pragma unroll
      for (int k = 0; k < TAIL; ++k) {
        b[k] = e + L * k < hi ? __ldg(val + e + L * k) : 0.f;
        q[k] = e + L * k < hi ? __ldg(col + e + L * k) : -1;
      }
#pragma unroll
      for (int k = 0; k < TAIL; ++k)
        if ((unsigned)q[k] < (unsigned)n) atomicAdd(&acc[q[k]], coef * b[k]);
    }
  }
}

// Bound: the entries once from HBM (8 bytes each).  A CSR matrix handed over per
// call cannot be cut by cost in advance, and most of its rows may be empty (the
// voxels outside the beams), so rows are dealt evenly: a step takes 4 rows, 8
// lanes each, and steps go round-robin over all warps of the grid, so that every
// warp gets its part of every region.  The 4 rows of a step lie `apart` rows apart:
// neighbouring rows share most of their spots, and lanes that meet on one spot
// retry their atomics.  Row offsets are loaded for kNaBatch steps at once; empty
// steps cost a ballot.  Rows longer than the 8 lanes keep in registers are left
// for the whole warp.  A matrix of few rows (kNaFew) has a step and a warp for each row,
// on as many CTAs as there are rows: with 4 rows a step, half as many warps and one of
// them after the other, 100 rows of 8000 entries took 607 us, 1000 of 2000 158 (103 and 56
// cut by entries), against
// 33 and 20.5 us; the line lies where short rows would gain by sharing a warp (10,000 rows of 10
// entries 10.6 us shared, 14.7 apart; 6000 of 200 16.7 and 14.5).  (kNaTail loads at a time
// in the other form cost its short rows 4 %.)  One scenario of the realistic plan (10.0 M entries, 299k
// rows of which 214k are empty, 5000 spots): 52 us for both kernels against
// 2568 us when CTAs were cut by entries, which left the empty rows at both ends
// of the volume to two CTAs, and each warp waited for one row at a time; 190k
// entries and 200 spots: 12 us against 49 us.
template <int ROWS>
__global__ void __launch_bounds__(kNaThreads)
k_noalloc_pass(int m, int n, int n_pad, int apart, const int32_t* __restrict__ rp, const int32_t* __restrict__ col,
               const float* __restrict__ val, const float* __restrict__ w, const float* __restrict__ v,
               float* __restrict__ scratch) {
  extern __shared__ float sm[];
  float* sv = sm;
  float* acc = sm + n_pad;
  const int tid = threadIdx.x, lane = tid & 31, nw = kNaThreads / 32;
  for (int j = tid; j < n_pad; j += kNaThreads) {
    sv[j] = j < n ? v[j] : 0.f;
    acc[j] = 0.f;
  }
  __syncthreads();
  const int sl = lane & (kNaLanes - 1);
  const int tile = ROWS * apart;
  const int steps = ((m - 1) / tile + 1) * apart;   // m / ROWS rounded up to whole tiles
  const int stride = gridDim.x * nw;
  // consecutive steps go to different CTAs
  const int first = (tid >> 5) * gridDim.x + blockIdx.x;
  for (int s0 = first; s0 < steps; s0 += stride * kNaBatch) {
    // lane l: row l & 3 (of ROWS) of the batch's step l >> 2
    const int s = s0 + stride * (lane >> 2);
    const long long i = (long long)(s / apart) * tile + s % apart + (lane & 3) * apart;
    int blo = 0, bhi = 0;
    float bw = 0.f;
    if (s < steps && i < m && (lane & 3) < ROWS) {
      blo = __ldg(rp + i);
      bhi = __ldg(rp + i + 1);
      if (bhi > blo) bw = __ldg(w + i);
      else bhi = blo;        // (offsets that decrease: an empty row; the entries are counted unsigned)
    }
    const unsigned any = __ballot_sync(0xffffffffu, bhi > blo);
    for (int b = 0; b < kNaBatch; ++b) {
      if (((any >> (4 * b)) & 15u) == 0) continue;
      const int from = 4 * b + lane / kNaLanes;
      const int lo = __shfl_sync(0xffffffffu, blo, from), hi = __shfl_sync(0xffffffffu, bhi, from);
      const float wi = __shfl_sync(0xffffffffu, bw, from);
      const bool wide = ROWS == 1 ? hi > lo : hi - lo > kNaLanes * kNaKeep;
      if (ROWS > 1) na_row<kNaLanes, kNaKeep, 1>(lo, wide ? lo : hi, sl, wi, n, col, val, sv, acc);
      unsigned left = __ballot_sync(0xffffffffu, wide && sl == 0);
      while (left) {
        const int src = __ffs(left) - 1;
        left &= left - 1;
        na_row<32, kNaKeep, ROWS == 1 ? kNaTail : 1>(__shfl_sync(0xffffffffu, lo, src), __shfl_sync(0xffffffffu, hi, src), lane,
                            __shfl_sync(0xffffffffu, wi, src), n, col, val, sv, acc);
      }
    }
  }
  __syncthreads();
  float4* out = reinterpret_cast<float4*>(scratch + (size_t)blockIdx.x * n_pad);
  for (int j = tid; j < n_pad / 4; j += kNaThreads) out[j] = reinterpret_cast<const float4*>(acc)[j];
}

// u[j] = sum over CTAs c of scratch[c][j] + (rho/2) v[j].  Latency-bound, so the
// CTAs' partials of 32 columns go to kNaSums thread rows (independent loads), each
// a compensated sum in a fixed order, and the rows' sums are added with
// compensation in row order; the partial of each CTA comes from shared-memory
// float atomics whose order varies between runs, so results are not bitwise
// reproducible (they stay within the float32 bound of the sums).
constexpr int kNaSums = 16;
__global__ void __launch_bounds__(32 * kNaSums)
k_noalloc_reduce(int n, int n_pad, int ctas, const float* __restrict__ scratch, const float* __restrict__ v,
                 float half_rho, float* __restrict__ u) {
  __shared__ float ss[kNaSums][32], sc[kNaSums][32];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  const int j = blockIdx.x * 32 + x;        // n_pad is a multiple of 32
  float s = 0.f, c = 0.f;
#pragma unroll 4
  for (int k = y; k < ctas; k += kNaSums) {
    float t, e;
    two_sum(s, __ldcg(scratch + (size_t)k * n_pad + j), t, e);
    s = t;
    c += e;
  }
  ss[y][x] = s;
  sc[y][x] = c;
  __syncthreads();
  if (y != 0 || j >= n) return;
#pragma unroll
  for (int k = 1; k < kNaSums; ++k) {
    float t, e;
    two_sum(s, ss[k][x], t, e);
    s = t;
    c += e + sc[k][x];
  }
  u[j] = (s + c) + half_rho * v[j];
}

std::mutex g_na_mutex;
// device address of the scratch array, per device ordinal; looked up by the first
// call on a device and kept for the process (not valid across a cudaDeviceReset
// of that device, which the rpt.h entry rules out)
float* g_na_ptr[64] = {nullptr};

}  // namespace
}  // namespace rpt

using namespace rpt;

extern "C" int rpt_normal_apply_noalloc(int32_t m, int32_t n, const int32_t* row_ptr_dev,
                                        const int32_t* col_idx_dev, const float* val_dev,
                                        const float* row_w_dev, const float* v_dev, double rho, float* u_dev,
                                        void* stream) {
  if (m < 1 || n < 1 || !row_ptr_dev || !col_idx_dev || !val_dev || !row_w_dev || !v_dev || !u_dev ||
      !(rho >= 0.0)) {
    set_error("rpt_normal_apply_noalloc: bad argument (sizes, null pointer or rho)");
    return RPT_EINVAL;
  }
  if (n > kNaMaxCols) {
    set_error("rpt_normal_apply_noalloc: n = " + std::to_string(n) + " exceeds the scratch limit of " +
              std::to_string(kNaMaxCols) + " spots");
    return RPT_EUNSUPPORTED;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (dev < 0 || dev >= 64) {
    set_error("rpt_normal_apply_noalloc: device ordinal out of range");
    return RPT_EUNSUPPORTED;
  }
  float* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (!g_na_ptr[dev]) {
      // one-time set-up on this device (must happen outside stream capture)
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress");
      g_na_ptr[dev] = static_cast<float*>(p);
    }
    scratch = g_na_ptr[dev];
  }
  const int n_pad = (n + 31) / 32 * 32;
  const size_t smem = (size_t)n_pad * 2 * sizeof(float);
  const bool few = m <= kNaFew;
  auto* pass = few ? k_noalloc_pass<1> : k_noalloc_pass<4>;
  if ((e = cudaFuncSetAttribute(pass, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)))
    return cuda_fail(e, "kernel attribute");
  int ctas = 0;
  if ((e = cudaDeviceGetAttribute(&ctas, cudaDevAttrMultiProcessorCount, dev)))
    return cuda_fail(e, "device attribute");
  // one CTA per SM, as many as have a partial row and rows, or steps for half of their warps
  ctas = std::min(ctas, na_ctas(n_pad));
  const int apart = few ? 1 : std::min(kNaApart, m / 4 + 1);
  ctas = std::min(ctas, few ? m : (m - 1) / (2 * (kNaThreads / 32)) + 1);
  cudaStream_t st = (cudaStream_t)stream;
  pass<<<ctas, kNaThreads, smem, st>>>(m, n, n_pad, apart, row_ptr_dev, col_idx_dev, val_dev, row_w_dev, v_dev, scratch);
  if ((e = cudaGetLastError())) return cuda_fail(e, "launch");
  k_noalloc_reduce<<<n_pad / 32, 32 * kNaSums, 0, st>>>(n, n_pad, ctas, scratch, v_dev, (float)(0.5 * rho), u_dev);
  if ((e = cudaGetLastError())) return cuda_fail(e, "launch");
  return RPT_OK;
}
