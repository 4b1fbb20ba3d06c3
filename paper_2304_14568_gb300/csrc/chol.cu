// Cached-factor x-update (App. A; the subproblem solver of the paper): for a
// fixed rho,
//     B_s = A~_s^T A~_s + (rho/2) I
// is formed once per (plan, rho), factored (Cholesky, B_s = L L^T) and inverted
// (B_s^{-1} = L^{-T} L^{-1}); every ADMM iteration then takes
//     x_s = B_s^{-1} c_s,   c_s = A~_s^T p~ + (rho/2) z - y_s / 2
// as one dense matrix-vector product per scenario, without a pass over the
// sparse matrices.  The paper factors in double precision on the CPU; here the
// factor, its inverse and the products are FP32 on the device (the solver state
// stays FP64), which bounds the relative error of an x-update by about
// cond(B_s) * n * eps32.
//
// Forming B_s uses the sparsity: rows are taken kRB at a time in voxel order
// (neighbouring voxels share most of their spots), their union of columns U is
// built in shared memory with the dense rows x |U| block of A~, and every nonzero
// pair sum over the block goes to the lower triangle of B_s with one global
// atomic.  The factorisation is blocked (64) and right-looking, the inverse of the
// factor is built by doubling from the diagonal blocks' inverses: a small kernel
// per diagonal block, everything else products on the FP32-accurate tensor-core
// GEMM of gemm_tf32.cuh (error-compensated TF32), batched over scenarios.  Rows of
// B_s, L^{-1} and B_s^{-1} are padded to 16 bytes (chol_ld).
// These products hold fewer bits than substitution in FP32 does: an operand's two
// halves hold about 22 bits of its 24 and the product of the low halves is dropped,
// and a diagonal block's inverse enters where a division did.  The error of an
// x-update is no larger for it: on nearly dependent spots (48 to 700, cond 1e3 to 2e6)
// 2.6e-5 to 1.7e-2 relative against 3.3e-5 to 2.1e-2 with substitution, 1.2 to 2.5
// times that of LAPACK's FP32 factor and inverse; on 200 to 1300 spots of the
// synthetic plans 1.1e-5 to 3.0e-5, the same.
#include <cmath>
#include <vector>

#include "gemm_tf32.cuh"
#include "plan.h"
#include "rowcommon.cuh"

namespace rpt {
namespace {

constexpr int kRB = 16;       // rows per outer-product block
constexpr int kUMax = 1024;   // columns a group of rows may touch (fewer on very wide plans)
constexpr int kDCap = 512 * kRB;   // floats of a group's dense block (kept to kBundleRows * kUMax at least)
constexpr int kBtbThreads = 256;
constexpr int kNB = 64;       // Cholesky / inverse block size
constexpr int kPB = 4;        // blocks per panel: the trailing matrix is updated once per panel (rank 256)
constexpr size_t kCholKeep = (size_t)128 << 20;   // bytes of L^{-1} that a plan keeps between factorisations
constexpr unsigned kFull = 0xffffffffu;

// Lower triangle of B_s (rows of ld floats, zero on entry) += sum over kept rows k
// in [blk * kRB, +kRB) of c_s w_k a_k a_k^T (A~ = diag(sqrt(c_s w)) A).  Blocks that
// run at the same time are of different scenarios and, within one, an eighth of its
// rows apart: neighbouring rows would add to the same elements (nblk: blocks of a
// scenario, grid N * 8 * ceil(nblk / 8)).
// BUN = false: CSR rows, rec_of[s][k] = position of kept row k in the row list.
// BUN = true: row bundles, rec_of[s][q] = position of the q-th bundle in creation
// (kept-row) order; the block takes kRB / 4 consecutive bundles.
// Bound: instruction issue (83 % of the cycles), about half of it the products of the
// dense block and the rest the address and the atomic of each pair.  Neighbouring rows
// share their columns, so a block of 16 rows has 0.86 of the pairs (and atomics) of two
// blocks of 8, but its dense rows are emptier: 64 rows have half the pairs and twice
// the products of 16.  A warp forms 8 x 64 pairs at a time from registers (16 products
// per 4 shared loads) and takes a unit's entries with its own lanes.  A block whose
// columns do not fit its dense block of 512 columns x 16 rows goes in halves.  13
// scenarios of 1250 spots in one launch: 1.57 ms (8 rows 1.53, 24 rows of 384 threads
// 1.58, 64 rows 3.8); 4.1 ms in 13 launches with one pair per lane and a unit's entries
// taken by all threads, unit after unit.  A unit of more than kUMax columns is added
// pair by pair: 600 units of four rows 2.65 ms at 1000 columns, 7.9 at 1100 (10.7 and
// 12.3 with those launches).
template <typename VT, typename IT, bool BUN>
__global__ void __launch_bounds__(kBtbThreads)
k_btb(DevPlan P, const int* __restrict__ rec_of, float* __restrict__ Ball, int ld, int umax, int cap, int nblk) {
  constexpr int RPU = BUN ? kBundleRows : 1;    // rows per unit (bundle or row)
  constexpr int UPB = kRB / RPU;                // units per block
  constexpr int NW = kBtbThreads / 32;
  const int s = blockIdx.x % P.N, order = blockIdx.x / P.N;
  const int blk = (order & 7) * ((nblk + 7) / 8) + (order >> 3);
  if ((order >> 3) >= (nblk + 7) / 8 || blk >= nblk) return;
  float* __restrict__ B = Ball + (size_t)s * P.n * ld;
  extern __shared__ __align__(16) unsigned char smem[];
  int* map = reinterpret_cast<int*>(smem);            // [n_pad]: flag, then position in U (-1: absent)
  int* U = map + P.n_pad;                             // [umax] sorted union of columns
  float* D = reinterpret_cast<float*>(U + umax);     // [rows][nz] dense block of A~, cap floats
  __shared__ int rlo[UPB], rhi[UPB];
  __shared__ float rw[kRB];
  __shared__ int wsum[NW];
  __shared__ int running;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int4* rec = P.rowrec + P.rec_base[s];
  const long long base = P.nnz_base[s];
  const VT* val = vals<VT>(P) + base * RPU;
  const IT* col = cols<IT>(P) + base;
  const float* cs = P.colscale ? P.colscale + (size_t)s * P.n_pad : nullptr;
  const int nunits = BUN ? (P.rec_base[s + 1] - P.rec_base[s]) / 4 - 1 : P.m_act;
  if ((long long)blk * UPB >= nunits) return;
  if (tid < UPB) {
    const int k = blk * UPB + tid;
    const int q = k < nunits ? rec_of[(size_t)s * P.m_act + k] : -1;
    rlo[tid] = q >= 0 ? rec[q * RPU].x : 0;
    rhi[tid] = q >= 0 ? rec[(q + 1) * RPU].x : 0;
  }
  if (tid < kRB) {
    const int u = tid / RPU, r = tid % RPU;
    const int k = blk * UPB + u;
    const int q = k < nunits ? rec_of[(size_t)s * P.m_act + k] : -1;
    const float wc = q < 0 ? 0.f
                     : BUN ? __int_as_float(reinterpret_cast<const int*>(&rec[4 * q + 1])[r])
                           : __int_as_float(rec[q].y);
    rw[tid] = sqrtf(wc);
  }
  auto entry = [&](int e, float (&a)[RPU]) {     // the unit's values at stored entry e
    if constexpr (BUN) {
      quad_v<true, VT>(val + 4 * (size_t)e, a);
    } else {
      a[0] = to_f<VT>(val[e]);
    }
  };
  int step = UPB;                                // units taken together: as many as fit
  for (int ua = 0; ua < UPB;) {
    const int ub = min(ua + step, UPB), rows = (ub - ua) * RPU;
    if (tid == 0) running = 0;
    for (int j = tid; j < P.n_pad; j += kBtbThreads) map[j] = 0;
    __syncthreads();
    for (int u = ua + w; u < ub; u += NW)
      for (int e = rlo[u] + lane; e < rhi[u]; e += 32) {
        float a[RPU];
        entry(e, a);
        bool nz = false;
        for (int r = 0; r < RPU; ++r) nz |= a[r] != 0.f;
        if (nz) map[(int)col[e]] = 1;
      }
    __syncthreads();
    // ordered compaction of the flags: map[c] = position in U, U[position] = c
    for (int c0 = 0; c0 < P.n_pad; c0 += kBtbThreads) {
      const int c = c0 + tid;
      const int f = c < P.n_pad ? map[c] : 0;
      const unsigned bal = __ballot_sync(kFull, f != 0);
      if (lane == 0) wsum[w] = __popc(bal);
      __syncthreads();
      int off = running, all = 0;
      for (int i = 0; i < NW; ++i) {
        if (i < w) off += wsum[i];
        all += wsum[i];
      }
      if (c < P.n_pad) {
        const int pos = off + __popc(bal & ((1u << lane) - 1u));
        map[c] = f ? pos : -1;
        if (f && pos < umax) U[pos] = c;
      }
      __syncthreads();
      if (tid == 0) running += all;
      __syncthreads();
    }
    const int nu = running, nz = (nu + 63) & ~63;
    const bool fits = nu <= umax && rows * nz <= cap;
    if (!fits && ub - ua > 1) {                  // too many columns: half the rows at a time
      step = (ub - ua) / 2;
      __syncthreads();
      continue;
    }
    if (!fits) {
      // rare: rows too spread out for one dense block; add each unit's pairs directly
      for (int u = ua; u < ub; ++u) {
        const int lo = rlo[u], len = rhi[u] - rlo[u];
        const long long pairs = (long long)len * len;
        for (long long p = tid; p < pairs; p += kBtbThreads) {
          const int e1 = lo + (int)(p / len), e2 = lo + (int)(p % len);
          const int c1 = (int)col[e1], c2 = (int)col[e2];
          if (c1 < c2) continue;
          float a1[RPU], a2[RPU];
          entry(e1, a1);
          entry(e2, a2);
          float v = 0.f;
          for (int r = 0; r < RPU; ++r) v += rw[u * RPU + r] * rw[u * RPU + r] * a1[r] * a2[r];
          if (cs) v *= cs[c1] * cs[c2];
          if (v != 0.f) atomicAdd(&B[(size_t)c1 * ld + c2], v);
        }
      }
      __syncthreads();
      ua = ub;
      continue;
    }
    for (int r = w; r < rows; r += NW)
      for (int c = lane; c < nz; c += 32) D[r * nz + c] = 0.f;
    __syncthreads();
    for (int u = ua + w; u < ub; u += NW)
      for (int e = rlo[u] + lane; e < rhi[u]; e += 32) {
        const int c = (int)col[e];
        float a[RPU];
        entry(e, a);
        for (int r = 0; r < RPU; ++r)
          if (a[r] != 0.f)
            D[((u - ua) * RPU + r) * nz + map[c]] = rw[u * RPU + r] * (cs ? a[r] * cs[c] : a[r]);
      }
    __syncthreads();
    // pairs a >= b of U (row U[a] >= column U[b]: the lower triangle) in tasks of 8
    // rows a and 64 columns b: the g-th eight of the row groups has g + 1 tasks a
    // group, 4 g (g + 1) before it
    const int na = (nu + 7) / 8;
    const int gl = (na - 1) / 8;
    const int tasks = 4 * gl * (gl + 1) + (na - 8 * gl) * (gl + 1);
    for (int t = tasks - 1 - w; t >= 0; t -= NW) {
      int g = (int)((sqrtf(1.f + (float)t) - 1.f) * 0.5f);
      while (4 * (g + 1) * (g + 2) <= t) ++g;
      while (4 * g * (g + 1) > t) --g;
      const int left = t - 4 * g * (g + 1);
      const int a0 = 8 * (8 * g + left / (g + 1)), b0 = 64 * (left % (g + 1));
      float acc[8][2];
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = 0.f;
#pragma unroll 4
      for (int r = 0; r < rows; ++r) {
        const float4 x = *reinterpret_cast<const float4*>(&D[r * nz + a0]);
        const float4 y = *reinterpret_cast<const float4*>(&D[r * nz + a0 + 4]);
        const float b1 = D[r * nz + b0 + lane], b2 = D[r * nz + b0 + 32 + lane];
        const float da[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          acc[i][0] = fmaf(da[i], b1, acc[i][0]);
          acc[i][1] = fmaf(da[i], b2, acc[i][1]);
        }
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int a = a0 + i;
        if (a >= nu) break;
        float* row = B + (size_t)U[a] * ld;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int b = b0 + 32 * h + lane;
          if (b <= a && acc[i][h] != 0.f) atomicAdd(&row[U[b]], acc[i][h]);
        }
      }
    }
    __syncthreads();
    ua = ub;
  }
}

// B_s[j][j] += half_rho for every scenario (grid.y = scenario).
__global__ void k_add_diag(float* B, int n, int ld, float half_rho) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < n) B[(size_t)blockIdx.y * n * ld + (size_t)j * ld + j] += half_rho;
}

// Upper triangle of every B_s^{-1} from its lower triangle (32 x 32 tiles through
// shared memory; grid (tiles, tiles, scenario), only tiles with row block >= column block).
__global__ void k_mirror_lower(float* X, int n, int ld) {
  __shared__ float t[32][33];
  const int bi = blockIdx.y, bj = blockIdx.x;
  if (bj > bi) return;
  float* Xs = X + (size_t)blockIdx.z * n * ld;
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int i = bi * 32 + r, j = bj * 32 + threadIdx.x;
    if (i < n && j < n) t[r][threadIdx.x] = Xs[(size_t)i * ld + j];
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int i = bj * 32 + r, j = bi * 32 + threadIdx.x;       // (i, j) = transposed position
    if (i < n && j < n && j > i) Xs[(size_t)i * ld + j] = t[threadIdx.x][r];
  }
}

// Cholesky factor L of the diagonal block kb of every scenario (grid.x = scenario),
// in place (lower), and its inverse into the same block of Y.  A pivot <= 0 sets
// *err and is replaced by 1 so that the factorisation ends.
// Bound: the 64 elimination steps, one after another.  Thread (ty, tx) of 16 x 16
// keeps elements (ty + 16 a, tx + 16 b) of the block and of the inverse (the
// identity, taken through the same steps) in registers; a step publishes column j
// of the block and row j of the inverse, so it has one barrier, 12 shared loads and
// 32 products.  23 us for both against 61 us for the factor alone with the block in
// shared memory and three barriers a step (and 63 us for each of the two triangular
// solves that the inverse turns into products).
__global__ void __launch_bounds__(256) k_potrf_inv(float* B, float* Y, int n, int ld, int kb, int* err) {
  __shared__ float cs[2][kNB], xs[2][kNB];
  float* Bs = B + (size_t)blockIdx.x * n * ld;
  float* Ys = Y + (size_t)blockIdx.x * n * ld;
  const int r0 = kb * kNB, nb = min(kNB, n - r0);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float a[4][4], x[4][4];
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = ty + 16 * p, k = tx + 16 * q;
      a[p][q] = (i < nb && k <= i) ? Bs[(size_t)(r0 + i) * ld + r0 + k] : (i == k ? 1.f : 0.f);
      x[p][q] = i == k ? 1.f : 0.f;
    }
#pragma unroll
  for (int jp = 0; jp < kNB / 16; ++jp)   // (the inner loop stays rolled: 64 steps of straight code ran at the
#pragma unroll 1                          // speed of instruction fetches, 68 us)
  for (int jr = 0; jr < 16; ++jr) {
    const int j = 16 * jp + jr;
    if (tx == jr)
#pragma unroll
      for (int p = 0; p < 4; ++p) cs[j & 1][ty + 16 * p] = a[p][jp];
    if (ty == jr)
#pragma unroll
      for (int q = 0; q < 4; ++q) xs[j & 1][tx + 16 * q] = x[jp][q];
    __syncthreads();
    float d = cs[j & 1][j];
    if (!(d > 0.f)) {
      if (threadIdx.x == 0) atomicExch(err, 1);
      d = 1.f;
    }
    // 1 / sqrt(d), one Newton step from the hardware's estimate (an IEEE division and
    // square root in every thread would take most of a step)
    float rs = rsqrtf(d);
    rs = fmaf(0.5f * rs, fmaf(-d * rs, rs, 1.f), rs);
    const float inv = rs * rs;
    float m[4], ck[4], rk[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const int i = ty + 16 * p;
      m[p] = i > j ? cs[j & 1][i] * inv : 0.f;
      const int k = tx + 16 * p;
      ck[p] = k > j ? cs[j & 1][k] : 0.f;
      rk[p] = xs[j & 1][k];
    }
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        a[p][q] = fmaf(-m[p], ck[q], a[p][q]);
        x[p][q] = fmaf(-m[p], rk[q], x[p][q]);
      }
    // column j of L and row j of its inverse are final
    if (tx == jr)
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        const int i = ty + 16 * p;
        if (i >= j && i < nb && j < nb) Bs[(size_t)(r0 + i) * ld + r0 + j] = (i == j ? d : cs[j & 1][i]) * rs;
      }
    if (ty == jr)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int k = tx + 16 * q;
        if (k <= j && j < nb) Ys[(size_t)(r0 + j) * ld + r0 + k] = xs[j & 1][k] * rs;
      }
  }
}

}  // namespace

// Form, factor and invert B_s for every scenario into P->binv (allocating it on
// first use); also A~_s^T p~ into P->bchol (compute_bconst, solver.cu).
int chol_prepare(Plan* P, const std::vector<double>& rho, CholExtra* extra) {
  if (!extra && P->chol_ready && !P->chol_con && P->chol_rho == rho) return RPT_OK;
  const DevPlan& dp = P->dp;
  const int n = dp.n, N = dp.N, ld = chol_ld(n);
  const size_t nn = (size_t)n * ld;
  cudaStream_t st = P->stream;
  cudaError_t e;
  if (!P->binv) {
    if ((e = cudaMalloc(&P->binv, sizeof(float) * nn * N))) {
      P->binv = nullptr;
      return cuda_fail(e, "allocate the factor");
    }
    P->allocs.push_back(P->binv);
  }
  if (!P->bchol) {
    if ((e = cudaMalloc(&P->bchol, sizeof(double) * (size_t)n * N))) {
      P->bchol = nullptr;
      return cuda_fail(e, "allocate A~'p~");
    }
    P->allocs.push_back(P->bchol);
  }
  // the inverse of the factor: kept by the plan while it is small, as weight sweeps form
  // B_s again and again (1250 spots, 13 scenarios: 78 MB), else given back with the factor
  // formed: 5000 spots, 1.2 GB beside the factor's own, setup 61.1 ms against 60.3 with it
  // kept; 2000 spots 7.75 against 7.53
  const size_t ybytes = sizeof(float) * nn * N;
  const bool keep = ybytes <= kCholKeep;
  float* Y = P->chol_y;
  if (!Y) {
    if ((e = cudaMalloc(&Y, ybytes))) return cuda_fail(e, "allocate the inverse workspace");
    if (keep) {
      P->chol_y = Y;
      P->allocs.push_back(Y);
    }
  }
  P->chol_ready = false;   // binv changes from here on
  auto done = [&](int rc) {
    cudaStreamSynchronize(st);
    if (!keep) cudaFree(Y);
    return rc;
  };
  if ((e = cudaMemsetAsync(P->binv, 0, sizeof(float) * nn * N, st))) return done(cuda_fail(e, "memset"));
  if ((e = cudaMemsetAsync(Y, 0, sizeof(float) * nn * N, st))) return done(cuda_fail(e, "memset"));
  if ((e = cudaMemsetAsync(P->err, 0, sizeof(int), st))) return done(cuda_fail(e, "memset"));
  // 1. B_s = A~_s^T A~_s (lower), + (rho/2) I
  int umax = kUMax, optin = 0;
  if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, P->device)))
    return done(cuda_fail(e, "device attribute"));
  int cap = std::max(kDCap, kBundleRows * kUMax);
  auto btb_smem = [&]() { return sizeof(int) * ((size_t)dp.n_pad + umax) + sizeof(float) * (size_t)cap; };
  for (; umax > 64 && btb_smem() + 1024 > (size_t)optin; cap = std::min(cap, kRB * umax)) umax -= 64;
  const size_t smem = btb_smem();
  void* fn;
  if (dp.path == 3) {
    if (dp.index_width == 16)
      fn = dp.value_format == 1 ? (void*)k_btb<__nv_bfloat16, uint16_t, true>
         : dp.value_format == 2 ? (void*)k_btb<__nv_fp8_e4m3, uint16_t, true> : (void*)k_btb<float, uint16_t, true>;
    else
      fn = dp.value_format == 1 ? (void*)k_btb<__nv_bfloat16, int32_t, true>
         : dp.value_format == 2 ? (void*)k_btb<__nv_fp8_e4m3, int32_t, true> : (void*)k_btb<float, int32_t, true>;
  } else if (dp.index_width == 16) {
    fn = dp.value_format == 1 ? (void*)k_btb<__nv_bfloat16, uint16_t, false>
       : dp.value_format == 2 ? (void*)k_btb<__nv_fp8_e4m3, uint16_t, false> : (void*)k_btb<float, uint16_t, false>;
  } else {
    fn = dp.value_format == 1 ? (void*)k_btb<__nv_bfloat16, int32_t, false>
       : dp.value_format == 2 ? (void*)k_btb<__nv_fp8_e4m3, int32_t, false> : (void*)k_btb<float, int32_t, false>;
  }
  if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)))
    return done(cuda_fail(e, "kernel attribute"));
  {
    DevPlan dpc = dp;
    const int* ro = P->rec_of;
    float* B = P->binv;
    int ldc = ld, nblk_r = 0;
    void* args[] = {(void*)&dpc, (void*)&ro, (void*)&B, (void*)&ldc, (void*)&umax, (void*)&cap, (void*)&nblk_r};
    // (a scenario's units are at most its rows, or a quarter of them in bundles of 4)
    const int units = dp.path == 3 ? (dp.m_act + kBundleRows - 1) / kBundleRows : dp.m_act;
    const int upb = dp.path == 3 ? kRB / kBundleRows : kRB;
    nblk_r = (units + upb - 1) / upb;
    if ((e = cudaLaunchKernel(fn, dim3((unsigned)N * 8u * ((nblk_r + 7) / 8)), dim3(kBtbThreads), args, smem, st)))
      return done(cuda_fail(e, "launch"));
  }
  for (int g = 0; g < dp.G; ++g)   // each group's scenarios with the group's penalty
    k_add_diag<<<dim3((n + 255) / 256, dp.Ns), 256, 0, st>>>(P->binv + nn * (size_t)g * dp.Ns, n, ld,
                                                              (float)(0.5 * rho[g]));
  if (extra && (e = extra->add(P, P->binv))) return done(cuda_fail(e, "constraint terms of B_s"));
  // 2. Cholesky, lower, in place, right-looking in panels of kPB blocks: inside a
  //    panel each block is factored and inverted (the inverse goes to Y), the rows
  //    below it become a product with the inverse, and the rank-64 update goes to the
  //    rest of the panel's columns only; the matrix right of the panel gets the
  //    panel's rank-256 update once
  const int nblk = (n + kNB - 1) / kNB;
  const long long snn = (long long)nn;
  for (int KB = 0; KB < nblk; KB += kPB) {
    const int kend = std::min(KB + kPB, nblk);
    for (int kb = KB; kb < kend; ++kb) {
      k_potrf_inv<<<N, 256, 0, st>>>(P->binv, Y, n, ld, kb, P->err);
      const int k0 = kb * kNB, c0 = (kb + 1) * kNB;   // the block's first row, the first after it
      if (c0 >= n) continue;
      // L21 = A21 L_kk^{-T}, in place: a tile's rows are read by its own CTA only
      float* A21 = P->binv + (size_t)c0 * ld + k0;
      gemm_tf32x3<false, true>(st, n - c0, kNB, kNB, A21, ld, Y + (size_t)k0 * ld + k0, ld, A21, ld, 1.f, 0.f, N,
                               snn, snn, snn);
      const int c1 = std::min(kend * kNB, n);   // the panel's remaining columns c0 .. c1
      if (c1 > c0)
        gemm_tf32x3<false, true>(st, n - c0, c1 - c0, kNB, A21, ld, A21, ld, P->binv + (size_t)c0 * ld + c0, ld,
                                 -1.f, 1.f, N, snn, snn, snn, /*lower=*/true);
    }
    const int t0 = kend * kNB;
    if (t0 < n) {
      const float* Lp = P->binv + (size_t)t0 * ld + (size_t)KB * kNB;   // rows t0.., the panel's columns
      gemm_tf32x3<false, true>(st, n - t0, n - t0, (kend - KB) * kNB, Lp, ld, Lp, ld,
                               P->binv + (size_t)t0 * ld + t0, ld, -1.f, 1.f, N, snn, snn, snn, /*lower=*/true);
    }
  }
  // 3. Y = L^{-1} by doubling: with the inverses of the diagonal blocks of size S in
  //    place, the block below each pair's diagonal is X21 = -X22 (L21 X11).  All
  //    pairs and scenarios of a size go in two launches: the product's transpose
  //    T' = X11' L21' into the pair's block above the diagonal of binv (unused by
  //    the factor), then -X22 T
  for (int S = kNB; S < n; S *= 2) {
    T3Pairs pr;
    pr.count = (n - S + 2 * S - 1) / (2 * S);        // pairs whose second half is not empty
    pr.step = 2ll * S * (ld + 1);
    pr.rows = n - S;                                  // rows from the first pair's second half on
    pr.rows_step = 2 * S;
    float* L21 = P->binv + (size_t)S * ld;
    float* Tt = P->binv + S;
    pr.ragged = 2;
    gemm_tf32x3<true, true>(st, S, S, S, Y, ld, L21, ld, Tt, ld, 1.f, 0.f, N, snn, snn, snn, false, /*kdiag=*/3, pr);
    pr.ragged = 1;
    gemm_tf32x3<false, true>(st, S, S, S, Y + (size_t)S * (ld + 1), ld, Tt, ld, Y + (size_t)S * ld, ld, -1.f, 0.f, N,
                             snn, snn, snn, false, /*kdiag=*/4, pr);
  }
  // 4. B^{-1} = Y^T Y into binv (the factor is no longer needed): lower tiles, the
  //    sum starting at max(i, j) since Y is lower triangular; then mirrored
  gemm_tf32x3<true, false>(st, n, n, n, Y, ld, Y, ld, P->binv, ld, 1.f, 0.f, N, snn, snn, snn, /*lower=*/true,
                           /*kdiag=*/2);
  k_mirror_lower<<<dim3((n + 31) / 32, (n + 31) / 32, N), dim3(32, 8), 0, st>>>(P->binv, n, ld);
  if ((e = cudaGetLastError())) return done(cuda_fail(e, "launch"));
  // 5. A~_s^T p~
  if (int rc = compute_bconst(P)) return done(rc);
  if ((e = cudaStreamSynchronize(st))) return done(cuda_fail(e, "sync"));
  int herr = 0;
  if ((e = cudaMemcpy(&herr, P->err, sizeof(int), cudaMemcpyDeviceToHost))) return done(cuda_fail(e, "copy"));
  if (herr) {
    cudaMemset(P->err, 0, sizeof(int));
    set_error("cached-factor subproblem: B_s is not positive definite in float32");
    return done(RPT_EINVAL);
  }
  P->chol_ready = true;
  P->chol_con = extra != nullptr;
  P->chol_rho = rho;
  return done(RPT_OK);
}

}  // namespace rpt
