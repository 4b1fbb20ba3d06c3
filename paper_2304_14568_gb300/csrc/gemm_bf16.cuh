// bfloat16 tensor-core GEMM for the learned warm start's network (the BF16
// compute form): warp-level mma.sync m16n8k16 with FP32 accumulation.
//   C = op(A) op(B) (+ bias[N], ReLU, or a ReLU-backward mask), and optionally a
//   bfloat16 copy Cb of the result (the next product's operand);
//   op(A)(i,k) = TA ? A[k*lda + i] : A[i*lda + k];  op(B)(k,j) = TB ? B[j*ldb + k] : B[k*ldb + j]
// Operands: 16-byte aligned rows (leading dimensions in multiples of 8), and
// zeros in the padding of a row that runs along k, so that every load is one
// 16-byte asynchronous copy.
//
// Bound: latency.  A minibatch of 128 rows through 512-wide layers is 67 MFLOP a
// product and a few hundred KB, so what counts is how many SMs take part and how
// few memory round trips a tile makes one after another.  A CTA of 4 warps
// computes a T x T tile, T = 32 unless 64 x 64 tiles alone fill the SMs, and
// keeps kTcStages K steps of 64 in flight (cp.async); operands reach the tensor
// cores by ldmatrix, transposed on the way where op() asks for it.  Every output
// is accumulated over k in steps of 16 in increasing order whatever the tile.
// Measured on a 128 x 9-512-512-512-200 minibatch: a 512-wide forward product 6 us
// against 70 us with 64 x 64 tiles staged by 2-byte loads without a pipeline; the
// whole loss and gradient call 107 us against 466 us, 500 x 9-384-384-702 129 us
// against 495 us.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace rpt {
namespace {

constexpr int kTcThreads = 128;
constexpr int kTcBK = 64, kTcPad = 8;

struct TcGemm {
  int M, N, K;
  const __nv_bfloat16 *A, *B;
  int lda, ldb;
  float* C;
  int ldc;
  __nv_bfloat16* Cb;      // or null
  int ldcb;
  const float* bias;      // [N] or null
  const float* mask;      // [M][ldc] or null: results where mask <= 0 become 0 (ReLU backward)
  int relu;
};

__device__ __forceinline__ void mma_bf16_m16n8k16(float (&d)[4], const uint32_t (&a)[4], const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
template <bool kTrans>
__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr) {
  if constexpr (kTrans)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// 16 bytes global -> shared, zeros when !ok (src is then not read)
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool ok) {
  const int n = ok ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}

// K steps in flight of a T x T tile.
template <int T> constexpr int kTcStages = T == 32 ? 4 : 2;
// elements of a stage: the larger of the [T][BK + pad] and [BK][T + pad] forms, both operands
template <int T>
constexpr int kTcTile = 2 * (T * (kTcBK + kTcPad) > kTcBK * (T + kTcPad) ? T * (kTcBK + kTcPad) : kTcBK * (T + kTcPad));

template <bool TA, bool TB, int T>
__device__ __forceinline__ void tc_gemm_tile(const TcGemm& g, int i0, int j0, __nv_bfloat16* sm) {
  constexpr int NS = kTcStages<T>;
  constexpr int kStage = kTcTile<T>, kHalf = kStage / 2;
  constexpr int SA = TA ? T + kTcPad : kTcBK + kTcPad, SB = TB ? kTcBK + kTcPad : T + kTcPad;
  constexpr int WT = T / 2, MT = WT / 16, NT2 = WT / 16;   // warp tile, its m16 tiles and pairs of n8 tiles
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = (warp >> 1) * WT, wn = (warp & 1) * WT;
  const int K8 = (g.K + 7) & ~7;       // the padding up to a multiple of 8 holds zeros
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(sm);
  auto load = [&](int kt, int st) {
    const int k0 = kt * kTcBK;
    const uint32_t sa = base + 2u * (uint32_t)(st * kStage), sb = sa + 2u * (uint32_t)kHalf;
#pragma unroll
    for (int q = 0; q < T * kTcBK / 8 / kTcThreads; ++q) {
      const int e = tid + q * kTcThreads;
      if constexpr (TA) {
        const int kk = e / (T / 8), ii = e % (T / 8) * 8, k = k0 + kk, i = i0 + ii;
        const bool ok = k < g.K && i < g.lda;
        cp_async16(sa + 2u * (uint32_t)(kk * SA + ii), ok ? g.A + (size_t)k * g.lda + i : g.A, ok);
      } else {
        const int ii = e / (kTcBK / 8), kk = e % (kTcBK / 8) * 8, k = k0 + kk, i = i0 + ii;
        const bool ok = i < g.M && k < K8;
        cp_async16(sa + 2u * (uint32_t)(ii * SA + kk), ok ? g.A + (size_t)i * g.lda + k : g.A, ok);
      }
      if constexpr (TB) {
        const int jj = e / (kTcBK / 8), kk = e % (kTcBK / 8) * 8, k = k0 + kk, j = j0 + jj;
        const bool ok = j < g.N && k < K8;
        cp_async16(sb + 2u * (uint32_t)(jj * SB + kk), ok ? g.B + (size_t)j * g.ldb + k : g.B, ok);
      } else {
        const int kk = e / (T / 8), jj = e % (T / 8) * 8, k = k0 + kk, j = j0 + jj;
        const bool ok = k < g.K && j < g.ldb;
        cp_async16(sb + 2u * (uint32_t)(kk * SB + jj), ok ? g.B + (size_t)k * g.ldb + j : g.B, ok);
      }
    }
  };
  const int nkt = (g.K + kTcBK - 1) / kTcBK;
#pragma unroll
  for (int s = 0; s < NS - 1; ++s) {
    if (s < nkt) load(s, s);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  float acc[MT][2 * NT2][4];
#pragma unroll
  for (int a = 0; a < MT; ++a)
#pragma unroll
    for (int b = 0; b < 2 * NT2; ++b)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[a][b][c] = 0.f;
  const int mat = lane >> 3, mr = lane & 7;   // ldmatrix: this lane addresses row mr of 8 x 8 matrix mat
  for (int kt = 0; kt < nkt; ++kt) {
    asm volatile("cp.async.wait_group %0;" ::"n"(NS - 2) : "memory");
    __syncthreads();   // the stage has arrived, and every warp is done with the stage refilled next
    if (kt + NS - 1 < nkt) load(kt + NS - 1, (kt + NS - 1) % NS);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const uint32_t sa = base + 2u * (uint32_t)(kt % NS * kStage), sb = sa + 2u * (uint32_t)kHalf;
#pragma unroll
    for (int ks = 0; ks < kTcBK; ks += 16) {
      uint32_t af[MT][4], bf[NT2][4];
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) {
        const int m0 = wm + mt * 16;
        // fragment order: (rows 0-7, k 0-7), (rows 8-15, k 0-7), (rows 0-7, k 8-15), (rows 8-15, k 8-15)
        const int row = TA ? ks + (mat >> 1) * 8 + mr : m0 + (mat & 1) * 8 + mr;
        const int cl = TA ? m0 + (mat & 1) * 8 : ks + (mat >> 1) * 8;
        ldmatrix_x4<TA>(af[mt], sa + 2u * (uint32_t)(row * SA + cl));
      }
#pragma unroll
      for (int nt = 0; nt < NT2; ++nt) {
        const int n0 = wn + nt * 16;
        // two n8 tiles: (k 0-7, n 0-7), (k 8-15, n 0-7), (k 0-7, n 8-15), (k 8-15, n 8-15)
        const int row = TB ? n0 + (mat >> 1) * 8 + mr : ks + (mat & 1) * 8 + mr;
        const int cl = TB ? ks + (mat & 1) * 8 : n0 + (mat >> 1) * 8;
        ldmatrix_x4<!TB>(bf[nt], sb + 2u * (uint32_t)(row * SB + cl));
      }
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int nt = 0; nt < 2 * NT2; ++nt) mma_bf16_m16n8k16(acc[mt][nt], af[mt], &bf[nt >> 1][(nt & 1) * 2]);
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  // accumulator layout: regs 0,1 at (row lane/4, cols 2 (lane%4), +1), regs 2,3 eight rows below
  const int gr = lane >> 2, gc = (lane & 3) * 2;
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int nt = 0; nt < 2 * NT2; ++nt)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = i0 + wm + mt * 16 + gr + (q >> 1) * 8;
        const int j = j0 + wn + nt * 8 + gc + (q & 1);
        if (i >= g.M || j >= g.N) continue;
        float v = acc[mt][nt][q];
        if (g.bias) v += g.bias[j];
        if (g.relu) v = fmaxf(v, 0.f);
        if (g.mask && !(g.mask[(size_t)i * g.ldc + j] > 0.f)) v = 0.f;
        g.C[(size_t)i * g.ldc + j] = v;
        if (g.Cb) g.Cb[(size_t)i * g.ldcb + j] = __float2bfloat16_rn(v);
      }
}

template <int T>
__host__ __device__ __forceinline__ int tc_tiles(const TcGemm& g) { return ((g.M + T - 1) / T) * ((g.N + T - 1) / T); }

// Tile edge: 64 when such tiles alone give every SM one, else 32.
inline bool tc_large(const TcGemm& g, int sm_count) { return tc_tiles<64>(g) >= sm_count; }

template <bool TA, bool TB, int T>
__device__ __forceinline__ void tc_gemm_block(const TcGemm& g, int blk, __nv_bfloat16* sm) {
  const int nj = (g.N + T - 1) / T;
  tc_gemm_tile<TA, TB, T>(g, blk / nj * T, blk % nj * T, sm);
}

}  // namespace
}  // namespace rpt
