// Row pass over row bundles with private accumulators (every mode of a plan whose
// shared memory holds them; the ring of rowpass.cu takes the others).
//
// The same pass as the bundled ring (one read of every stored block column;
// layout.h), with the same lanes per bundle and so the same dot products bit for
// bit, but without atomics and without a pace that all warps share:
//  * A CTA has A accumulators of n columns, each used by W / A warps in turn.  The
//    block columns of a bundle are distinct spots, so the one warp that adds a
//    bundle does it with plain loads and stores.  (A float atomic on shared memory
//    is a load, an add and a compare-and-swap in a retry loop; the ring spends a
//    third of its instructions there.)  The turns on an accumulator follow the
//    order of the work, and the accumulators are added in order at the end.
//  * The unit of work is an item: one bundle of 32 lanes, two of 16 or four of 8,
//    which are consecutive in memory.  Items go round-robin to the warps (the
//    bundles of a scenario are sorted by width, so neighbours cost the same), and
//    each is handled by code unrolled for its number of block columns per lane:
//    no warp looks at another warp's work.
//  * The shared memory left beside the accumulators is one ring of bytes.  Three
//    producer warps, one item per lane, place items of any size one after another
//    and copy them in (cp.async.bulk, one mbarrier per item).  A consumer frees an
//    item as soon as its values are in registers, before the reduction and the
//    scatter, so nearly the whole ring is in flight.
//  * CTA b takes the b-th share of the active scenarios' work (in units of equal
//    cost, layout.h): no queues, and the sums run in the same order every time.
//    A share is contiguous, so it holds one segment per scenario it touches, and
//    segment b + (rank of the scenario among the active ones) numbers the partial
//    sums without gaps: the slots of a scenario are consecutive, and no CTA has
//    to wait for the others to publish them.
// What bounds it: on the large plan the bytes on their way (HBM latency times
// bandwidth is about 50 KB an SM, and the accumulators of 5000 columns leave a ring
// of 128 KB for those, the items waiting and the gaps), on narrow bundles the
// instructions per bundle, on small plans the start (about 5 us).
// Measured, operator pass, against the ring with 1024 threads: realistic plan (F32,
// 862 MB) 0.153-0.158 ms against 0.181 (5.5 TB/s); BF16 + 16-bit plan of 3001 spots
// 0.074 against 0.099; 2000 spots 0.0575 against 0.082; 950 spots 0.034 against
// 0.055; 7000 spots, 3 scenarios 0.055 against 0.072; 250 spots 0.0124 against
// 0.029; 200 spots 0.0103 against 0.0275.
#include "rowcommon.cuh"

namespace rpt {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kProducers = 3;      // producer warps
constexpr int kPrivThreads = 512;  // largest CTA: 3 producer and 13 consumer warps (128 registers a thread)
constexpr int kItems = 128;        // descriptors, each with its mbarrier (a power of two)
// Most items in flight.  A consumer warp may wait for an item up to one round of
// the warps beyond the last one placed; with this bound the previous item of that
// descriptor has been freed by then, so the parity it waits for is not that of an
// item still on its way.
constexpr int kInFlight = 96;
constexpr int kPrivHdr = kItems * (8 + 16 + 4 + 4);   // full barriers, descriptors, done flags, ring ends
static_assert(kInFlight + kPrivThreads / 32 <= kItems, "see kInFlight");
constexpr int kWideMax = 12;       // = kWideKeep of layout.h: block columns per lane kept in registers by 32 lanes

// Item it of a scenario with cls = {bundles of 32 lanes, of 16, of 8}: its first
// bundle, bundle count and log2 of the lanes per bundle.
__device__ __forceinline__ void item_bundles(int it, const int4& cls, int& q, int& cnt, int& lg) {
  if (it < cls.x) {
    q = it;
    cnt = 1;
    lg = 5;
    return;
  }
  it -= cls.x;
  const int n16 = (cls.y + 1) >> 1;
  if (it < n16) {
    q = cls.x + 2 * it;
    cnt = min(2, cls.y - 2 * it);
    lg = 4;
    return;
  }
  it -= n16;
  q = cls.x + cls.y + 4 * it;
  cnt = min(4, cls.z - 4 * it);
  lg = 3;
}

__device__ __forceinline__ void st_release(uint32_t addr, int v) {
  asm volatile("st.release.cta.shared.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_acquire(uint32_t addr) {
  int v;
  asm volatile("ld.acquire.cta.shared.s32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}

// Bounded wait of a whole warp for a flag in shared memory to take the value v (one
// answer for all lanes, as warp_mbar_wait).  The first tries don't read the clock, whose
// read is slow: most turns come within them (200 spots 10.25 us a pass against 10.4-10.8,
// BF16 at 3001 73.7 against 74.6), which pays for the votes.
__device__ __forceinline__ bool warp_flag_wait(uint32_t addr, int v) {
  for (int k = 0; k < 16; ++k)
    if (__all_sync(kFull, ld_acquire(addr) == v)) return true;
  const unsigned long long t0 = global_ns();
  for (;;) {
    if (__all_sync(kFull, ld_acquire(addr) == v)) return true;
    if (__any_sync(kFull, global_ns() - t0 > kWaitLimitNs)) return false;
    __nanosleep(40);
  }
}

// What a consumer warp knows while it works on a segment.
struct Seg {
  const float* sv;       // staged vector, zero in the 32 idle columns behind the spots
  float* acc;            // this warp's accumulator (float, or int64 fixed point)
  int idle;              // this lane's idle column
  float fscale;          // fixed point: 2^F
  uint32_t turn_a;       // the accumulator's turn counter (modes that scatter)
  int turn;              // the item's turn
  bool ok;               // no wait ran out
  bool want_obj;
  float* dose;           // kDose: doses of the scenario
  double obj;
};

// One item: 32 / G bundles, G lanes each (wide: one of len block columns); block columns sl, sl + G, ... of a
// bundle are lane sl's, NS of them in registers.  CHK: slots from the end that may
// be absent (wide items: the earlier ones are full in every lane).  done: the
// item's flag, set to gen once its values are in registers (after the whole item
// when kTail: block columns beyond NS per lane are read from the ring twice).
template <int MODE, typename VT, typename IT, bool FIX, int NS, int CHK, bool kWide, bool kTail>
__device__ __forceinline__ void process_item(Seg& S, const int4* __restrict__ rec, int lo0, int len, bool valid, int lg,
                                             const VT* __restrict__ val, const IT* __restrict__ col, uint32_t done,
                                             int gen) {
  constexpr bool kScatter = (MODE == kNormal || MODE == kResid);
  const int lane = threadIdx.x & 31;
  const int G = kWide ? 32 : 1 << lg, sl = lane & (G - 1), sub = kWide ? 0 : lane >> lg;
  long long* acc = reinterpret_cast<long long*>(S.acc);
  int lo = 0, hi = len;
  if (!kWide && !valid) hi = 0;
  if (!kWide && valid) {
    lo = rec[4 * sub].x - lo0;
    hi = rec[4 * sub + 4].x - lo0;
  }
  float a[NS][4], o[NS];
  int c[NS];
  const int last = max(hi - 1, 0);   // absent lanes read a stored column (finite values) and meet sv = 0
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const int idx = lo + sl + G * k;
    if (k < NS - CHK) {
      quad_v<false, VT>(val + 4 * idx, a[k]);
      c[k] = (int)col[idx];
    } else {
      const int at = min(idx, last);
      quad_v<false, VT>(val + 4 * at, a[k]);
      c[k] = idx < hi ? (int)col[at] : S.idle;
    }
  }
  const int qd = G >> 2, rho = kWide ? sl >> 3 : sl >> (lg - 2);
  float wc = 0.f, pr = 0.f;
  int kept = -1;
  if (kWide || valid) {
    wc = __int_as_float(reinterpret_cast<const int*>(&rec[4 * sub + 1])[rho]);
    if (MODE != kNormal) pr = __int_as_float(reinterpret_cast<const int*>(&rec[4 * sub + 2])[rho]);
    if (MODE == kDose) kept = reinterpret_cast<const int*>(&rec[4 * sub + 3])[rho];
  }
  if (!kTail) {
    __syncwarp();
    if (lane == 0) st_release(done, gen);
  }
  float t[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const float v = S.sv[c[k]];
#pragma unroll
    for (int r = 0; r < 4; ++r) t[r] = fmaf(a[k][r], v, t[r]);
  }
  if (kTail)
    for (int idx = lo + 32 * NS + sl; idx < hi; idx += 32) {
      float q[4];
      quad_v<false, VT>(val + 4 * idx, q);
      const float v = S.sv[(int)col[idx]];
#pragma unroll
      for (int r = 0; r < 4; ++r) t[r] = fmaf(q[r], v, t[r]);
    }
  // transposing butterfly: halves exchange rows {0,1} / {2,3}, quarters one row;
  // after it, lane sl holds the whole dot of row sl / (G / 4)
  const int h = G >> 1;
  const bool up = (sl & h) != 0, up2 = (sl & qd) != 0;
  const float k0 = up ? t[2] : t[0], k1 = up ? t[3] : t[1];
  const float g0 = up ? t[0] : t[2], g1 = up ? t[1] : t[3];
  const float u0 = k0 + __shfl_xor_sync(kFull, g0, h);
  const float u1 = k1 + __shfl_xor_sync(kFull, g1, h);
  float tw = (up2 ? u1 : u0) + __shfl_xor_sync(kFull, up2 ? u0 : u1, qd);
  if (kWide) {
#pragma unroll
    for (int d = 4; d > 0; d >>= 1) tw += __shfl_xor_sync(kFull, tw, d);
  } else {
    for (int d = qd >> 1; d > 0; d >>= 1) tw += __shfl_xor_sync(kFull, tw, d);
  }
  float own;
  if (MODE == kNormal) {
    own = wc * tw;
  } else {
    const float rr = tw - pr;
    own = wc * rr;
    if ((kWide || valid) && (sl & (qd - 1)) == 0) {
      if (S.want_obj) S.obj += (double)(own * rr);
      if (MODE == kDose && kept >= 0) S.dose[kept] = tw;
    }
  }
  if (kScatter) {
    float cf[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) cf[r] = __shfl_sync(kFull, own, (kWide ? 0 : lane - sl) + r * qd);
    float sc[NS];
    long long qv[NS];    // fixed point: rounded before the turn is taken
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      sc[k] = cf[0] * a[k][0] + cf[1] * a[k][1] + cf[2] * a[k][2] + cf[3] * a[k][3];
      if (FIX) qv[k] = fixed_round(sc[k] * S.fscale);
    }
    S.ok = warp_flag_wait(S.turn_a, S.turn);
    if (!S.ok) return;   // nothing is added out of turn, and no turn is handed on
    // a bundle's columns are distinct: no two lanes or slots meet
    if (kWide) {
      if (FIX) {
        long long p[NS];
#pragma unroll
        for (int k = 0; k < NS; ++k) p[k] = acc[c[k]];
#pragma unroll
        for (int k = 0; k < NS; ++k) acc[c[k]] = p[k] + qv[k];
      } else {
#pragma unroll
        for (int k = 0; k < NS; ++k) o[k] = S.acc[c[k]];
#pragma unroll
        for (int k = 0; k < NS; ++k) S.acc[c[k]] = o[k] + sc[k];
      }
      if (kTail)
        for (int idx = lo + 32 * NS + sl; idx < hi; idx += 32) {
          float q[4];
          quad_v<false, VT>(val + 4 * idx, q);
          const float x = cf[0] * q[0] + cf[1] * q[1] + cf[2] * q[2] + cf[3] * q[3];
          if (FIX) acc[(int)col[idx]] += fixed_round(x * S.fscale);
          else S.acc[(int)col[idx]] += x;
        }
      __syncwarp();   // the next item's adds see these
    } else {
#pragma unroll
      for (int q = 0; q < 32; q += 8) {   // the item's bundles take turns
        if ((q & (G - 1)) != 0) continue;
        if (lane - sl == q) {
          if (FIX) {
            long long p[NS];
#pragma unroll
            for (int k = 0; k < NS; ++k) p[k] = acc[c[k]];
#pragma unroll
            for (int k = 0; k < NS; ++k) acc[c[k]] = p[k] + qv[k];
          } else {
#pragma unroll
            for (int k = 0; k < NS; ++k) o[k] = S.acc[c[k]];
#pragma unroll
            for (int k = 0; k < NS; ++k) S.acc[c[k]] = o[k] + sc[k];
          }
        }
        __syncwarp();
      }
    }
    if (lane == 0) st_release(S.turn_a, S.turn + 1);
  }
  if (kTail) {
    __syncwarp();
    if (lane == 0) st_release(done, gen);
  }
}

template <int MODE, typename VT, typename IT, bool FIX>
__global__ void __launch_bounds__(kPrivThreads, 1)
k_rowpass_priv(DevPlan P, const float* __restrict__ vin, int v_stride, const int* __restrict__ active,
               float* __restrict__ partial, double* __restrict__ objp, float* __restrict__ dose) {
  constexpr bool kScatter = (MODE == kNormal || MODE == kResid);
  constexpr bool FX = FIX && kScatter;
  constexpr int ACCB = FIX ? 8 : 4;             // accumulator bytes per column
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ long long wsum[kPrivThreads / 32];
  __shared__ int sh_start[3];                   // this CTA's first scenario, first unit in it, rank
  __shared__ double wobj[kPrivThreads / 32];
  __shared__ float wmax[kPrivThreads / 32];
  __shared__ int sh_fail;                       // a consumer's wait ran out
  __shared__ int turns[kPrivThreads / 32];      // items added to each accumulator
  __shared__ int2 post[2];                      // producers: items placed, ring position before them
  uint64_t* full = reinterpret_cast<uint64_t*>(smem);
  int4* desc = reinterpret_cast<int4*>(smem + 8 * kItems);
  int* done = reinterpret_cast<int*>(smem + 24 * kItems);
  unsigned* ends = reinterpret_cast<unsigned*>(smem + 28 * kItems);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int A = P.priv_acc;                                      // accumulators
  const int nthr = blockDim.x, W = (nthr >> 5) - kProducers;     // consumer warps
  const int AS = P.n_pad + 32;
  float* sv = reinterpret_cast<float*>(smem + kPrivHdr);
  unsigned char* acc0 = smem + kPrivHdr + sizeof(float) * AS;
  const size_t accs = kScatter ? (size_t)AS * ACCB : 0;
  unsigned char* ring = smem + round128(kPrivHdr + sizeof(float) * AS + (size_t)A * AS * (P.acc64 ? 8 : 4));

  if (tid < kItems) {
    mbar_init(smem_u32(&full[tid]), 1);
    done[tid] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid == 0) sh_fail = 0;
  if (tid < kPrivThreads / 32) turns[tid] = P.inject_timeout == 2 ? -1 : 0;   // (testing: no turn ever comes)
  // ---- this CTA's share of the active scenarios' units ----
  // thread t sums the units of scenarios [t per, (t + 1) per); (rank, units)
  // packed in one 64-bit prefix sum over the block
  const int per = (P.N + nthr - 1) / nthr;
  auto units_of = [&](int s) {
    return (active == nullptr || __ldcg(&active[s]) != 0) ? P.uoff[s + 1] - P.uoff[s] : 0;
  };
  long long mine = 0;
  for (int s = tid * per; s < min((tid + 1) * per, P.N); ++s) {
    const int u = units_of(s);
    mine += u + (u > 0 ? (1ll << 32) : 0);
  }
  long long incl = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const long long y = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += y;
  }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  long long before = incl - mine, total = 0;
  for (int k = 0; k < (nthr >> 5); ++k) {
    if (k < warp) before += wsum[k];
    total += wsum[k];
  }
  const int T = (int)(total & 0xffffffffll);
  const int G = min((int)gridDim.x, T);
  const int b = blockIdx.x;
  // CTA b's share is [floor(b T / G), floor((b + 1) T / G)), so unit u belongs to
  // CTA ceil((u + 1) G / T) - 1
  const int U0 = b < G ? (int)((long long)b * T / G) : 0, U1 = b < G ? (int)((long long)(b + 1) * T / G) : 0;
  {
    int pre = (int)(before & 0xffffffffll), rank = (int)(before >> 32);
    for (int s = tid * per; s < min((tid + 1) * per, P.N); ++s) {
      const int u = units_of(s);
      if (u > 0 && b < G && U0 >= pre && U0 < pre + u) {
        sh_start[0] = s;
        sh_start[1] = U0 - pre;
        sh_start[2] = rank;
      }
      if (b == 0) {   // the scenario's slots: consecutive segments
        int cnt = 0;
        if (u > 0) {
          const int b0 = (int)(((long long)(pre + 1) * G - 1) / T), b1 = (int)(((long long)(pre + u) * G - 1) / T);
          cnt = b1 - b0 + 1;
          P.slot_list[(size_t)s * P.slot_cap] = b0 + rank;   // the first; the others follow it
        }
        P.slot_count[s] = cnt;
      }
      pre += u;
      rank += u > 0;
    }
  }
  __syncthreads();
  int left = U1 - U0;                                   // units
  int s = left > 0 ? sh_start[0] : 0;
  int u0 = left > 0 ? P.uoff[s] + sh_start[1] : 0;      // next unit, of scenario s
  // items [ib, ie) of scenario s in the units [u0, u0 + take) (a scenario's last unit ends with its items)
  auto seg_items = [&](int take, int& ib, int& ie, int4& cls) {
    cls = P.cls[s];
    ib = P.ubeg[u0];
    ie = u0 + take < P.uoff[s + 1] ? P.ubeg[u0 + take] : cls.w;
  };
  auto next_scenario = [&]() {
    do ++s;
    while (units_of(s) == 0);
    u0 = P.uoff[s];
  };

  if (warp < kProducers) {
    // ---------------- producers: one item per lane ----------------
    // warp 0 places the items and copies their values, warps 1 and 2 their spot
    // indices and records: a warp issues a bulk copy per lane in about 70 cycles
    if (P.inject_timeout == 1) left = 0;
    constexpr int VA = 16 / (4 * (int)sizeof(VT)), IA = 16 / (int)sizeof(IT);   // columns per 16 bytes
    const unsigned R = (unsigned)P.ring_bytes;
    const uint32_t ring_a = smem_u32(ring), done_a = smem_u32(done);
    unsigned pos = 0, head = 0, tail = 0;   // ring position; bytes placed and freed (skipped ends included)
    int issued = 0, freed = 0;              // items
    int par = 0;
    bool ok = true;
    while (left > 0 && ok) {
      const int take = min(left, P.uoff[s + 1] - u0);
      int ib, ie;
      int4 cls;
      seg_items(take, ib, ie, cls);
      const int4* rec = P.rowrec + P.rec_base[s];
      const VT* gval = vals<VT>(P);
      const IT* gcol = cols<IT>(P);
      const long long base = P.nnz_base[s];
      int q = 0, cnt = 0, lg = 0, lo = 0, hi = 0;
      auto fetch = [&](int at) {            // bundles and column range of this lane's item of the batch
        cnt = 0;
        if (at + lane < ie) {
          item_bundles(at + lane, cls, q, cnt, lg);
          lo = __ldg(&rec[4 * (size_t)q].x);
          hi = __ldg(&rec[4 * (size_t)(q + cnt)].x);
        }
      };
      fetch(ib);
      for (int at = ib; at < ie && ok; at += 32) {
        const int q_ = q, cnt_ = cnt, lg_ = lg, lo_ = lo, hi_ = hi;
        fetch(at + 32);                     // the next batch's, in flight meanwhile
        // bytes of the item: values, spot indices, records
        const long long g0 = base + lo_, g1 = base + hi_;
        const long long v0 = g0 & ~(long long)(VA - 1), i0 = g0 & ~(long long)(IA - 1);
        const unsigned vb = cnt_ ? (unsigned)(((g1 + VA - 1) & ~(long long)(VA - 1)) - v0) * (4u * sizeof(VT)) : 0u;
        const unsigned cb = cnt_ ? (unsigned)(((g1 + IA - 1) & ~(long long)(IA - 1)) - i0) * (unsigned)sizeof(IT) : 0u;
        const unsigned rb = cnt_ ? (unsigned)cnt_ * 64u + 16u : 0u;
        const unsigned size = vb + cb + rb;
        const int n_at = min(32, ie - at);
        unsigned sum = size;                // bytes of the batch's items up to and with this one
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const unsigned y = __shfl_up_sync(kFull, sum, d);
          if (lane >= d) sum += y;
        }
        int from = 0;                       // items of the batch placed so far
        unsigned used = 0;                  // their bytes
        while (from < n_at) {
          if (warp == 0) {
            unsigned long long t0 = 0;
            int k = 0;                      // items placed now, -1: no room came free in time
            while (k == 0) {
              // the items that fit at pos, in the free bytes and descriptors, without wrapping
              const bool fits = lane >= from && lane < n_at && pos + (sum - used) <= R &&
                                head + (sum - used) - tail <= R && issued + (lane - from) - freed < kInFlight;
              k = __popc(__ballot_sync(kFull, fits));   // the first ones, as all bounds grow along the batch
              if (k > 0) break;
              const unsigned need = __shfl_sync(kFull, size, from);
              if (pos + need > R) {         // does not fit before the end: skip to the start
                head += R - pos;
                pos = 0;
                if (freed == issued) tail = head;
                continue;
              }
              // free the items done, in order
              int f = 0;
              if (freed + lane < issued) {
                const int i = freed + lane, e = i & (kItems - 1);
                f = ld_acquire(done_a + 4u * (unsigned)e) == i / kItems + 1;
              }
              const unsigned bal = __ballot_sync(kFull, f);
              const int nf = bal == kFull ? 32 : __ffs(~bal) - 1;
              if (nf > 0) {
                tail = ends[(freed + nf - 1) & (kItems - 1)];
                freed += nf;
                if (freed == issued) tail = head;   // nothing in flight: skipped bytes are free too
                t0 = 0;
              } else {
                const unsigned long long now = global_ns();
                if (t0 == 0) t0 = now;
                if (now - t0 > kWaitLimitNs) k = -1;
                else __nanosleep(20);
              }
            }
            if (lane == 0) post[par] = make_int2(k, (int)pos);
          }
          named_sync(2, kProducers * 32);   // the placement is posted, and the previous one taken
          const int2 m = post[par];
          par ^= 1;
          if (m.x < 0) {
            ok = false;
            break;
          }
          pos = (unsigned)m.y;
          if (lane >= from && lane < from + m.x) {
            const int e = (issued + lane - from) & (kItems - 1);
            const uint32_t fb = smem_u32(&full[e]);
            const unsigned p = pos + (sum - used) - size;
            if (warp == 0) {
              int4 d;
              d.x = (int)(p + (unsigned)(g0 - v0) * (4u * sizeof(VT)));
              d.y = (int)(p + vb + (unsigned)(g0 - i0) * (unsigned)sizeof(IT));
              d.z = (int)(p + vb + cb) | (cnt_ << 20) | (lg_ << 24);
              d.w = lo_;
              desc[e] = d;
              ends[e] = head + (sum - used);
              mbar_arrive_expect_tx(fb, size);   // (the other copies may complete first: the phase waits for this arrival)
              bulk_g2s(ring_a + p, gval + v0 * 4, vb, fb);
            } else if (warp == 1) {
              bulk_g2s(ring_a + p + vb, gcol + i0, cb, fb);
            } else {
              bulk_g2s(ring_a + p + vb + cb, rec + 4 * (size_t)q_, rb, fb);
            }
          }
          const unsigned add = __shfl_sync(kFull, sum, from + m.x - 1) - used;
          pos += add;
          head += add;
          used += add;
          issued += m.x;
          from += m.x;
          __syncwarp();
        }
      }
      left -= take;
      if (left > 0 && ok) next_scenario();
    }
    if (warp == 0) {
      if (!ok && lane == 0) atomicExch(P.err, 1);
      // the copies in flight end before the CTA does, whatever became of its consumers
      for (int i = freed + lane; i < issued; i += 32)
        if (!mbar_wait(smem_u32(&full[i & (kItems - 1)]), (uint32_t)(i / kItems) & 1u)) atomicExch(P.err, 2);
    }
  } else {
    // ---------------- consumers ----------------
    const int cw = warp - kProducers, ct = tid - 32 * kProducers, nc = W * 32;
    Seg S;
    S.sv = sv;
    S.acc = reinterpret_cast<float*>(acc0 + accs * (cw % A));
    S.turn_a = smem_u32(&turns[cw % A]);   // (turns are always taken: a plan has fewer accumulators than warps)
    S.ok = true;
    S.idle = P.n_pad + lane;
    S.want_obj = MODE != kNormal && objp != nullptr;
    int seg = left > 0 ? b + sh_start[2] : 0;
    int it = cw;               // this warp's next item, counted over the CTA's share
    int seg_first = 0;         // the segment's first item
    bool ok = true;
    const uint32_t done_a = smem_u32(done);
    while (left > 0 && ok) {
      const int take = min(left, P.uoff[s + 1] - u0);
      int ib, ie;
      int4 cls;
      seg_items(take, ib, ie, cls);
      // ---- stage v_s (scaled by the column scales of quantised values), zero the accumulator ----
      float vm = 0.f;
      {
        const float4* v4 = reinterpret_cast<const float4*>(vin + (size_t)s * v_stride);
        const float4* cs4 = P.colscale ? reinterpret_cast<const float4*>(P.colscale + (size_t)s * P.n_pad) : nullptr;
        bool bad = false;
        for (int k = ct; k < AS / 4; k += nc) {
          float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
          if (k < P.n_pad / 4) {
            x = v4[k];
            if (cs4) {
              const float4 q = cs4[k];
              x.x *= q.x; x.y *= q.y; x.z *= q.z; x.w *= q.w;
            }
          }
          reinterpret_cast<float4*>(sv)[k] = x;
          if (FX) {
            vm = fmaxf(vm, fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w))));
            bad |= !(isfinite(x.x) && isfinite(x.y) && isfinite(x.z) && isfinite(x.w));
          }
        }
        if (FX && bad) vm = __int_as_float(0x7f800000);
        if (kScatter)
          for (int k = ct; k < A * (AS * ACCB / 16); k += nc)
            reinterpret_cast<float4*>(acc0)[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
      int fexp = 0;
      S.fscale = 0.f;
      if (FX) {
        vm = warp_max(vm);
        if (lane == 0) wmax[cw] = vm;
      }
      named_sync(1, nc);
      if (FX) {
        float vmax = 0.f;     // +inf if the vector is not finite
        for (int k = 0; k < W; ++k) vmax = fmaxf(vmax, wmax[k]);
        fexp = fixed_exp(vmax, P.kbound[2 * s], MODE == kResid ? P.kbound[2 * s + 1] : 0.0);
        S.fscale = (fexp == kFexpNaN) ? 0.f : __int_as_float((fexp + 127) << 23);
      }
      S.dose = MODE == kDose ? dose + (size_t)s * P.m_act : nullptr;
      S.obj = 0.0;
      const int seg_end = seg_first + (ie - ib);
      for (; it < seg_end; it += W) {
        const int e = it & (kItems - 1), gen = it / kItems + 1;
        if (!warp_mbar_wait(smem_u32(&full[e]), (uint32_t)(it / kItems) & 1u)) {
          if (lane == 0) {
            atomicExch(P.err, 3);
            sh_fail = 1;
          }
          break;
        }
        const int4 d = desc[e];
        const int lo = d.w;
        const VT* val = reinterpret_cast<const VT*>(ring + d.x);
        const IT* col = reinterpret_cast<const IT*>(ring + d.y);
        const int4* rec = reinterpret_cast<const int4*>(ring + (d.z & 0xfffff));
        const int cnt = (d.z >> 20) & 15, lg = d.z >> 24;
        const uint32_t fl = done_a + 4u * (unsigned)e;
        S.turn = it / A;
        const int len = rec[4].x - lo;     // block columns of the item's first bundle, its widest
        if (lg == 5) {
          switch ((len + 31) >> 5) {
#define RPT_WIDE(NS, CHK) process_item<MODE, VT, IT, FX, NS, CHK, true, false>(S, rec, lo, len, true, 5, val, col, fl, gen)
            case 0: case 1: case 2: case 3: case 4: RPT_WIDE(4, 4); break;
            case 5: RPT_WIDE(5, 1); break;
            case 6: RPT_WIDE(6, 1); break;
            case 7: RPT_WIDE(7, 1); break;
            case 8: RPT_WIDE(8, 1); break;
            case 9: case 10: RPT_WIDE(10, 2); break;
            case 11: case 12: RPT_WIDE(kWideMax, 2); break;
#undef RPT_WIDE
            default:
              process_item<MODE, VT, IT, FX, kWideMax, 0, true, true>(S, rec, lo, len, true, 5, val, col, fl, gen);
          }
        } else {
          const bool valid = (lane >> lg) < cnt;
          const int ns = (len + (1 << lg) - 1) >> lg;      // at most kBundleKeep (layout.h)
          if (ns <= 2)
            process_item<MODE, VT, IT, FX, 2, 2, false, false>(S, rec, lo, len, valid, lg, val, col, fl, gen);
          else if (ns <= 4)
            process_item<MODE, VT, IT, FX, 4, 4, false, false>(S, rec, lo, len, valid, lg, val, col, fl, gen);
          else
            process_item<MODE, VT, IT, FX, kBundleKeep, kBundleKeep, false, false>(S, rec, lo, len, valid, lg, val, col,
                                                                                   fl, gen);
        }
        if (!S.ok) break;
      }
      if (!S.ok && lane == 0) {
        atomicExch(P.err, 4);
        sh_fail = 1;
      }
      seg_first = seg_end;
      if (MODE != kNormal) {
        const double obj = warp_sum_d(S.obj);
        if (lane == 0) wobj[cw] = obj;
      }
      named_sync(1, nc);
      // ---- the segment's sums over the warps, in warp order ----
      if (FX) {
        const unsigned long long* a0 = reinterpret_cast<const unsigned long long*>(acc0);
        unsigned long long* out = reinterpret_cast<unsigned long long*>(partial) + (size_t)seg * P.n_pad;
        for (int k = ct; k < P.n_pad; k += nc) {
          unsigned long long x = 0;
          for (int i = 0; i < A; ++i) x += a0[(size_t)i * AS + k];
          out[k] = x;
        }
        if (ct == 0) P.fexp[s] = fexp;
      } else if (kScatter) {
        const float4* cs4 = P.colscale ? reinterpret_cast<const float4*>(P.colscale + (size_t)s * P.n_pad) : nullptr;
        float4* out = reinterpret_cast<float4*>(partial + (size_t)seg * P.n_pad);
        for (int k = ct; k < P.n_pad / 4; k += nc) {
          float4 x = reinterpret_cast<const float4*>(acc0)[k];
          for (int i = 1; i < A; ++i) {
            const float4 y = reinterpret_cast<const float4*>(acc0 + accs * i)[k];
            x.x += y.x; x.y += y.y; x.z += y.z; x.w += y.w;
          }
          if (cs4) {
            const float4 q = cs4[k];
            x.x *= q.x; x.y *= q.y; x.z *= q.z; x.w *= q.w;
          }
          out[k] = x;
        }
      }
      if (MODE != kNormal && objp != nullptr && ct == 0) {
        double q = 0.0;
        for (int k = 0; k < W; ++k) q += wobj[k];
        objp[seg] = q;
      }
      left -= take;
      ok = *(volatile int*)&sh_fail == 0;   // the same answer in every warp: the next segment starts behind a barrier
      if (left > 0) {
        named_sync(1, nc);
        ++seg;
        next_scenario();
      }
    }
  }
  if (MODE == kNormal || objp == nullptr) return;
  // ---- objective per scenario: the CTA that finishes last sums the segments in order ----
  __shared__ bool last_cta;
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    last_cta = (atomicAdd(P.done_ctr, 1u) + 1u == gridDim.x);
  }
  __syncthreads();
  if (!last_cta) return;
  __threadfence();
  for (int q = warp; q < P.N; q += nthr >> 5) {
    const int cnt = __ldcg(&P.slot_count[q]);
    const int first = cnt > 0 ? __ldcg(&P.slot_list[(size_t)q * P.slot_cap]) : 0;
    double o = 0.0;
    for (int k = lane; k < cnt; k += 32) o += __ldcg(&objp[first + k]);
    o = warp_sum_d(o);
    if (lane == 0) P.objs[q] = o;
  }
  if (tid == 0) *P.done_ctr = 0u;
}

template <int MODE, typename IT, bool FIX>
void* pick_v(const DevPlan& P) {
  switch (P.value_format) {
    case 1: return (void*)k_rowpass_priv<MODE, __nv_bfloat16, IT, FIX>;
    case 2: return (void*)k_rowpass_priv<MODE, __nv_fp8_e4m3, IT, FIX>;
    default: return (void*)k_rowpass_priv<MODE, float, IT, FIX>;
  }
}

template <int MODE>
constexpr bool kScatterMode = (MODE == kNormal || MODE == kResid);

template <int MODE>
void* pick_m(const DevPlan& P) {
  if (P.acc64)   // fixed-point sums (of the modes that scatter)
    return P.index_width == 16 ? pick_v<MODE, uint16_t, kScatterMode<MODE>>(P)
                               : pick_v<MODE, int32_t, kScatterMode<MODE>>(P);
  return P.index_width == 16 ? pick_v<MODE, uint16_t, false>(P) : pick_v<MODE, int32_t, false>(P);
}

}  // namespace

int priv_threads(int warps) { return 32 * (warps + kProducers); }

void* priv_rowpass_kernel(const DevPlan& P, int mode) {
  switch (mode) {
    case kNormal: return pick_m<kNormal>(P);
    case kResid: return pick_m<kResid>(P);
    case kObj: return pick_m<kObj>(P);
    default: return pick_m<kDose>(P);
  }
}

// Shared memory before the ring: the header, the staged vector and the
// accumulators.
size_t priv_fixed_bytes(int n_pad, int accs, bool fixed) {
  const size_t as = (size_t)n_pad + 32;
  return round128(kPrivHdr + 4 * as + (size_t)accs * as * (fixed ? 8 : 4));
}

}  // namespace rpt
