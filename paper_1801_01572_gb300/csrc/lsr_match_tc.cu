// lsr_match_tc.cu -- the feature pre-matching cache (Algorithm 1, "Parallel
// FPFH feature pre-matching") on the 5th-generation tensor cores.
//
// The squared descriptor distance |a - b|^2 = |a|^2 + |b|^2 - 2 a.b is a dense
// contraction. Descriptors are first centred on a mean descriptor c (distances
// do not change; the magnitudes that set the FP32 accumulation error shrink)
// and rounded to BF16. Two operand layouts:
//   plain (K = 48):  x ~ h = bf16(x); the contraction is h_a . h_b.
//   split (K = 112): x ~ h + l with l = bf16(x - h); the contraction is
//                    h_a.h_b + l_a.h_b + h_a.l_b (the l_a.l_b term, below
//                    2^-16 |a||b|, is left out and bounded).
// Three spare K columns carry |b~|^2 as three BF16 parts (query side 1.0) and
// the query side is pre-scaled by -2 (exact), so the FP32 accumulator holds the
// score s = |b~|^2 - 2 a~.b~ and the epilogue only compares.
//
// Both sets are put in the matchers' descriptor order (lsr_order.cu), so a tile
// of 128 rows is a box of a k-d tree, and a first pass of the FP32 matcher over
// the two nearest leaves gives every query a row at a known distance. A work
// item is one unit of 128 or 256 queries (one or two M = 128 tiles sharing
// every database tile; the shape is chosen per size by the autotuner) and the
// tiles, of 64 consecutive ones, whose boxes some query of the unit reaches
// within that distance: k_tc_items lists the items, largest first. On room
// descriptors a tenth of the tiles is left: k_match_tc takes 1.0 ms for 200k x
// 200k instead of 8.5, the matching stage 1.8 instead of 10.0 (40k x 40k, the
// whole call: 0.54 ms instead of 1.04).
// Sets too small to repay the ordering, or too large for the item list, take
// all tiles in the caller's order.
//
// Persistent CTAs take items in turn: one thread streams their tiles through
// shared memory and issues tcgen05.mma into TMEM (two accumulator buffers, so
// the tensor pipe runs while the epilogue drains the other), and four or eight
// epilogue warps, one query per thread, read a whole accumulator row with one
// wait, release the buffer at once, and keep the 8 smallest minima of 16-row
// chunks (a chunk enters when its minimum beats the lane's current 8th).
//
// At the end of an item the chunks are re-ranked, best first, with the exact
// FP32 distance of the original descriptors in the FP32 matcher's operation
// order, as long as a chunk can hold a row at or below the query's best
// distance so far, which all items of a query share (a 64-bit atomic minimum of
// distance and index). D~^2 = s + |a~|^2 is within efp of |a~ - b~|^2
// (accumulation, the left-out l_a.l_b term) and |a~ - b~| within eta of the
// true distance, so a chunk whose minimum, less efp and eta, exceeds the best
// holds no nearer row and no tie, and neither does any chunk after it. A query
// whose eight chunks were all within reach, with a ninth possibly so, is left
// to the FP32 matcher (its search through the boxes; without the order, a scan
// of the whole database). The result is the FP32 matcher's, bit for bit.
// The accumulation error is bounded with the truncating-adder model of tensor
// core FP32 accumulation: each MMA of 16 products adds at most 17 errors of
// 2^-23 times the largest magnitude involved, i.e. 15e-6 * sum |products| for
// the 7 MMAs of the split layout (the validation entry point measures it).
//
// Tiles sit in global memory already in the layout the MMA reads from shared
// memory (K-major, no swizzle: 8 rows x 16 bytes per core matrix, K-adjacent
// core matrices 128 bytes apart, 8-row groups K/8 * 128 bytes apart), so every
// tile arrives with one bulk copy completed on an mbarrier. Every wait is
// bounded in time: a CTA that gives up records an error, stops issuing work,
// waits (bounded) for its copies and MMAs in flight, releases TMEM and returns.
#include <cuda_bf16.h>
#include <float.h>

#include "lsr_internal.cuh"

namespace lsr {

namespace {

constexpr int kTcM = 128;                       // queries per MMA tile (TMEM lanes)
constexpr int kTcN = 128;                       // database rows per tile
constexpr int kLBO = 128;                       // bytes between K-adjacent core matrices
constexpr int kTopK = 8;                        // candidate chunks per query and item
constexpr int kChunkW = 16;                     // database rows per chunk
constexpr int kChunks = kTcN / kChunkW;         // chunks per tile
constexpr int kLoads = kTcN / 32;               // 32-column TMEM loads per accumulator row
constexpr unsigned long long kWaitNs = 2000000000ull;  // give up after 2 s (the default limit; drains always)
constexpr float kPadScore = 1.2676506e30f;      // 2^100: |b~|^2 of padding rows
constexpr float kAccErr = 1.5e-5f;              // accumulation error per unit of sum |products|
constexpr int kCenterGroups = 8;                // row groups of the centring kernel

// Operand layout of one mode: KS MMA k-steps of 16.
template <int KS>
struct Shape {
  static constexpr bool kSplit = KS == 7;
  static constexpr int K = 16 * KS;
  static constexpr int SBO = (K / 8) * 128;      // bytes between 8-row groups
  static constexpr int TileBytes = kTcM * K * 2;
  static constexpr int SqCol = kSplit ? 3 * kD : kD;  // first |b~|^2 column
  static_assert(SqCol + 3 <= K, "operand layout");
};

// Tile shape of the persistent CTA: QT query tiles of 128 per work unit.
//   QT = 2: 256 queries share every database tile; 4 copy stages; 512 TMEM
//           columns (two buffers of 2 x 128): one CTA per SM.
//   QT = 1: 128 queries; 3 stages; 256 TMEM columns: two CTAs per SM, so
//           small clouds still spread over every SM.
template <int KS, int QT>
struct Cfg {
  static constexpr int Stages = QT == 2 ? 4 : 3;
  static constexpr int EpiWarps = 4 * QT;        // warps 0..EpiWarps-1: epilogue; the next: copies + MMA
  static constexpr int Threads = (EpiWarps + 1) * 32;
  static constexpr int UnitQ = QT * kTcM;
  static constexpr uint32_t AccCols = QT * kTcN; // one accumulator buffer
  static constexpr uint32_t TmemCols = 2 * AccCols;
  static constexpr int CtasPerSm = QT == 2 ? 1 : 2;
  static constexpr int UnitBytes = QT * Shape<KS>::TileBytes;
  static constexpr int SmemUsed = UnitBytes + Stages * Shape<KS>::TileBytes + 128;
  // enough shared memory that no more CTAs than TMEM holds share an SM
  static constexpr int SmemFloor = CtasPerSm == 1 ? 120 * 1024 : 80 * 1024;
  static constexpr int SmemBytes = SmemUsed > SmemFloor ? SmemUsed : SmemFloor;
  static_assert(CtasPerSm * (SmemBytes + 1024) <= 228 * 1024, "shared memory plan");
  static_assert(CtasPerSm * TmemCols <= 512, "tensor memory plan");
};

template <int KS>
__host__ __device__ inline int tc_off(int r, int k) {
  return (r >> 3) * Shape<KS>::SBO + (k >> 3) * kLBO + (r & 7) * 16 + (k & 7) * 2;
}

// ---------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t s2u(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned long long gtime() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint64_t *b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s2u(b)), "r"(count));
}
__device__ __forceinline__ bool mbar_try(uint64_t *b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(s2u(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Waits for the phase of the given parity; gives up after limit_ns (flagging
// the CTA) or as soon as another thread of the CTA has given up.
__device__ __forceinline__ bool mbar_wait(uint64_t *b, uint32_t parity, volatile int *fail,
                                          unsigned long long limit_ns) {
  if (mbar_try(b, parity)) return true;
  unsigned long long t0 = gtime();
  for (;;) {
    if (mbar_try(b, parity)) return true;
    if (*fail) return false;
    if (gtime() - t0 > limit_ns) {
      *fail = 1;
      return false;
    }
  }
}
// Bounded wait used only while cleaning up after a failure.
__device__ __forceinline__ void mbar_drain(uint64_t *b, uint32_t parity) {
  unsigned long long t0 = gtime();
  while (!mbar_try(b, parity) && gtime() - t0 < kWaitNs) {
  }
}
__device__ __forceinline__ void mbar_arrive(uint64_t *b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(s2u(b)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(s2u(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *b) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(s2u(dst)),
      "l"(src), "r"(bytes), "r"(s2u(b))
      : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: start address, leading (K) and stride
// (8-row) byte offsets, all >> 4; fixed version bits 46-47 = 1; no swizzle.
template <int KS>
__device__ __forceinline__ uint64_t smem_desc(const void *p) {
  uint64_t a = (uint64_t)((s2u(p) & 0x3FFFF) >> 4);
  return a | ((uint64_t)(kLBO >> 4) << 16) | ((uint64_t)(Shape<KS>::SBO >> 4) << 32) | (1ull << 46);
}
// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), BF16 A
// and B (bits 7-9 and 10-12 = 1), both K-major, N >> 3 at bit 17, M >> 4 at 24.
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTcN >> 3) << 17) |
                            ((uint32_t)(kTcM >> 4) << 24);

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(kIdesc), "r"(accumulate));
}
__device__ __forceinline__ void mma_commit(uint64_t *b) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(s2u(b))
               : "memory");
}
// 32 consecutive FP32 columns of this warp's 32 TMEM lanes (no wait).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float *v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
      "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),
        "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]),
        "=f"(v[16]), "=f"(v[17]), "=f"(v[18]), "=f"(v[19]), "=f"(v[20]), "=f"(v[21]), "=f"(v[22]), "=f"(v[23]),
        "=f"(v[24]), "=f"(v[25]), "=f"(v[26]), "=f"(v[27]), "=f"(v[28]), "=f"(v[29]), "=f"(v[30]), "=f"(v[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ---------------------------------------------------------------- operand preparation
__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// Error-free transformations (Knuth's TwoSum; the FMA product error).
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
  s = a + b;
  float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

// The centre c: mean of up to 2048 evenly spaced database rows, summed in a
// fixed order (one block of kCenterGroups x 33 threads), so it is the same on
// every run.
__global__ void k_center(const float *__restrict__ FQ, int nQ, float *__restrict__ c) {
  __shared__ float part[kCenterGroups][kD];
  const int col = threadIdx.x % kD, grp = threadIdx.x / kD;
  const int step = nQ > 2048 ? nQ / 2048 : 1;
  const int m = (nQ + step - 1) / step;  // sampled rows 0, step, 2 step, ...
  if (grp < kCenterGroups) {
    float s = 0.f;
    for (int i = grp; i < m; i += kCenterGroups) s += FQ[(size_t)i * step * kDS + col];
    part[grp][col] = s;
  }
  __syncthreads();
  if (threadIdx.x < kD) {
    float s = 0.f;
    for (int g = 0; g < kCenterGroups; ++g) s += part[g][threadIdx.x];
    c[threadIdx.x] = s / (float)m;
  }
}

struct PrepOut {
  char *tiles;
  float *aa;             // query side: |a~|^2 (rows padded to the unit size)
  float *eta;            // query side: |a - c - a~| bound
  unsigned *eta_max;     // database side: max |b - c - b~| bound (float bits)
  unsigned *bb_max;      // database side: max |b~|^2 (float bits)
};

// One thread per (padded) row of the order: centring, BF16 rounding (and
// split), the tile layout, |x~|^2 (compensated) and the rounding bound eta.
// Query rows lie one after another, database rows chunk-major per tile of 32;
// both have their bins in desc_order, which the contraction keeps (K columns
// may come in any order). Eight K columns of a row are one 16-byte store.
template <int KS, bool kQuery>
__global__ void k_prep_tiles(const float *__restrict__ F, int n, int rows, const float *__restrict__ c, PrepOut o) {
  using S = Shape<KS>;
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned eta_b = 0u, bb_b = 0u;
  if (r < rows) {
    char *base = o.tiles + (size_t)(r / kTcM) * S::TileBytes;
    const int rr = r % kTcM;
    const bool real = r < n;
    float h[kD], l[kD];
    float s_hi = 0.f, s_lo = 0.f, e2 = 0.f, x2 = 0.f;
    const float4 *src = kQuery ? reinterpret_cast<const float4 *>(F) + (size_t)r * (kDS / 4)
                               : reinterpret_cast<const float4 *>(F) + (size_t)(r / kOrdTile) * (9 * kOrdTile) + r % kOrdTile;
#pragma unroll
    for (int q = 0; q < kDS / 4; ++q) {
      const float4 v4 = real ? __ldg(src + q * (kQuery ? 1 : kOrdTile)) : make_float4(0.f, 0.f, 0.f, 0.f);
      const float v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int k = 4 * q + e;
        if (k >= kD) continue;
        const float x = real ? v[e] - __ldg(c + desc_order(k)) : 0.f;
        h[k] = bf16r(x);
        l[k] = S::kSplit ? bf16r(x - h[k]) : 0.f;  // x - h is exact
        const float xt = h[k] + l[k];              // exact (at most 16 significant bits)
        const float res = x - xt;                  // exact
        e2 = fmaf(res, res, e2);
        x2 = fmaf(x, x, x2);
        const float p = xt * xt, pe = fmaf(xt, xt, -p);
        float t, err;
        two_sum(s_hi, p, t, err);
        s_hi = t;
        s_lo += err + pe;
      }
    }
    float sq[3];
    if (kQuery) {
      sq[0] = sq[1] = sq[2] = 1.f;
    } else if (real) {
      const float p0 = bf16r(s_hi), r1 = s_hi - p0;  // exact
      const float p1 = bf16r(r1);
      sq[0] = p0, sq[1] = p1, sq[2] = bf16r((r1 - p1) + s_lo);
    } else {
      sq[0] = kPadScore, sq[1] = sq[2] = 0.f;
    }
    // column k of the operand (every value is a BF16 number)
    auto col = [&](int k) {
      if (k < kD) return kQuery ? -2.f * h[k] : h[k];
      if (S::kSplit && k < 2 * kD) return kQuery ? -2.f * l[k - kD] : h[k - kD];
      if (S::kSplit && k < 3 * kD) return kQuery ? -2.f * h[k - 2 * kD] : l[k - 2 * kD];
      if (k >= S::SqCol && k < S::SqCol + 3) return sq[k - S::SqCol];
      return 0.f;
    };
#pragma unroll
    for (int k = 0; k < S::K; k += 8) {
      unsigned w[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 p = __floats2bfloat162_rn(col(k + 2 * e), col(k + 2 * e + 1));
        w[e] = *reinterpret_cast<const unsigned *>(&p);
      }
      *reinterpret_cast<uint4 *>(base + tc_off<KS>(rr, k)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    // rounding of x~ plus the rounding of the centring (2^-24 |x| per component)
    const float eta = sqrtf(e2) * (1.f + 1e-5f) + 1.2e-7f * sqrtf(x2);
    if (kQuery) {
      o.aa[r] = s_hi + s_lo;
      o.eta[r] = eta;
    } else if (real) {
      eta_b = __float_as_uint(eta), bb_b = __float_as_uint(fmaxf(s_hi + s_lo, 0.f));
    }
  }
  if (!kQuery) {
    eta_b = __reduce_max_sync(0xffffffffu, eta_b), bb_b = __reduce_max_sync(0xffffffffu, bb_b);
    if ((threadIdx.x & 31) == 0) {
      atomicMax(o.eta_max, eta_b);
      atomicMax(o.bb_max, bb_b);
    }
  }
}

// Work items: unit u (of UnitQ queries) and the tiles 64 b + k of the set bits
// k of mask. Listed by size class (popcount) so that the largest come first;
// every class has room for all items.
constexpr int kItemTiles = 64, kClasses = 8;
struct TcItem {
  int u, b;
  unsigned long long mask;
};

// A block of 128 threads, one per query of a query tile; a warp's lanes first
// test 32 tiles' boxes against the query tile's box and largest published
// distance, then every query is tested against the boxes left. gridDim =
// (units, blocks of 64 tiles).
template <int QT>
__global__ void __launch_bounds__(QT * kTcM) k_tc_items(DescOrder o, int nP, int nQ,
                                                        const unsigned long long *__restrict__ packed, int cap,
                                                        TcItem *__restrict__ items, int *__restrict__ counts) {
  __shared__ unsigned s_far[QT];
  __shared__ unsigned s_open[QT][2], s_hit[2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, qt = warp >> 2;
  const int u = blockIdx.x, b = blockIdx.y;
  const int nt = (int)lsr_div_up(nQ, kTcN);
  const int q = u * QT * kTcM + threadIdx.x;
  const bool valid = q < nP;
  unsigned far = 0u;
  if (valid) {
    const unsigned long long pv = packed[q];
    far = pv == ~0ull ? __float_as_uint(FLT_MAX) : (unsigned)(pv >> 32);
  }
  const float best = __uint_as_float(far);
  if (threadIdx.x < QT) s_far[threadIdx.x] = 0u;
  if (threadIdx.x < 2) s_hit[threadIdx.x] = 0u;
  __syncthreads();
  far = __reduce_max_sync(0xffffffffu, far);
  if (lane == 0) atomicMax(&s_far[qt], far);
  __syncthreads();
  const float fac = o.pp->fac;
  // warps 0 and 1 of each query tile: 32 tiles each, a lane a tile
  if ((warp & 3) < 2) {
    const int t = b * kItemTiles + 32 * (warp & 3) + lane;
    const int leaf = u * QT + qt;
    bool open = t < nt && leaf * kTcM < nP;
    if (open) {
      float s = 0.f;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 tl = __ldg(o.lbox + 4 * (size_t)t + h), th = __ldg(o.lbox + 4 * (size_t)t + 2 + h);
        const float4 ql = __ldg(o.qbox + 4 * (size_t)leaf + h), qh = __ldg(o.qbox + 4 * (size_t)leaf + 2 + h);
        s = gap_add(s, fmaxf(__fsub_rd(tl.x, qh.x), __fsub_rd(ql.x, th.x)));
        s = gap_add(s, fmaxf(__fsub_rd(tl.y, qh.y), __fsub_rd(ql.y, th.y)));
        s = gap_add(s, fmaxf(__fsub_rd(tl.z, qh.z), __fsub_rd(ql.z, th.z)));
        s = gap_add(s, fmaxf(__fsub_rd(tl.w, qh.w), __fsub_rd(ql.w, th.w)));
      }
      open = !(__fmul_rd(s, fac) > __uint_as_float(s_far[qt]));
    }
    const unsigned m = __ballot_sync(0xffffffffu, open);
    if (lane == 0) s_open[qt][warp & 3] = m;
  }
  __syncthreads();
  unsigned long long todo = s_open[qt][0] | ((unsigned long long)s_open[qt][1] << 32);
  if (todo) {
    float p[kAx], e = 0.f;
    if (valid) {
      const float4 p0 = __ldg(o.qp + 2 * (size_t)q), p1 = __ldg(o.qp + 2 * (size_t)q + 1);
      p[0] = p0.x, p[1] = p0.y, p[2] = p0.z, p[3] = p0.w, p[4] = p1.x, p[5] = p1.y, p[6] = p1.z, p[7] = p1.w;
      e = __ldg(o.qe + q);
    }
    unsigned long long hit = 0ull;
    while (todo) {
      const int k = __ffsll(todo) - 1;
      todo &= todo - 1;
      bool reach = false;
      if (valid) {
        const float4 *box = o.lbox + 4 * ((size_t)b * kItemTiles + k);
        const float4 l0 = __ldg(box), l1 = __ldg(box + 1), h0 = __ldg(box + 2), h1 = __ldg(box + 3);
        const float lo[kAx] = {l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z, l1.w};
        const float hi[kAx] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
        float s = 0.f;
#pragma unroll
        for (int d = 0; d < kAx; ++d)
          s = gap_add(s, __fsub_rd(fmaxf(__fsub_rd(lo[d], p[d]), __fsub_rd(p[d], hi[d])), e));
        reach = !(__fmul_rd(s, fac) > best);
      }
      if (__any_sync(0xffffffffu, reach)) hit |= 1ull << k;
    }
    if (lane == 0 && hit) {
      if ((unsigned)hit) atomicOr(&s_hit[0], (unsigned)hit);
      if ((unsigned)(hit >> 32)) atomicOr(&s_hit[1], (unsigned)(hit >> 32));
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned long long m = s_hit[0] | ((unsigned long long)s_hit[1] << 32);
    if (m) {
      const int cls = (kItemTiles - __popcll(m)) / (kItemTiles / kClasses);  // 0: 57 to 64 tiles
      items[(size_t)cls * cap + atomicAdd(counts + cls, 1)] = TcItem{u, b, m};
    }
  }
}

struct TcArgs {
  const char *A, *B;            // query units and database tiles (BF16, MMA layout)
  const float *aa, *eta_a;      // per query position
  const unsigned *eta_b, *bb;   // database maxima (float bits)
  const float *FPs, *FQs;       // FP32 descriptors in the order for the re-rank (bins in desc_order)
  const int *dorig;             // original index of a database position
  int nP, nQ, nU, nNT;
  const TcItem *items;          // kClasses lists of item_cap items; null: every unit with every tile
  const int *item_counts;
  int item_cap;
  unsigned long long *packed;   // per query position: best (distance bits << 32 | original index)
  const int *qorig;             // original index of a query position
  int *fb_flag;                 // per query position, then per group of 32: already listed
  int *fb_rows, *fb_count;      // queries (original index) left to the exact FP32 search
  int *fb_groups, *fb_ngroups;  // and their groups
  int *err;                     // set to 1 by a CTA that gave up
  float *d2;                    // optional: all D~^2 = s + |a~|^2 (nP x nNT * kTcN) instead of matching
  unsigned long long wait_ns;   // limit of every wait of the pipeline (the drain after a failure keeps kWaitNs)
  int stall;                    // fault injection: the producer issues nothing, so the first wait runs out
};

// The items of one CTA, one after another, and an item's tiles. The producer
// runs two of these (copies ahead of MMAs), every epilogue thread one.
struct ItemIter {
  long long i;                  // next item of this CTA
  unsigned long long mask = 0ull;
  int u = 0, b = 0;
  __device__ __forceinline__ explicit ItemIter(int first) : i(first) {}
  // Moves to the next item; false when there is none.
  __device__ __forceinline__ bool next_item(const TcArgs &g) {
    if (g.items) {
      long long k = i;
      for (int c = 0; c < kClasses; ++c) {
        const int n = __ldg(g.item_counts + c);
        if (k < n) {
          const int4 v = __ldg(reinterpret_cast<const int4 *>(g.items + (size_t)c * g.item_cap + k));
          u = v.x, b = v.y;
          mask = (unsigned)v.z | ((unsigned long long)(unsigned)v.w << 32);
          i += gridDim.x;
          return true;
        }
        k -= n;
      }
      return false;
    }
    const int nb = (g.nNT + kItemTiles - 1) / kItemTiles;
    if (i >= (long long)g.nU * nb) return false;
    u = (int)(i / nb), b = (int)(i - (long long)u * nb);
    const int left = g.nNT - b * kItemTiles;
    mask = left >= kItemTiles ? ~0ull : (1ull << left) - 1ull;
    i += gridDim.x;
    return true;
  }
  // The next tile of the current item (mask != 0).
  __device__ __forceinline__ int next_tile() {
    const int k = __ffsll((long long)mask) - 1;
    mask &= mask - 1;
    return b * kItemTiles + k;
  }
};
static_assert(sizeof(TcItem) == 16, "an item is one 16-byte load");

// Exact FP32 squared distance in the FP32 matcher's operation order (one
// fused multiply-add per bin, bins in desc_order on both sides) to row j of a
// tile of 32 (chunk-major: chunk c at T4[c * 32 + j]).
__device__ __forceinline__ float exact_d2(const float (&a)[kD], const float4 *__restrict__ T4, int j) {
  float r[36];
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    const float4 x = __ldg(T4 + q * kOrdTile + j);
    r[4 * q] = x.x, r[4 * q + 1] = x.y, r[4 * q + 2] = x.z, r[4 * q + 3] = x.w;
  }
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < kD; ++k) {
    float t = a[k] - r[k];
    s = fmaf(t, t, s);
  }
  return s;
}

__device__ __forceinline__ void top8_insert(float (&ts)[kTopK], int (&ti)[kTopK], float v, int id) {
  if (!(v < ts[kTopK - 1])) return;
  ts[kTopK - 1] = v;
  ti[kTopK - 1] = id;
#pragma unroll
  for (int q = kTopK - 1; q > 0; --q)
    if (ts[q] < ts[q - 1]) {
      float a = ts[q];
      ts[q] = ts[q - 1];
      ts[q - 1] = a;
      int b = ti[q];
      ti[q] = ti[q - 1];
      ti[q - 1] = b;
    }
}

template <int KS, int QT>
__global__ void __launch_bounds__(Cfg<KS, QT>::Threads, Cfg<KS, QT>::CtasPerSm) k_match_tc(TcArgs g) {
  using S = Shape<KS>;
  using C = Cfg<KS, QT>;
  constexpr int kStages = C::Stages, kEpiWarps = C::EpiWarps, kUnitQ = C::UnitQ;
  constexpr uint32_t kAccCols = C::AccCols, kTmemCols = C::TmemCols;
  extern __shared__ __align__(128) unsigned char smem[];
  char *sA = reinterpret_cast<char *>(smem);
  char *sB = sA + C::UnitBytes;
  uint64_t *bars = reinterpret_cast<uint64_t *>(sB + kStages * S::TileBytes);
  uint64_t *barA = bars;                 // 1
  uint64_t *barB = bars + 1;             // kStages
  uint64_t *barDone = barB + kStages;    // 2: accumulator buffer written
  uint64_t *barEmpty = barDone + 2;      // 2: accumulator buffer drained
  uint32_t *tslot = reinterpret_cast<uint32_t *>(barEmpty + 2);
  volatile int *fail = reinterpret_cast<volatile int *>(tslot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    mbar_init(barA, 1);
    for (int s = 0; s < kStages; ++s) mbar_init(barB + s, 1);
    for (int s = 0; s < 2; ++s) mbar_init(barDone + s, 1), mbar_init(barEmpty + s, kEpiWarps);
    *fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kEpiWarps) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s2u(tslot)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = *tslot;

  // producer state, kept for the clean-up after a failure
  int loaded[kStages];
  int last_commit = -1, a_pending = -1;
  for (int s = 0; s < kStages; ++s) loaded[s] = -1;

  if (warp == kEpiWarps) {
    // ------------------------------------------------ copies + MMA (one thread)
    if (lane == 0 && !g.stall) {
      ItemIter ahead(blockIdx.x), at(blockIdx.x);
      bool more = ahead.next_item(g);
      int jl = 0;  // copies issued
      auto load_b = [&]() {
        const int st = jl % kStages, t = ahead.next_tile();
        if (!ahead.mask) more = ahead.next_item(g);
        mbar_expect_tx(barB + st, S::TileBytes);
        bulk_g2s(sB + st * S::TileBytes, g.B + (size_t)t * S::TileBytes, S::TileBytes, barB + st);
        loaded[st] = jl++;
      };
      while (more && jl < kStages) load_b();
      int items = 0, j = 0;
      bool ok = true;
      while (ok && at.next_item(g)) {
        // the previous item's MMAs must be done reading the query tiles
        if (j > 0 && !mbar_wait(barDone + ((j - 1) & 1), ((j - 1) >> 1) & 1, fail, g.wait_ns)) break;
        mbar_expect_tx(barA, C::UnitBytes);
        bulk_g2s(sA, g.A + (size_t)at.u * C::UnitBytes, C::UnitBytes, barA);
        a_pending = items & 1;
        if (!mbar_wait(barA, items & 1, fail, g.wait_ns)) break;
        a_pending = -1;
        ++items;
        for (; at.mask; ++j) {
          at.next_tile();
          const int st = j % kStages;
          ok = mbar_wait(barB + st, (j / kStages) & 1, fail, g.wait_ns);
          if (!ok) break;
          loaded[st] = -1;
          ok = j < 2 || mbar_wait(barEmpty + (j & 1), ((j - 2) >> 1) & 1, fail, g.wait_ns);
          if (!ok) break;
          tc_fence_after();
          const uint32_t d = tbase + (uint32_t)((j & 1) * kAccCols);
#pragma unroll
          for (int qt = 0; qt < QT; ++qt)
#pragma unroll
            for (int k = 0; k < KS; ++k)
              mma_bf16(d + qt * kTcN, smem_desc<KS>(sA + qt * S::TileBytes + k * 2 * kLBO),
                       smem_desc<KS>(sB + st * S::TileBytes + k * 2 * kLBO), k > 0 ? 1u : 0u);
          mma_commit(barDone + (j & 1));
          last_commit = j;
          // refill the stage of step j-1 once its MMAs are done
          if (j >= 1 && more) {
            ok = mbar_wait(barDone + ((j - 1) & 1), ((j - 1) >> 1) & 1, fail, g.wait_ns);
            if (!ok) break;
            load_b();
          }
        }
      }
    }
  } else {
    // ------------------------------------------------ epilogue: one query per thread
    const int qt = warp >> 2;
    const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
    const int row_in_unit = qt * kTcM + 32 * (warp & 3) + lane;
    const int ncols = g.nNT * kTcN;
    int j = 0;
    bool ok = true;
    ItemIter it(blockIdx.x);
    while (ok && it.next_item(g)) {
      const int r = it.u * kUnitQ + row_in_unit;
      const bool many = __popcll(it.mask) > 1;  // more chunks than are kept
      float ts[kTopK];
      int ti[kTopK];
#pragma unroll
      for (int q = 0; q < kTopK; ++q) ts[q] = FLT_MAX, ti[q] = -1;
      for (; it.mask; ++j) {
        const int t = it.next_tile();
        const int buf = j & 1;
        ok = mbar_wait(barDone + buf, (j >> 1) & 1, fail, g.wait_ns);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        // the whole row of the accumulator with one wait
        const uint32_t row = tbase + lane_base + (uint32_t)(buf * kAccCols + qt * kTcN);
        float v[kTcN];
        __syncwarp();  // the loads below are warp-collective
#pragma unroll
        for (int q = 0; q < kLoads; ++q) tmem_ld32(row + q * 32, v + q * 32);
        tmem_wait_ld();
        const int c0 = t * kTcN;
        // the scores are in registers: the buffer goes back to the MMA at once
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(barEmpty + buf);
        if (g.d2) {
          if (r < g.nP) {
            const float aa = g.aa[r];
            for (int k = 0; k < kTcN; ++k) g.d2[(size_t)r * ncols + c0 + k] = v[k] + aa;
          }
          continue;
        }
        // minimum of each chunk; the 8 smallest chunk minima are kept
#pragma unroll
        for (int q = 0; q < kChunks; ++q) {
          const float *w = v + q * kChunkW;
          float a0 = w[0], a1 = w[1], a2 = w[2], a3 = w[3];
#pragma unroll
          for (int k = 4; k < kChunkW; k += 4) {
            a0 = fminf(a0, w[k]), a1 = fminf(a1, w[k + 1]);
            a2 = fminf(a2, w[k + 2]), a3 = fminf(a3, w[k + 3]);
          }
          top8_insert(ts, ti, fminf(fminf(a0, a1), fminf(a2, a3)), t * kChunks + q);
        }
      }
      if (!ok || g.d2 || r >= g.nP) continue;
      // exact FP32 re-rank of the candidate chunks that can hold a row at or
      // below the query's best distance (its own items' or another's)
      const float aa = g.aa[r], bbm = __uint_as_float(*g.bb);
      const float na = sqrtf(aa), nb = sqrtf(bbm);
      // accumulation (sum |products| <= 2.05 |a~||b~| + |b~|^2) and, split
      // layout, the left-out 2 l_a.l_b (<= 2^-15 |a~||b~|)
      const float efp = kAccErr * (2.05f * na * nb + bbm) + (S::kSplit ? 3.1e-5f * na * nb : 0.f);
      const float eta = g.eta_a[r] + __uint_as_float(*g.eta_b);
      const unsigned long long pv = __ldcg(g.packed + r);
      float best = pv == ~0ull ? FLT_MAX : __uint_as_float((unsigned)(pv >> 32));
      int bi = -1;
      // no row of a chunk of minimum m is at or below best (a computed
      // distance is >= (1 - 35 * 2^-24) of the true one); false for NaN
      auto beyond = [&](float m) {
        return sqrtf(fmaxf(m + aa - efp, 0.f)) - eta > sqrtf(best) * (1.f + 1e-5f);
      };
      // an item has at least 8 chunks: one fewer kept had a minimum that is no
      // finite number, and proves nothing
      const bool all = ti[kTopK - 1] >= 0;
      bool cert = false;
      float a[kD];
      {
        const float4 *row = reinterpret_cast<const float4 *>(g.FPs + (size_t)r * kDS);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const float4 x = __ldg(row + c);
          a[4 * c] = x.x, a[4 * c + 1] = x.y, a[4 * c + 2] = x.z, a[4 * c + 3] = x.w;
        }
        a[32] = __ldg(reinterpret_cast<const float *>(row + 8));
      }
#pragma unroll 1
      for (int q = 0; q < kTopK; ++q) {
        if (ti[0] < 0) break;
        if (beyond(ts[0])) {
          cert = all;
          break;
        }
        const int c0 = ti[0] * kChunkW, c1 = min(g.nQ, c0 + kChunkW);
        const float4 *T4 = reinterpret_cast<const float4 *>(g.FQs) + (size_t)(c0 / kOrdTile) * (9 * kOrdTile);
#pragma unroll 1
        for (int c = c0; c < c1; ++c) {
          if (!LSR_IN_BOUNDS(c, g.nQ, kSiteMatchRow)) break;
          const float d = exact_d2(a, T4, c % kOrdTile);
          if (d <= best) {
            const int id = __ldg(g.dorig + c);
            if (d < best || bi < 0 || id < bi) best = d, bi = id;
          }
        }
        const float t0 = ts[0];
#pragma unroll
        for (int k = 0; k + 1 < kTopK; ++k) ts[k] = ts[k + 1], ti[k] = ti[k + 1];
        ts[kTopK - 1] = t0;  // the last one looked at, kept for the certificate
      }
      // all eight within reach: the chunks left out are no nearer than the eighth
      if (!cert) cert = all && (!many || beyond(ts[kTopK - 1]));
      if (bi >= 0) atomicMin(g.packed + r, ((unsigned long long)__float_as_uint(best) << 32) | (unsigned)bi);
      if (!cert && atomicExch(g.fb_flag + r, 1) == 0) {
        const int slot = atomicAdd(g.fb_count, 1);
        if (LSR_IN_BOUNDS(slot, g.nP, kSiteMatchQuery)) g.fb_rows[slot] = g.qorig[r];
        const int gr = r / kOrdTile;
        if (atomicExch(g.fb_flag + g.nP + gr, 1) == 0) g.fb_groups[atomicAdd(g.fb_ngroups, 1)] = gr;
      }
    }
  }

  // teardown: every epilogue warp has finished its TMEM reads
  tc_fence_before();
  __syncthreads();
  if (warp == kEpiWarps) {
    if (lane == 0 && *fail) {
      // a wait gave up: nothing may still write TMEM or shared memory
      if (last_commit >= 0) mbar_drain(barDone + (last_commit & 1), (last_commit >> 1) & 1);
      for (int s = 0; s < kStages; ++s)
        if (loaded[s] >= 0) mbar_drain(barB + s, (loaded[s] / kStages) & 1);
      if (a_pending >= 0) mbar_drain(barA, (uint32_t)a_pending);
      atomicExch(g.err, 1);
    }
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(kTmemCols));
  }
}

constexpr int kCounters = 2 + kClasses + 1;
struct TcLayout {
  DescOrder o;
  char *A = nullptr, *B = nullptr;
  float *aa = nullptr, *eta = nullptr, *center = nullptr;
  unsigned *maxes = nullptr;      // eta_b, bb, the kClasses item counts, the number of listed groups
  int *fb_flag = nullptr, *fb_rows = nullptr, *fb_groups = nullptr;
  unsigned long long *fb_work = nullptr;
  unsigned long long *packed = nullptr, *fb_packed = nullptr;
  TcItem *items = nullptr;
  int item_cap = 0;               // 0: no item list (all tiles)
  size_t bytes = 0;
};

// Whether the order and the item list pay. The order and the first pass cost
// about 0.15 ms at any size; the contraction over all tiles 0.2 ps a pair of
// rows (8.5 ms for 4e10), of which the list leaves a tenth to a fifth. Whole
// calls on room descriptors, all tiles against listed ones: 8k x 8k 289 and 413
// us, 16k 350 and 467, 20k 471 and 511, 23k (about where the line lies) 479 and
// 520, 28k 533 and 525.
// Above 2^22 items (about 2M x 2M rows) the list would outgrow its use of memory.
constexpr int64_t kWindowPairs = (int64_t)1 << 29;
constexpr int64_t kMaxItems = (int64_t)1 << 22;
int item_cap_for(int nP, int nQ, bool list) {
  if (!list && (int64_t)nP * nQ < kWindowPairs) return 0;
  const int64_t n = lsr_div_up(nP, kTcM) * lsr_div_up(lsr_div_up(nQ, kTcN), kItemTiles);
  return n <= kMaxItems ? (int)n : 0;
}

// Query rows are padded to a multiple of 256 (a whole number of units for
// either tile shape); unit u of shape QT is tiles QT u .. QT u + QT - 1.
template <int KS>
TcLayout tc_layout(char *base, int nP, int nQ, bool list) {
  using S = Shape<KS>;
  auto al = [](size_t x) { return (x + 255) / 256 * 256; };
  size_t tilesA = 2 * (size_t)lsr_div_up(nP, 2 * kTcM), nNT = (size_t)lsr_div_up(nQ, kTcN);
  size_t rowsA = tilesA * kTcM;
  TcLayout L;
  size_t off = desc_order_layout(base, nP, nQ, L.o);
  auto take = [&](size_t bytes) {
    char *p = base ? base + off : nullptr;
    off += al(bytes);
    return p;
  };
  L.A = take(tilesA * S::TileBytes);
  L.B = take(nNT * S::TileBytes);
  L.aa = reinterpret_cast<float *>(take(rowsA * 4));
  L.eta = reinterpret_cast<float *>(take(rowsA * 4));
  L.center = reinterpret_cast<float *>(take(kD * 4));
  const size_t groups = (size_t)lsr_div_up(nP, kOrdTile);
  L.maxes = reinterpret_cast<unsigned *>(take(kCounters * 4));
  L.fb_work = reinterpret_cast<unsigned long long *>(take(8));
  L.fb_flag = reinterpret_cast<int *>(take(((size_t)nP + groups) * 4));
  L.fb_groups = reinterpret_cast<int *>(take(groups * 4));
  L.fb_rows = reinterpret_cast<int *>(take((size_t)nP * 4));
  L.packed = reinterpret_cast<unsigned long long *>(take((size_t)nP * 8));
  L.fb_packed = reinterpret_cast<unsigned long long *>(take((size_t)nP * 8));
  L.item_cap = item_cap_for(nP, nQ, list);
  L.items = reinterpret_cast<TcItem *>(take(sizeof(TcItem) * (size_t)L.item_cap * kClasses));
  L.bytes = off;
  return L;
}

int sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return 148;
  }
  return n > 0 ? n : 148;
}

template <int KS, int QT>
cudaError_t launch_tc(const TcLayout &L, int nP, int nQ, bool window, int *fb_count, int *err, float *d2,
                      const TcFault &f, cudaStream_t s) {
  using C = Cfg<KS, QT>;
  const int nU = (int)lsr_div_up(nP, C::UnitQ), nNT = (int)lsr_div_up(nQ, kTcN);
  const int nb = (int)lsr_div_up(nNT, kItemTiles);
  int *counts = reinterpret_cast<int *>(L.maxes + 2);
  if (window)
    LSR_LAUNCH(k_tc_items<QT><<<dim3(nU, nb), C::UnitQ, 0, s>>>(L.o, nP, nQ, L.packed, L.item_cap, L.items, counts));
  LSR_CUDA_TRY(cudaFuncSetAttribute(k_match_tc<KS, QT>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SmemBytes));
  TcArgs g{L.A, L.B, L.aa, L.eta, L.maxes, L.maxes + 1, L.o.FPs, L.o.FQs, L.o.dorig, nP, nQ, nU, nNT,
           window ? L.items : nullptr, counts, L.item_cap, L.packed, L.o.qorig, L.fb_flag, L.fb_rows, fb_count,
           L.fb_groups, counts + kClasses, err,
           d2, f.wait_ns ? f.wait_ns : kWaitNs, f.stall};
  const int64_t slots = (int64_t)sm_count() * C::CtasPerSm, items = (int64_t)nU * nb;
  const int grid = (int)(items < slots ? items : slots);
  LSR_LAUNCH(k_match_tc<KS, QT><<<grid, C::Threads, C::SmemBytes, s>>>(g));
  return cudaGetLastError();
}

template <int KS>
cudaError_t run_tc(const float *FP, int nP, const float *FQ, int nQ, int qt, char *ws, int *nn, float *d1,
                   int *fb_count, int *err, float *d2, const TcFault &f, cudaStream_t s) {
  TcLayout L = tc_layout<KS>(ws, nP, nQ, f.list != 0);
  const int nNT = (int)lsr_div_up(nQ, kTcN);
  const bool window = L.item_cap > 0 && !d2;
  // the counters, the search's work word and the flags lie one after another
  LSR_CUDA_TRY(cudaMemsetAsync(L.maxes, 0, (char *)(L.fb_flag + nP + lsr_div_up(nP, kOrdTile)) - (char *)L.maxes, s));
  LSR_CUDA_TRY(cudaMemsetAsync(L.packed, 0xFF, sizeof(unsigned long long) * (size_t)nP, s));
  LSR_CUDA_TRY(cudaMemsetAsync(fb_count, 0, sizeof(int), s));
  LSR_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int), s));
  LSR_LAUNCH(k_center<<<1, kCenterGroups * kD, 0, s>>>(FQ, nQ, L.center));
  if (window) {
    LSR_CUDA_TRY(launch_desc_order(FP, nP, FQ, nQ, L.o, s));
    LSR_CUDA_TRY(launch_match_seed(L.o, nP, nQ, L.packed, s));
  } else {
    LSR_CUDA_TRY(launch_desc_rows(FP, nP, FQ, nQ, L.o, s));
  }
  const int rowsA = 2 * (int)lsr_div_up(nP, 2 * kTcM) * kTcM, rowsB = nNT * kTcN;
  PrepOut pa{L.A, L.aa, L.eta, nullptr, nullptr};
  PrepOut pb{L.B, nullptr, nullptr, L.maxes, L.maxes + 1};
  LSR_LAUNCH(k_prep_tiles<KS, true><<<(int)lsr_div_up(rowsA, 128), 128, 0, s>>>(L.o.FPs, nP, rowsA, L.center, pa));
  LSR_LAUNCH(k_prep_tiles<KS, false><<<(int)lsr_div_up(rowsB, 128), 128, 0, s>>>(L.o.FQs, nQ, rowsB, L.center, pb));
  if (qt == 1)
    LSR_CUDA_TRY((launch_tc<KS, 1>(L, nP, nQ, window, fb_count, err, d2, f, s)));
  else
    LSR_CUDA_TRY((launch_tc<KS, 2>(L, nP, nQ, window, fb_count, err, d2, f, s)));
  if (!d2) {
    // the queries without a certificate: through the boxes where there are any
    if (window)
      LSR_CUDA_TRY(launch_match_listed(L.o, nP, nQ, L.fb_groups, reinterpret_cast<int *>(L.maxes + 2 + kClasses),
                                       L.fb_flag, L.packed, L.fb_work, s));
    LSR_CUDA_TRY(launch_match_finish(L.packed, L.o.qorig, nP, nn, d1, s));
    if (!window)
      LSR_CUDA_TRY(launch_match_fp32_rows(FP, nP, FQ, nQ, L.fb_rows, fb_count, L.fb_packed, nn, d1, s));
  }
  return cudaGetLastError();
}

constexpr int kKsPlain = 3, kKsSplit = 7;

}  // namespace

LSR_CHECK_READER(match_tc)

size_t tc_workspace_bytes(int nP, int nQ, bool split, bool list) {
  return split ? tc_layout<kKsSplit>(nullptr, nP, nQ, list).bytes : tc_layout<kKsPlain>(nullptr, nP, nQ, list).bytes;
}

int tc_score_cols(int nQ) { return (int)lsr_div_up(nQ, kTcN) * kTcN; }

// One query tile per CTA (two CTAs per SM) unless the autotuner chose for the
// size: on the 150k-point room pair (its listed tiles) it takes 0.64 ms against
// 0.84 ms with two query tiles per CTA (one CTA per SM); a whole match of 200k x
// 200k room descriptors 1.93 ms against 2.29.
int tc_default_tile(int) { return 1; }

cudaError_t launch_match_bf16(const float *FP, int nP, const float *FQ, int nQ, bool split, int qt, char *ws, int *nn,
                              float *d1, int *fb_count, int *err, float *d2, cudaStream_t s, TcFault f) {
  if (nP < 1 || nQ < 1 || (qt != 0 && qt != 1 && qt != 2)) return cudaErrorInvalidValue;
  if (qt == 0) qt = tc_default_tile(nP);
  return split ? run_tc<kKsSplit>(FP, nP, FQ, nQ, qt, ws, nn, d1, fb_count, err, d2, f, s)
               : run_tc<kKsPlain>(FP, nP, FQ, nQ, qt, ws, nn, d1, fb_count, err, d2, f, s);
}

int device_sm_count() { return sm_count(); }

}  // namespace lsr
