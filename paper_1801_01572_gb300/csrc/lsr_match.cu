// lsr_match.cu -- feature pre-matching cache on the FP32 cores (Algorithm 1,
// "Parallel FPFH feature pre-matching": nn[i] = NN of F(p_i) in F(Q)).
//
// Exact: nn[i] = argmin_j sum_k (a_k - b_k)^2 with ties to the smallest j,
// each distance accumulated as s = fma(t, t, s) over the 33 bins taken in
// desc_order (central bins first). What is exact is the result; the search
// visits only the database rows that could change it.
//
// Projection boxes. Both sets are projected on the first kAx principal axes of
// a sample of the database (any axes give the same result, good ones visit
// fewer rows) and ordered so that kTile consecutive rows lie close together in
// that space (lsr_order.cu). For the stored FP32 axes U, |U^T (a - b)|^2 <=
// lambda |a - b|^2 with lambda bounding the Gram matrix's largest eigenvalue,
// so a row whose projections lie farther than sqrt(lambda * best) from the
// query's cannot be nearer than the current best. A warp takes a group of 32
// consecutive queries. A first pass scans the two leaves (128 rows) nearest to
// the group, which already gives distances close to the final ones (a replay
// on room descriptors: 11.5% of the tiles of 128 within their reach, 10.7%
// within the nearest rows'). The second pass takes items of one group and 32
// tiles from a counter: a lane tests a tile's box against the group's, then
// the tiles left are tested query by query and scanned if any query can find a
// nearer row there. Best distances are shared between the warps of a group by
// a 64-bit atomic minimum of (distance, index). The FP32 rounding of the
// projections (a bound per row from the error of an fma chain), of the axes
// and of the distance itself is taken into the test by directed rounding, so a
// row or a tile is left out only when every computed distance in it exceeds a
// distance some row has: the nearest row and its ties are always scanned, and
// ties go to the smaller original index whatever the scan order.
//
// Eight axes and a k-d order instead of two axes in slabs of 1024 rows: of the
// definition's 7.4e11 terms (150k x 150k room descriptors) 1.5e10 are evaluated
// instead of 3.9e10, and the match takes 3.4 ms instead of 7.5; 60k x 90k 1.81
// ms instead of 2.42 (the whole call); 5k x 5k 0.26 ms instead of 0.86.
//
// Each lane keeps one query descriptor in registers; a warp copies the tiles
// that it is going to scan to shared memory one ahead (asynchronous copies) and
// reads their rows as broadcasts. Rows go eight at a time: the first eight
// terms (bins in desc_order) of all eight without a branch, then, for the rows
// that some lane still wants, the rest. The partial sums only grow (t^2 >= 0
// and rounding is monotone), so a row whose partial sum already exceeds every
// query's current best in the warp can neither win nor tie: after 8, 16 and 24
// terms the warp tests that and skips the rest of the row (same result).
// Reading rows through L1 instead, one at a time with a test after every four
// terms, was a chain of dependent loads: 6.7 ms at 150k x 150k for the same
// tiles. The listed-rows scan of the tensor-core path's exact fallback
// (k_match_rows_chunked) stages tiles in shared memory too.
#include <float.h>
#include <stddef.h>

#include <algorithm>

#include "lsr_internal.cuh"

namespace lsr {

namespace {

constexpr int kMT = 128;   // threads per block
constexpr int kQR = 2;     // queries per thread, listed rows (k_match_rows_chunked)
constexpr int kTile = 32;  // database rows per tile (32 measured faster than 64 or 128 in the window search)
constexpr int kStageThreads = 9 * (kMT / 9);  // staging threads: one float4 column each
static_assert(kTile * 9 > kStageThreads, "staging covers the tile in several passes");
static_assert(kTile == kOrdTile, "the search scans the tiles of the order");
constexpr int kMatchBlocks = 5;      // resident blocks per SM: 41 KB of shared memory each
constexpr int kSeedLeaves = 2;       // leaves a group scans first

// Database rows [base, base + kTile) (zero past lim) into the tile, bin
// desc_order(k) at slot k and zeros at slots 33..35. Thread t < kStageThreads
// copies float4 column t % 9 of rows t / 9, t / 9 + kMT / 9, ...; rk holds the
// slots of that column's four bins (-1 past the descriptor).
__device__ __forceinline__ void stage_tile(float4 (*tile)[9], const float *__restrict__ FQ, int base, int lim,
                                           const int (&rk)[4]) {
  if (threadIdx.x >= kStageThreads) return;
  float *tf = reinterpret_cast<float *>(tile);
  const int c = threadIdx.x % 9;
  for (int r = threadIdx.x / 9; r < kTile; r += kMT / 9) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (base + r < lim) v = reinterpret_cast<const float4 *>(FQ + (size_t)(base + r) * kDS)[c];
    float *row = tf + r * 36;
    row[rk[0]] = v.x;
    if (rk[1] >= 0) {
      row[rk[1]] = v.y, row[rk[2]] = v.z, row[rk[3]] = v.w;
    } else {
      row[33] = 0.f, row[34] = 0.f, row[35] = 0.f;
    }
  }
}

__device__ __forceinline__ void stage_ranks(int (&rk)[4]) {
  const int c = threadIdx.x % 9;
#pragma unroll
  for (int i = 0; i < 4; ++i) rk[i] = 4 * c + i < kD ? desc_rank(4 * c + i) : -1;
}

// Scan the m staged rows for the Q queries of this thread (a in
// desc_order), updating best / bj; row j of the tile is database row base + j.
// A row replaces the best when its distance is smaller, or equal with a smaller
// index, so the result does not depend on the order in which rows are scanned.
template <int Q>
__device__ __forceinline__ void scan_tile(const float4 (*tile)[9], int m, int base, const float (&a)[Q][kD],
                                          float (&best)[Q], int (&bj)[Q]) {
  for (int j = 0; j < m; ++j) {
    float s[Q];
#pragma unroll
    for (int u = 0; u < Q; ++u) s[u] = 0.f;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      if (c >= 1 && (c <= 4 || c == 6)) {
        bool past = true;
#pragma unroll
        for (int u = 0; u < Q; ++u) past &= s[u] > best[u];
        if (__all_sync(0xffffffffu, past)) break;
      }
      float4 b = tile[j][c];
#pragma unroll
      for (int u = 0; u < Q; ++u) {
        float t0 = a[u][4 * c] - b.x, t1 = a[u][4 * c + 1] - b.y, t2 = a[u][4 * c + 2] - b.z,
              t3 = a[u][4 * c + 3] - b.w;
        s[u] = fmaf(t0, t0, s[u]);
        s[u] = fmaf(t1, t1, s[u]);
        s[u] = fmaf(t2, t2, s[u]);
        s[u] = fmaf(t3, t3, s[u]);
      }
      if (c == 7) {
        float b32 = tile[j][8].x;
        const int id = base + j;
#pragma unroll
        for (int u = 0; u < Q; ++u) {
          float t = a[u][32] - b32;
          s[u] = fmaf(t, t, s[u]);
          if (s[u] < best[u] || (s[u] == best[u] && id < bj[u])) best[u] = s[u], bj[u] = id;
        }
      }
    }
  }
}

// Asynchronous copy of a database tile (kOrdTile x kDS floats, chunk-major:
// float4 chunk c of row j at c * kTile + j) to this warp's buffer.
constexpr int kTileV = 9 * kTile;  // float4 of a tile
__device__ __forceinline__ void stage_async(float4 *buf, const float4 *__restrict__ src) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int u = 0; u < kTileV / 32; ++u)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(buf + 32 * u + lane)),
                 "l"(src + 32 * u + lane)
                 : "memory");
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void stage_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
  __syncwarp();
}

// Scan the m rows of a staged tile for this lane's query a. best is the lane's
// pruning bound (its own best or a smaller one another warp published); a row
// is taken when its distance is smaller, or equal with a smaller index than a
// row already taken (bj = -2: the bound came from elsewhere, so an equal row is
// taken and the atomic minimum of the published pairs decides); taken marks
// that there is a pair to publish.
template <bool kCount>
__device__ __forceinline__ void scan_rows(const float4 *__restrict__ T4, const int *__restrict__ ids, int m,
                                          const float (&a)[kD], float &best, int &bj, bool &taken, unsigned &terms) {
  constexpr int kR = 8;
  auto add = [](float s, float x, float y) {
    const float t = x - y;
    return fmaf(t, t, s);
  };
#pragma unroll 1
  for (int j0 = 0; j0 < m; j0 += kR) {
    float s[kR];
    unsigned live = 0u;
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      const float4 b0 = T4[j0 + r], b1 = T4[kTile + j0 + r];
      float v = add(0.f, a[0], b0.x);
      v = add(v, a[1], b0.y), v = add(v, a[2], b0.z), v = add(v, a[3], b0.w);
      v = add(v, a[4], b1.x), v = add(v, a[5], b1.y), v = add(v, a[6], b1.z), v = add(v, a[7], b1.w);
      s[r] = v;
      if (__any_sync(0xffffffffu, !(v > best))) live |= 1u << r;
    }
    if (m - j0 < kR) live &= (1u << (m - j0)) - 1u;
    if (kCount) terms += 8 * min(m - j0, kR);
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      if (!((live >> r) & 1u)) continue;
      float v = s[r];
      bool past = false;
#pragma unroll
      for (int c = 2; c < 8; ++c) {
        if (c == 2 || c == 4 || c == 6) {
          past = __all_sync(0xffffffffu, v > best);  // (best may have fallen since the row was found live)
          if (past) break;
        }
        const float4 b = T4[c * kTile + j0 + r];
        v = add(v, a[4 * c], b.x), v = add(v, a[4 * c + 1], b.y);
        v = add(v, a[4 * c + 2], b.z), v = add(v, a[4 * c + 3], b.w);
        if (kCount) terms += c == 7 ? 5 : 4;
      }
      if (past) continue;
      v = add(v, a[32], reinterpret_cast<const float *>(T4 + 8 * kTile + j0 + r)[0]);
      if (v < best || (v == best && bj != -1)) {
        const int id = __ldg(ids + j0 + r);
        if (v < best || (unsigned)id < (unsigned)bj) best = v, bj = id, taken = true;
      }
    }
  }
}

__device__ __forceinline__ unsigned long long pack_pair(float d, int j) {
  return ((unsigned long long)__float_as_uint(d) << 32) | (unsigned)j;
}

// The queries of a group (a lane each): descriptor, projections, pruning state.
struct QueryLane {
  float a[kD];
  float e;       // error bound of the projections
  float best;
  int bj;
  bool valid, taken;
};

__device__ __forceinline__ void load_query(QueryLane &q, const DescOrder &o, int g, int nP,
                                           const unsigned long long *packed, float (*sp)[32],
                                           const int *flag = nullptr) {
  const int lane = threadIdx.x & 31, k = g * 32 + lane;
  q.valid = k < nP && (!flag || flag[k]);
  const int kq = q.valid ? k : 0;
  const float4 *row = reinterpret_cast<const float4 *>(o.FPs + (size_t)kq * kDS);
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const float4 v = __ldg(row + c);
    q.a[4 * c] = v.x, q.a[4 * c + 1] = v.y, q.a[4 * c + 2] = v.z, q.a[4 * c + 3] = v.w;
  }
  q.a[32] = __ldg(reinterpret_cast<const float *>(row + 8));
  const float4 p0 = __ldg(o.qp + 2 * kq), p1 = __ldg(o.qp + 2 * kq + 1);
  __syncwarp();
  sp[0][lane] = p0.x, sp[1][lane] = p0.y, sp[2][lane] = p0.z, sp[3][lane] = p0.w;
  sp[4][lane] = p1.x, sp[5][lane] = p1.y, sp[6][lane] = p1.z, sp[7][lane] = p1.w;
  __syncwarp();
  q.e = __ldg(o.qe + kq);
  // invalid lanes: bound below any distance, so they never hold the warp
  // back; valid ones start from the smallest distance published so far
  q.best = -1.f;
  q.bj = -1;
  q.taken = false;
  if (q.valid) {
    const unsigned long long pv = __ldcg(packed + kq);
    q.best = pv == ~0ull ? FLT_MAX : __uint_as_float((unsigned)(pv >> 32));
    q.bj = pv == ~0ull ? -1 : -2;
  }
}

// Whether this lane's query can find a row at or below its best in a box.
__device__ __forceinline__ bool reaches(const QueryLane &q, const float4 *__restrict__ box, const float (*sp)[32],
                                        float fac) {
  const int lane = threadIdx.x & 31;
  float s = 0.f;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float4 lo = __ldg(box + h), hi = __ldg(box + 2 + h);
    const float l[4] = {lo.x, lo.y, lo.z, lo.w}, u[4] = {hi.x, hi.y, hi.z, hi.w};
#pragma unroll
    for (int d = 0; d < 4; ++d) {
      const float p = sp[4 * h + d][lane];
      s = gap_add(s, __fsub_rd(fmaxf(__fsub_rd(l[d], p), __fsub_rd(p, u[d])), q.e));
    }
  }
  return q.valid && !(__fmul_rd(s, fac) > q.best);
}

// A warp's shared memory: two tiles and its queries' projections.
struct MatchWarp {
  float4 buf[2][kTileV];
  float sp[kAx][32];
};

// Scans the tiles t0 + k of the set bits k of todo that some query of the warp
// reaches, the next one copied while one is scanned.
template <bool kCount>
__device__ __forceinline__ void visit_tiles(QueryLane &q, const DescOrder &o, int t0, unsigned todo, int nQ,
                                            MatchWarp &w, float fac, unsigned &terms) {
  const float4 *F4 = reinterpret_cast<const float4 *>(o.FQs);
  auto find = [&]() {
    while (todo) {
      const int t = t0 + __ffs(todo) - 1;
      todo &= todo - 1;
      if (__any_sync(0xffffffffu, reaches(q, o.tbox + 4 * (size_t)t, w.sp, fac))) return t;
    }
    return -1;
  };
  int cur = find(), bi = 0;
  if (cur < 0) return;
  stage_async(w.buf[0], F4 + (size_t)cur * kTileV);
#pragma unroll 1
  while (cur >= 0) {
    const int nxt = find();
    if (nxt >= 0) {
      stage_async(w.buf[bi ^ 1], F4 + (size_t)nxt * kTileV);
      stage_wait<1>();
    } else {
      stage_wait<0>();
    }
    const int base = cur * kTile;
    scan_rows<kCount>(w.buf[bi], o.dorig + base, nQ - base < kTile ? nQ - base : kTile, q.a, q.best, q.bj, q.taken,
                      terms);
    __syncwarp();  // the buffer is refilled next
    cur = nxt, bi ^= 1;
  }
}

__device__ __forceinline__ void publish(const QueryLane &q, int g, int nP, unsigned long long *packed) {
  const int k = g * 32 + (threadIdx.x & 31);
  if (q.valid && q.taken && LSR_IN_BOUNDS(k, nP, kSiteMatchQuery)) atomicMin(packed + k, pack_pair(q.best, q.bj));
}

template <bool kCount>
__device__ __forceinline__ void count_terms(unsigned long long mine, unsigned long long *terms) {
  if (!kCount) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mine += __shfl_down_sync(0xffffffffu, mine, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(terms, mine);
}

// First pass, a warp per group: the leaves nearest to the group's box (a lane
// per leaf; ties to the smaller index) are scanned.
template <bool kCount>
__global__ void __launch_bounds__(kMT, kMatchBlocks) k_match_seed(DescOrder o, int nP, int nQ,
                                                                  unsigned long long *packed,
                                                                  unsigned long long *__restrict__ terms) {
  __shared__ MatchWarp sm[kMT / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int g = blockIdx.x * (kMT / 32) + w;
  if (g >= (int)lsr_div_up(nP, 32)) return;
  const int nl = (int)lsr_div_up(nQ, kOrdLeaf);
  // distance from the middle of the group's box to every leaf's box
  float mid[kAx];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float4 lo = __ldg(o.gbox + 4 * (size_t)g + h), hi = __ldg(o.gbox + 4 * (size_t)g + 2 + h);
    mid[4 * h] = 0.5f * (lo.x + hi.x), mid[4 * h + 1] = 0.5f * (lo.y + hi.y);
    mid[4 * h + 2] = 0.5f * (lo.z + hi.z), mid[4 * h + 3] = 0.5f * (lo.w + hi.w);
  }
  unsigned long long near[kSeedLeaves];
#pragma unroll
  for (int u = 0; u < kSeedLeaves; ++u) near[u] = ~0ull;
  for (int l = lane; l < nl; l += 32) {
    float s = 0.f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float4 lo = __ldg(o.lbox + 4 * (size_t)l + h), hi = __ldg(o.lbox + 4 * (size_t)l + 2 + h);
      const float a[4] = {lo.x, lo.y, lo.z, lo.w}, b[4] = {hi.x, hi.y, hi.z, hi.w};
#pragma unroll
      for (int d = 0; d < 4; ++d) {
        const float x = fmaxf(fmaxf(a[d] - mid[4 * h + d], mid[4 * h + d] - b[d]), 0.f);
        s = fmaf(x, x, s);
      }
    }
    unsigned long long key = pack_pair(s, l);
#pragma unroll
    for (int u = 0; u < kSeedLeaves; ++u)
      if (key < near[u]) {
        const unsigned long long x = near[u];
        near[u] = key;
        key = x;
      }
  }
  QueryLane q;
  load_query(q, o, g, nP, packed, sm[w].sp);
  unsigned uterm = 0;
  const float fac = o.pp->fac;
#pragma unroll 1
  for (int u = 0; u < kSeedLeaves; ++u) {
    unsigned long long m = near[0];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const unsigned long long x = __shfl_xor_sync(0xffffffffu, m, off);
      m = x < m ? x : m;
    }
    if (m == ~0ull) break;
    if (near[0] == m) {
#pragma unroll
      for (int v = 0; v + 1 < kSeedLeaves; ++v) near[v] = near[v + 1];
      near[kSeedLeaves - 1] = ~0ull;
    }
    const int t0 = (int)(unsigned)(m & 0xffffffffu) * (kOrdLeaf / kTile);
    const int nt = min(kOrdLeaf / kTile, (int)lsr_div_up(nQ, kTile) - t0);
    visit_tiles<kCount>(q, o, t0, (1u << nt) - 1u, nQ, sm[w], fac, uterm);
  }
  publish(q, g, nP, packed);
  count_terms<kCount>(q.valid ? uterm : 0, terms);
}

// Second pass, persistent warps. Item u = b * G + g: group g and the kTpi (8 or
// 32) tiles of block b, taken from a counter in runs of `run` (neighbouring
// groups read the same tiles, so they share L2). Small sets take blocks of 8
// tiles so that there are items for every warp. kCount: also add the number of
// terms (a_k - b_k)^2 evaluated for the valid queries to *terms (a separate
// instantiation, used when profiling). list: only its groups, and of those the
// queries with flag set.
struct MatchList {
  const int *groups, *count, *flag;
};
template <int kTpi, bool kCount>
__global__ void __launch_bounds__(kMT, kMatchBlocks) k_match_win(DescOrder o, int nP, int nQ, int run,
                                                                 MatchList list, unsigned long long *packed,
                                                                 unsigned long long *work,
                                                                 unsigned long long *__restrict__ terms) {
  __shared__ MatchWarp sm[kMT / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nt = (int)lsr_div_up(nQ, kTile);
  const int G = list.groups ? *list.count : (int)lsr_div_up(nP, 32);
  const long long nitems = lsr_div_up(nt, kTpi) * (long long)G;
  if (nitems <= 0) return;
  const float fac = o.pp->fac;
  unsigned long long nterm = 0;
  for (;;) {
    long long u0 = 0;
    if (lane == 0) u0 = (long long)atomicAdd(work, (unsigned long long)run);
    u0 = __shfl_sync(0xffffffffu, u0, 0);
    if (u0 >= nitems) break;
    int b = (int)(u0 / G), at = (int)(u0 - (long long)b * G);
#pragma unroll 1
    for (int r = 0; r < run && u0 + r < nitems; ++r, ++at) {
      if (at == G) at = 0, ++b;
      const int g = list.groups ? list.groups[at] : at;
      // the group's largest published distance against this lane's tile
      const int k = g * 32 + lane, t = b * kTpi + lane;
      unsigned far = 0u;
      if (k < nP && (!list.flag || list.flag[k])) {
        const unsigned long long pv = __ldcg(packed + k);
        far = pv == ~0ull ? __float_as_uint(FLT_MAX) : (unsigned)(pv >> 32);
      }
      const float most = __uint_as_float(__reduce_max_sync(0xffffffffu, far));
      bool open = lane < kTpi && t < nt;
      if (open) {
        float s = 0.f;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float4 tl = __ldg(o.tbox + 4 * (size_t)t + h), th = __ldg(o.tbox + 4 * (size_t)t + 2 + h);
          const float4 ql = __ldg(o.gbox + 4 * (size_t)g + h), qh = __ldg(o.gbox + 4 * (size_t)g + 2 + h);
          s = gap_add(s, fmaxf(__fsub_rd(tl.x, qh.x), __fsub_rd(ql.x, th.x)));
          s = gap_add(s, fmaxf(__fsub_rd(tl.y, qh.y), __fsub_rd(ql.y, th.y)));
          s = gap_add(s, fmaxf(__fsub_rd(tl.z, qh.z), __fsub_rd(ql.z, th.z)));
          s = gap_add(s, fmaxf(__fsub_rd(tl.w, qh.w), __fsub_rd(ql.w, th.w)));
        }
        open = !(__fmul_rd(s, fac) > most);
      }
      const unsigned todo = __ballot_sync(0xffffffffu, open);
      if (!todo) continue;
      QueryLane q;
      load_query(q, o, g, nP, packed, sm[w].sp, list.flag);
      unsigned uterm = 0;  // terms of this item (at most 33 per database row)
      visit_tiles<kCount>(q, o, b * kTpi, todo, nQ, sm[w], fac, uterm);
      publish(q, g, nP, packed);
      if (kCount && q.valid) nterm += uterm;
    }
  }
  count_terms<kCount>(nterm, terms);
}

// nn / d1 from the published minimum of every query position (none: -1 / FLT_MAX).
__global__ void k_win_finish(const unsigned long long *__restrict__ packed, const int *__restrict__ qorig, int nP,
                             int *__restrict__ nn, float *__restrict__ d1) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nP) return;
  const unsigned long long v = packed[k];
  const int q = qorig[k];
  if (!LSR_IN_BOUNDS(q, nP, kSiteMatchQuery)) return;
  const bool none = v == ~0ull;
  nn[q] = none ? -1 : (int)(unsigned)(v & 0xFFFFFFFFu);
  if (d1) d1[q] = none ? FLT_MAX : __uint_as_float((unsigned)(v >> 32));
}

// Exact FP32 scan of the queries rows[0..*nrows), split over database chunks
// (blockIdx.y) so that a short list still fills the GPU. Each block computes
// the chunk-local minimum, ties to the smaller index; chunks are combined
// with a 64-bit atomicMin on (distance bits << 32 | index), which for the
// non-negative distances keeps the smallest distance and, among equal
// distances, the smallest index -- the sequential scan's result.
__global__ void __launch_bounds__(kMT) k_match_rows_chunked(const float *__restrict__ FP, int nP,
                                                            const float *__restrict__ FQ, int nQ, int chunk,
                                                            const int *__restrict__ rows, const int *nrows,
                                                            unsigned long long *__restrict__ packed) {
  __shared__ float4 tile[kTile][9];
  const int nq = *nrows;
  const int j0 = blockIdx.y * chunk, j1 = min(nQ, j0 + chunk);
  if (j0 >= j1) return;
  int rk[4];
  stage_ranks(rk);
  for (int t0 = blockIdx.x; t0 * (kMT * kQR) < nq; t0 += gridDim.x) {
    float a[kQR][kD];
    int slot[kQR];
#pragma unroll
    for (int u = 0; u < kQR; ++u) {
      int q = t0 * (kMT * kQR) + u * kMT + threadIdx.x;
      slot[u] = q < nq ? q : -1;
      int qi = q < nq ? rows[q] : 0;
      const float *row = FP + (size_t)(qi < nP ? qi : 0) * kDS;
#pragma unroll
      for (int k = 0; k < kD; ++k) a[u][k] = row[desc_order(k)];
    }
    float best[kQR];
    int bj[kQR];
#pragma unroll
    for (int u = 0; u < kQR; ++u) best[u] = FLT_MAX, bj[u] = -1;
    for (int base = j0; base < j1; base += kTile) {
      __syncthreads();
      stage_tile(tile, FQ, base, j1, rk);
      __syncthreads();
      scan_tile<kQR>(tile, j1 - base < kTile ? j1 - base : kTile, base, a, best, bj);
    }
#pragma unroll
    for (int u = 0; u < kQR; ++u)
      if (slot[u] >= 0 && bj[u] >= 0 && LSR_IN_BOUNDS(slot[u], nP, kSiteMatchQuery))
        atomicMin(packed + slot[u], ((unsigned long long)__float_as_uint(best[u]) << 32) | (unsigned)bj[u]);
    __syncthreads();
  }
}

__global__ void k_rows_init(const int *nrows, int nP, unsigned long long *packed) {
  const int nq = *nrows;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nq; q += gridDim.x * blockDim.x)
    if (LSR_IN_BOUNDS(q, nP, kSiteMatchQuery)) packed[q] = ~0ull;
}

__global__ void k_rows_finish(const int *rows, const int *nrows, int nP, const unsigned long long *packed, int *nn,
                              float *d1) {
  const int nq = *nrows;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nq; q += gridDim.x * blockDim.x) {
    if (!LSR_IN_BOUNDS(q, nP, kSiteMatchQuery) || !LSR_IN_BOUNDS(rows[q], nP, kSiteMatchQuery)) continue;
    unsigned long long v = packed[q];
    int r = rows[q];
    bool none = v == ~0ull;
    nn[r] = none ? -1 : (int)(unsigned)(v & 0xFFFFFFFFu);
    if (d1) d1[r] = none ? FLT_MAX : __uint_as_float((unsigned)(v >> 32));
  }
}

}  // namespace

LSR_CHECK_READER(match)

namespace {

struct Fp32Layout {
  DescOrder o;
  unsigned long long *packed;  // per query position: published (distance bits << 32 | index) minimum
  unsigned long long *work;    // work-item counter
  size_t bytes;
};

Fp32Layout fp32_layout(char *base, int nP, int nQ) {
  Fp32Layout L;
  size_t off = desc_order_layout(base, nP, nQ, L.o);
  auto take = [&](size_t bytes) {
    char *p = base ? base + off : nullptr;
    off += (bytes + 255) / 256 * 256;
    return p;
  };
  L.packed = reinterpret_cast<unsigned long long *>(take(sizeof(unsigned long long) * (size_t)nP));
  L.work = reinterpret_cast<unsigned long long *>(take(sizeof(unsigned long long)));
  L.bytes = off;
  return L;
}

}  // namespace

// Five blocks of 41 KB want the whole of the SM's shared memory.
static cudaError_t prefer_shared() {
  for (auto k : {k_match_win<8, false>, k_match_win<8, true>, k_match_win<32, false>, k_match_win<32, true>})
    LSR_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
  for (auto k : {k_match_seed<false>, k_match_seed<true>})
    LSR_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
  return cudaSuccess;
}

size_t fp32_workspace_bytes(int nP, int nQ) { return fp32_layout(nullptr, nP, nQ).bytes; }

cudaError_t launch_match_fp32(const float *FP, int nP, const float *FQ, int nQ, void *ws, int *nn, float *d1,
                              cudaStream_t s, unsigned long long *terms) {
  if (nP < 1) return cudaSuccess;
  const Fp32Layout L = fp32_layout(static_cast<char *>(ws), nP, nQ);
  const int G = (int)lsr_div_up(nP, 32);
  LSR_CUDA_TRY(cudaMemsetAsync(L.packed, 0xFF, sizeof(unsigned long long) * (size_t)nP, s));
  LSR_CUDA_TRY(cudaMemsetAsync(L.work, 0, sizeof(unsigned long long), s));
  LSR_CUDA_TRY(launch_desc_order(FP, nP, FQ, nQ, L.o, s));
  if (nQ > 0) {
    LSR_CUDA_TRY(prefer_shared());
    const int seed_blocks = (int)lsr_div_up(G, kMT / 32);
    if (terms)
      LSR_LAUNCH(k_match_seed<true><<<seed_blocks, kMT, 0, s>>>(L.o, nP, nQ, L.packed, terms));
    else
      LSR_LAUNCH(k_match_seed<false><<<seed_blocks, kMT, 0, s>>>(L.o, nP, nQ, L.packed, nullptr));
    // persistent warps, as many blocks as fit on the GPU at once, or fewer;
    // runs of items as long as leaves every warp about eight
    const long long resident = (long long)kMatchBlocks * device_sm_count();
    const long long warps = resident * (kMT / 32);
    const int nt = (int)lsr_div_up(nQ, kTile);
    const bool small = lsr_div_up(nt, 32) * (long long)G < 8 * warps;
    const long long items = lsr_div_up(nt, small ? 8 : 32) * (long long)G;
    const int run = (int)std::max(1ll, std::min(8ll, items / (8 * warps)));
    const int blocks = (int)std::min(resident, (long long)lsr_div_up(lsr_div_up(items, run), kMT / 32));
    if (small && terms)
      LSR_LAUNCH(k_match_win<8, true><<<blocks, kMT, 0, s>>>(L.o, nP, nQ, run, MatchList{}, L.packed, L.work, terms));
    else if (small)
      LSR_LAUNCH(k_match_win<8, false><<<blocks, kMT, 0, s>>>(L.o, nP, nQ, run, MatchList{}, L.packed, L.work, nullptr));
    else if (terms)
      LSR_LAUNCH(k_match_win<32, true><<<blocks, kMT, 0, s>>>(L.o, nP, nQ, run, MatchList{}, L.packed, L.work, terms));
    else
      LSR_LAUNCH(k_match_win<32, false><<<blocks, kMT, 0, s>>>(L.o, nP, nQ, run, MatchList{}, L.packed, L.work, nullptr));
  }
  return launch_match_finish(L.packed, L.o.qorig, nP, nn, d1, s);
}

cudaError_t launch_match_seed(const DescOrder &o, int nP, int nQ, unsigned long long *packed, cudaStream_t s) {
  LSR_CUDA_TRY(prefer_shared());
  const int blocks = (int)lsr_div_up(lsr_div_up(nP, 32), kMT / 32);
  LSR_LAUNCH(k_match_seed<false><<<blocks, kMT, 0, s>>>(o, nP, nQ, packed, nullptr));
  return cudaGetLastError();
}

cudaError_t launch_match_listed(const DescOrder &o, int nP, int nQ, const int *groups, const int *ngroups,
                                const int *flag, unsigned long long *packed, unsigned long long *work,
                                cudaStream_t s) {
  LSR_CUDA_TRY(prefer_shared());
  const int blocks = kMatchBlocks * device_sm_count();
  LSR_LAUNCH(k_match_win<8, false><<<blocks, kMT, 0, s>>>(o, nP, nQ, 1, MatchList{groups, ngroups, flag}, packed, work,
                                                          nullptr));
  return cudaGetLastError();
}

cudaError_t launch_match_finish(const unsigned long long *packed, const int *qorig, int nP, int *nn, float *d1,
                                cudaStream_t s) {
  LSR_LAUNCH(k_win_finish<<<(int)lsr_div_up(nP, 256), 256, 0, s>>>(packed, qorig, nP, nn, d1));
  return cudaGetLastError();
}

cudaError_t launch_match_fp32_rows(const float *FP, int nP, const float *FQ, int nQ, const int *rows,
                                   const int *nrows, unsigned long long *packed, int *nn, float *d1,
                                   cudaStream_t s) {
  constexpr int kChunks = 64;
  int chunk = (int)lsr_div_up(lsr_div_up(nQ, kChunks), kTile) * kTile;
  int ny = (int)lsr_div_up(nQ, chunk);
  int nx = (int)lsr_div_up(nP, kMT * kQR);
  nx = nx < 1 ? 1 : (nx > 10 ? 10 : nx);
  int fin = (int)lsr_div_up(nP, 256);
  fin = fin < 1 ? 1 : (fin > 1216 ? 1216 : fin);
  LSR_LAUNCH(k_rows_init<<<fin, 256, 0, s>>>(nrows, nP, packed));
  LSR_LAUNCH(k_match_rows_chunked<<<dim3(nx, ny), kMT, 0, s>>>(FP, nP, FQ, nQ, chunk, rows, nrows, packed));
  LSR_LAUNCH(k_rows_finish<<<fin, 256, 0, s>>>(rows, nrows, nP, packed, nn, d1));
  return cudaGetLastError();
}

}  // namespace lsr
