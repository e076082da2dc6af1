// lsr_order.cu -- an order of both descriptor sets in which neighbouring rows
// are near in descriptor space, with bounding boxes, for the matchers of
// Algorithm 1's feature pre-matching.
//
// FPFH descriptors of indoor surfaces vary along few directions (room
// fragments: 81% of the variance on the first principal axis, 97% on the first
// six of 33), so the projections of a row on kAx axes bound its distance to
// others well: |U^T (a - b)|^2 <= lambda |a - b|^2 for the stored FP32 axes U,
// lambda >= the largest eigenvalue of their Gram matrix. Rows are put in an
// order in which kOrdTile = 32 consecutive ones are a leaf of a k-d tree: a
// counting sort by the first projection, then slabs of kOrdSlab = 4096
// consecutive rows are split at their medians along the widest of the first
// four projections, seven times, by one block each in shared memory. On room
// descriptors the tiles of 32 rows within reach of 32 queries' nearest rows
// are 4.7% of all; slabs of two axes gave 10% with these boxes and 15% with
// boxes on two axes. The order changes no result: it decides what a matcher
// can leave out.
#include <float.h>
#include <stddef.h>

#include "lsr_internal.cuh"

namespace lsr {

namespace {

constexpr int kAxThreads = 512;
constexpr int kAxSamples = 1024;  // database rows sampled for the axes (in shared memory)
constexpr int kAxRounds = 3;      // orthogonal iteration: rounds of two products and one orthogonalisation
constexpr int kKdThreads = 1024;
constexpr int kKdItems = kOrdSlab / kKdThreads;
constexpr int kKdDims = 4;        // projections the k-d splits choose from
constexpr int kGatherThreads = kOrdLeaf;
static_assert(kKdItems == 4, "a thread of the k-d sort holds four consecutive elements");
static_assert(kOrdSlab % kOrdLeaf == 0 && kOrdLeaf % kOrdTile == 0 && kOrdTile == 32, "tiles nest");

// Float -> unsigned key whose unsigned order is the float order.
__device__ __forceinline__ unsigned f2key(float f) {
  const unsigned b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float key2f(unsigned k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

// Gram-Schmidt of the kAx columns of V (kD rows), by one warp: lane holds row
// `lane`, lane 0 row 32 too. A column that is (almost) in the span of those
// before becomes zero. The products of a column with all before it are reduced
// together, so that their shuffles overlap.
__device__ __forceinline__ void orthonormalise(float (*V)[kAx]) {
  const int lane = threadIdx.x & 31;
  float x[kAx], y[kAx];
#pragma unroll
  for (int d = 0; d < kAx; ++d) x[d] = V[lane][d], y[d] = lane == 0 ? V[32][d] : 0.f;
#pragma unroll
  for (int d = 0; d < kAx; ++d) {
    float c[kAx];
#pragma unroll
    for (int p = 0; p <= d; ++p) c[p] = fmaf(x[p], x[d], y[p] * y[d]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int p = 0; p <= d; ++p) c[p] += __shfl_xor_sync(0xffffffffu, c[p], o);
#pragma unroll
    for (int p = 0; p < d; ++p) x[d] = fmaf(-c[p], x[p], x[d]), y[d] = fmaf(-c[p], y[p], y[d]);
    const float n2 = warp_sum(fmaf(x[d], x[d], y[d] * y[d]));
    const bool ok = n2 > 1e-8f * c[d] && n2 > 1e-30f && n2 <= FLT_MAX;
    const float inv = ok ? rsqrtf(n2) : 0.f;
    x[d] = ok ? x[d] * inv : 0.f, y[d] = ok ? y[d] * inv : 0.f;
  }
#pragma unroll
  for (int d = 0; d < kAx; ++d) {
    V[lane][d] = x[d];
    if (lane == 0) V[32][d] = y[d];
  }
  __syncwarp();
}

// The first kAx principal axes of up to kAxSamples evenly spaced database rows
// (covariance in shared memory, then orthogonal iteration), the factor fac by
// which a sum of squared projection gaps bounds a computed distance from below,
// and the initial keys of the first projection's range. fac = (1 - 6e-6) /
// lambda, lambda >= the largest eigenvalue of the Gram matrix of the stored
// FP32 axes (Gershgorin: max over rows of |u_i|^2 + sum |u_i . u_j|, rounded
// up), and a computed distance is >= (1 - 35 * 2^-24) |a - b|^2.
// One block, latency bound, 30 us: two axes by power iteration over the samples
// themselves took 55 us.
__global__ void __launch_bounds__(kAxThreads) k_axes(const float *__restrict__ FQ, int nQ, int ntot, OrderParams *pp) {
  extern __shared__ float xs[];  // kAxSamples x kD
  constexpr int kB = kD / 3, kPairs = kB * (kB + 1) / 2, kGroups = kAxThreads / kPairs, kCols = kAxThreads / kD;
  static_assert(kD % 3 == 0, "the covariance goes in 3 x 3 blocks");
  __shared__ float C[kD][kD + 1], V[kD][kAx], W[kD][kAx], mean[kD], part[kCols][kD], gram[kAx][kAx], lam_i[kAx];
  __shared__ float red[kGroups][kPairs * 9];
  const int tid = threadIdx.x;
  const int m = nQ < kAxSamples ? nQ : kAxSamples;
  // eight loads in flight per thread
  for (int k0 = tid; k0 < m * (kDS / 4); k0 += 8 * kAxThreads) {
    float4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = k0 + u * kAxThreads, r = k / (kDS / 4), c = k - r * (kDS / 4);
      if (k < m * (kDS / 4)) v[u] = reinterpret_cast<const float4 *>(FQ + (size_t)((long long)r * nQ / m) * kDS)[c];
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int k = k0 + u * kAxThreads, r = k / (kDS / 4), c = k - r * (kDS / 4);
      if (k >= m * (kDS / 4)) continue;
      float *dst = xs + r * kD + 4 * c;
      dst[0] = v[u].x;
      if (c < kD / 4) dst[1] = v[u].y, dst[2] = v[u].z, dst[3] = v[u].w;
    }
  }
  for (int k = tid; k < kD * kAx; k += kAxThreads) V[k / kAx][k % kAx] = (float)((k * 37 + (k % kAx) * 101 + 13) % 64) * 0.03125f - 0.984375f;
  __syncthreads();
  if (tid < kCols * kD) {
    float t = 0.f;
    for (int r = tid / kD; r < m; r += kCols) t += xs[r * kD + tid % kD];
    part[tid / kD][tid % kD] = t;
  }
  __syncthreads();
  if (tid < kD) {
    float t = 0.f;
    for (int q = 0; q < kCols; ++q) t += part[q][tid];
    mean[tid] = m > 0 ? t / (float)m : 0.f;
  }
  __syncthreads();
  if (tid < kCols * kD)
    for (int r = tid / kD; r < m; r += kCols) xs[r * kD + tid % kD] -= mean[tid % kD];
  __syncthreads();
  // covariance: a thread per 3 x 3 block (upper triangle) and sample group
  if (tid < kGroups * kPairs) {
    int bi = 0, q = tid % kPairs;
    while (q >= kB - bi) q -= kB - bi, ++bi;
    const int bj = bi + q;
    float acc[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) acc[k] = 0.f;
    for (int r = tid / kPairs; r < m; r += kGroups) {
      const float *x = xs + r * kD;
      const float a0 = x[3 * bi], a1 = x[3 * bi + 1], a2 = x[3 * bi + 2];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float b = x[3 * bj + k];
        acc[k] = fmaf(a0, b, acc[k]), acc[3 + k] = fmaf(a1, b, acc[3 + k]), acc[6 + k] = fmaf(a2, b, acc[6 + k]);
      }
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) red[tid / kPairs][(tid % kPairs) * 9 + k] = acc[k];
  }
  __syncthreads();
  for (int k = tid; k < kPairs * 9; k += kAxThreads) {
    float t = 0.f;
    for (int q = 0; q < kGroups; ++q) t += red[q][k];
    int bi = 0, q = k / 9;
    while (q >= kB - bi) q -= kB - bi, ++bi;
    const int i = 3 * bi + (k % 9) / 3, j = 3 * (bi + q) + k % 3;
    C[i][j] = t;
    if (bi + q != bi) C[j][i] = t;
  }
  __syncthreads();
  for (int it = 0; it < kAxRounds; ++it) {
    for (int half = 0; half < 2; ++half) {
      if (tid < kD * kAx) {
        float t = 0.f;
#pragma unroll
        for (int k = 0; k < kD; ++k) t = fmaf(C[tid / kAx][k], V[k][tid % kAx], t);
        W[tid / kAx][tid % kAx] = t;
      }
      __syncthreads();
      if (tid < kD * kAx) V[tid / kAx][tid % kAx] = W[tid / kAx][tid % kAx];
      __syncthreads();
    }
    if (tid < 32) {
      orthonormalise(V);
      if (it + 1 == kAxRounds) orthonormalise(V);
    }
    __syncthreads();
  }
  if (tid < kAx * kAx) {
    const int i = tid / kAx, j = tid % kAx;
    float t = 0.f;
    for (int k = 0; k < kD; ++k) t = i == j ? __fmaf_ru(V[k][i], V[k][j], t) : fmaf(V[k][i], V[k][j], t);
    // |u_i . u_j| <= |computed| + gamma_33 |u_i| |u_j| (both norms below 1 + 1e-6)
    gram[i][j] = i == j ? t : __fadd_ru(fabsf(t), 2.1e-6f);
  }
  __syncthreads();
  if (tid < kAx) {
    float t = 0.f;
    for (int j = 0; j < kAx; ++j) t = __fadd_ru(t, gram[tid][j]);
    lam_i[tid] = t;
  }
  __syncthreads();
  if (tid == 0) {
    float lam = 1.f;
    for (int d = 0; d < kAx; ++d) lam = fmaxf(lam, lam_i[d]);
    pp->fac = __fdiv_rd(0.999994f, lam);
    pp->key_min = 0xFFFFFFFFu;
    pp->key_max = 0u;
    pp->ntot = ntot;
  }
  for (int k = tid; k < kD * kAx; k += kAxThreads) pp->u[k / kAx][k % kAx] = V[k / kAx][k % kAx];
}

// Projections p_d = u_d . x (fma chains over the 33 bins in column order) of
// every database row (elements 0..nQ) and every query (elements nQ..nQ+nP), a
// bound pe >= |p_d - u_d . x| for all d (gamma_33 < 2e-6 of sum |x_k|, as no
// entry of a unit axis exceeds one; rounded up), and the range of p_0. A row
// whose projections are not all finite gets p = 0 and an infinite bound: no
// box leaves it out.
__global__ void k_proj(const float *__restrict__ FP, int nP, const float *__restrict__ FQ, int nQ, OrderParams *pp,
                       float4 *__restrict__ pq, float *__restrict__ pe) {
  __shared__ float4 su[kD][kAx / 4];
  for (int k = threadIdx.x; k < kD * kAx; k += blockDim.x) reinterpret_cast<float *>(su)[k] = (&pp->u[0][0])[k];
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned kmin = 0xFFFFFFFFu, kmax = 0u;
  if (i < nQ + nP) {
    const float4 *row = reinterpret_cast<const float4 *>(i < nQ ? FQ + (size_t)i * kDS : FP + (size_t)(i - nQ) * kDS);
    float p[kAx], S = 0.f;
#pragma unroll
    for (int d = 0; d < kAx; ++d) p[d] = 0.f;
#pragma unroll
    for (int c = 0; c < kDS / 4; ++c) {
      const float4 v = row[c];
      const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int k = 4 * c + e;
        if (k >= kD) break;
        const float4 u0 = su[k][0], u1 = su[k][1];
        p[0] = fmaf(u0.x, x[e], p[0]), p[1] = fmaf(u0.y, x[e], p[1]);
        p[2] = fmaf(u0.z, x[e], p[2]), p[3] = fmaf(u0.w, x[e], p[3]);
        p[4] = fmaf(u1.x, x[e], p[4]), p[5] = fmaf(u1.y, x[e], p[5]);
        p[6] = fmaf(u1.z, x[e], p[6]), p[7] = fmaf(u1.w, x[e], p[7]);
        S = __fadd_ru(S, fabsf(x[e]));
      }
    }
    float err = __fmaf_ru(S, 2.0e-6f, 1e-37f);
    bool fine = isfinite(err);
#pragma unroll
    for (int d = 0; d < kAx; ++d) fine = fine && isfinite(p[d]);
    if (!fine) {
      err = INFINITY;
#pragma unroll
      for (int d = 0; d < kAx; ++d) p[d] = 0.f;
    } else {
      kmin = kmax = f2key(p[0]);
    }
    pq[2 * (size_t)i] = make_float4(p[0], p[1], p[2], p[3]);
    pq[2 * (size_t)i + 1] = make_float4(p[4], p[5], p[6], p[7]);
    pe[i] = err;
  }
  const unsigned lo = __reduce_min_sync(0xffffffffu, kmin), hi = __reduce_max_sync(0xffffffffu, kmax);
  if ((threadIdx.x & 31) == 0 && lo <= hi) {
    atomicMin(&pp->key_min, lo);
    atomicMax(&pp->key_max, hi);
  }
}

// Counting sort by p_0: as many buckets per set as the set has elements, the
// database's first; each element's arrival number in its bucket is kept.
__global__ void k_bucket(const float4 *__restrict__ pq, int nQ, int nP, const OrderParams *pp, int *__restrict__ slot,
                         int *__restrict__ rank, int *__restrict__ counts) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nQ + nP) return;
  const bool db = i < nQ;
  const int nb = db ? nQ : nP;
  const unsigned k0 = pp->key_min, k1 = pp->key_max;
  int b = nb - 1;
  if (k0 <= k1) {
    const float lo = key2f(k0), hi = key2f(k1);
    const float f = (pq[2 * (size_t)i].x - lo) * (hi > lo ? (float)nb / (hi - lo) : 0.f);
    b = f < (float)nb ? (int)f : nb - 1;
    b = b < 0 ? 0 : b;
  }
  const int s = (db ? 0 : nQ) + b;
  slot[i] = s;
  rank[i] = atomicAdd(counts + s, 1);
}

__global__ void k_bucket_scatter(int n, const int *__restrict__ slot, const int *__restrict__ rank,
                                 const int *__restrict__ start, int *__restrict__ out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const int pos = start[slot[j]] + rank[j];
  if (LSR_IN_BOUNDS(pos, n, kSiteMatchRow)) out[pos] = j;
}

// One block per slab of kOrdSlab positions of the first order (the database's
// slabs first): k-d splits down to tiles of 32. A level sorts every segment of
// L positions by its widest of kKdDims projections and halves it. The sort is
// bitonic on 32-bit keys, the projection in 2^20 steps of the segment's range
// above the element's 12-bit number (64-bit keys with all of the projection
// took 117 us for the slabs of 300k rows, these 74); four consecutive elements a thread: partners within a
// thread or a warp by registers and shuffles, the others through shared
// memory. Positions past the end sort last everywhere.
__global__ void __launch_bounds__(kKdThreads) k_kd(const float4 *__restrict__ pq, const int *__restrict__ order1, int nQ,
                                                   int nP, int slabs_db, int *__restrict__ order) {
  extern __shared__ float4 kd_smem[];
  float4 *sp = kd_smem;                                      // kOrdSlab projections
  uint4 *sk = reinterpret_cast<uint4 *>(sp + kOrdSlab);      // kOrdSlab keys, four a thread
  __shared__ float wlo[32][kKdDims], whi[32][kKdDims];
  static_assert(kOrdSlab == 4096, "an element's number is 12 bits");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool db = (int)blockIdx.x < slabs_db;
  const int base = db ? blockIdx.x * kOrdSlab : nQ + (blockIdx.x - slabs_db) * kOrdSlab;
  const int lim = db ? nQ : nQ + nP;
  const int m = min(kOrdSlab, lim - base);
  for (int j = tid; j < m; j += kKdThreads) sp[j] = pq[2 * (size_t)order1[base + j]];
  __syncthreads();
  unsigned x[kKdItems];  // the element's number in the low 12 bits
#pragma unroll
  for (int u = 0; u < kKdItems; ++u) x[u] = kKdItems * tid + u;
  for (int L = kOrdSlab; L > kOrdTile; L >>= 1) {
    float lo[kKdDims], hi[kKdDims];
#pragma unroll
    for (int d = 0; d < kKdDims; ++d) lo[d] = INFINITY, hi[d] = -INFINITY;
    float4 v[kKdItems];
#pragma unroll
    for (int u = 0; u < kKdItems; ++u) {
      const int e = x[u] & 4095u;
      v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (e >= m) continue;
      v[u] = sp[e];
      lo[0] = fminf(lo[0], v[u].x), hi[0] = fmaxf(hi[0], v[u].x), lo[1] = fminf(lo[1], v[u].y), hi[1] = fmaxf(hi[1], v[u].y);
      lo[2] = fminf(lo[2], v[u].z), hi[2] = fmaxf(hi[2], v[u].z), lo[3] = fminf(lo[3], v[u].w), hi[3] = fmaxf(hi[3], v[u].w);
    }
    for (int o = 1; o < 32 && o < L / kKdItems; o <<= 1)
#pragma unroll
      for (int d = 0; d < kKdDims; ++d) {
        lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
        hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
      }
    if (L > 32 * kKdItems) {
      __syncthreads();  // the previous level has read the table
      if (lane == 0)
#pragma unroll
        for (int d = 0; d < kKdDims; ++d) wlo[warp][d] = lo[d], whi[warp][d] = hi[d];
      __syncthreads();
      const int nw = L / (32 * kKdItems), w0 = warp / nw * nw;
      for (int w = w0; w < w0 + nw; ++w)
#pragma unroll
        for (int d = 0; d < kKdDims; ++d) lo[d] = fminf(lo[d], wlo[w][d]), hi[d] = fmaxf(hi[d], whi[w][d]);
    }
    int dim = 0;
    float from = lo[0], wide = hi[0] - lo[0];
#pragma unroll
    for (int d = 1; d < kKdDims; ++d)
      if (hi[d] - lo[d] > wide) wide = hi[d] - lo[d], from = lo[d], dim = d;
    const float scale = wide > 0.f && wide <= FLT_MAX ? 1048574.f / wide : 0.f;
#pragma unroll
    for (int u = 0; u < kKdItems; ++u) {
      const int e = x[u] & 4095u;
      const float p = dim == 0 ? v[u].x : dim == 1 ? v[u].y : dim == 2 ? v[u].z : v[u].w;
      const unsigned step = e < m ? min((unsigned)fmaxf((p - from) * scale, 0.f), 1048574u) : 1048575u;
      x[u] = (step << 12) | (unsigned)e;
    }
    for (int k = 2; k <= L; k <<= 1)
      for (int j = k >> 1; j > 0; j >>= 1) {
        if (j >= 32 * kKdItems) {
          __syncthreads();
          sk[tid] = make_uint4(x[0], x[1], x[2], x[3]);
          __syncthreads();
          // the partners of four consecutive elements are consecutive too
          const int i = kKdItems * tid;
          const uint4 y = sk[(i ^ j) / kKdItems];
          const bool keep_min = (((i & (L - 1)) & k) == 0) == ((i & j) == 0);
          x[0] = keep_min ? min(x[0], y.x) : max(x[0], y.x), x[1] = keep_min ? min(x[1], y.y) : max(x[1], y.y);
          x[2] = keep_min ? min(x[2], y.z) : max(x[2], y.z), x[3] = keep_min ? min(x[3], y.w) : max(x[3], y.w);
        } else if (j >= kKdItems) {
          const int i = kKdItems * tid;
          const bool keep_min = (((i & (L - 1)) & k) == 0) == ((i & j) == 0);
#pragma unroll
          for (int u = 0; u < kKdItems; ++u) {
            const unsigned y = __shfl_xor_sync(0xffffffffu, x[u], j / kKdItems);
            x[u] = keep_min ? min(x[u], y) : max(x[u], y);
          }
        } else {
#pragma unroll
          for (int u = 0; u < kKdItems; ++u) {
            if (j == 2 ? u >= 2 : (u & 1)) continue;
            const int i = kKdItems * tid + u;
            const bool up = ((i & (L - 1)) & k) == 0;
            unsigned &a = x[u], &b = j == 2 ? x[(u + 2) & 3] : x[u | 1];
            const unsigned mn = min(a, b), mx = max(a, b);
            a = up ? mn : mx, b = up ? mx : mn;
          }
        }
      }
  }
#pragma unroll
  for (int u = 0; u < kKdItems; ++u) {
    const int pos = kKdItems * tid + u, e = x[u] & 4095u;
    if (pos < m && e < m) order[base + pos] = order1[base + e];
  }
}

// One block per leaf (kOrdLeaf positions) of the database, then of the
// queries: the rows in the final order with their original indices, and the
// boxes of the projection intervals [p - pe, p + pe]. Database rows go
// chunk-major per tile of 32 (float4 chunk c of row j at c * 32 + j), query
// rows one after another, both with bins in desc_order and zeros in slots
// 33..35; a box is (lo 0..3, lo 4..7, hi 0..3, hi 4..7). Without kBoxes: the
// rows alone, in the caller's order.
template <bool kBoxes>
__global__ void __launch_bounds__(kGatherThreads) k_gather(const float *__restrict__ FP, int nP,
                                                           const float *__restrict__ FQ, int nQ, int leaves_db,
                                                           DescOrder o) {
  __shared__ float4 sb[kOrdLeaf / kOrdTile][4];
  const bool db = (int)blockIdx.x < leaves_db;
  const int leaf = db ? blockIdx.x : blockIdx.x - leaves_db, n = db ? nQ : nP;
  const int pos = leaf * kOrdLeaf + threadIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float lo[kAx], hi[kAx];
#pragma unroll
  for (int d = 0; d < kAx; ++d) lo[d] = INFINITY, hi[d] = -INFINITY;
  if (pos < n) {
    int e = kBoxes ? o.order[(db ? 0 : nQ) + pos] : (db ? 0 : nQ) + pos;
    if (!LSR_IN_BOUNDS(db ? e : e - nQ, n, db ? kSiteMatchRow : kSiteMatchQuery)) e = db ? 0 : nQ;
    const int i = db ? e : e - nQ;
    const float *src = (db ? FQ : FP) + (size_t)i * kDS;
    float4 *dst = db ? reinterpret_cast<float4 *>(o.FQs) + (size_t)(pos / kOrdTile) * (9 * kOrdTile) + lane
                     : reinterpret_cast<float4 *>(o.FPs) + (size_t)pos * (kDS / 4);
    const int step = db ? kOrdTile : 1;
#pragma unroll
    for (int c = 0; c < kDS / 4; ++c) {
      float v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = 4 * c + k < kD ? src[desc_order(4 * c + k)] : 0.f;
      dst[c * step] = make_float4(v[0], v[1], v[2], v[3]);
    }
    (db ? o.dorig : o.qorig)[pos] = i;
    if (!kBoxes) return;
    const float4 p0 = o.pq[2 * (size_t)e], p1 = o.pq[2 * (size_t)e + 1];
    const float err = o.pe[e];
    if (!db) {
      o.qp[2 * (size_t)pos] = p0, o.qp[2 * (size_t)pos + 1] = p1;
      o.qe[pos] = err;
    }
    const float p[kAx] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
#pragma unroll
    for (int d = 0; d < kAx; ++d) lo[d] = __fsub_rd(p[d], err), hi[d] = __fadd_ru(p[d], err);
  }
  if (!kBoxes) return;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
#pragma unroll
    for (int d = 0; d < kAx; ++d) {
      lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], off));
      hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], off));
    }
  const float4 bx[4] = {make_float4(lo[0], lo[1], lo[2], lo[3]), make_float4(lo[4], lo[5], lo[6], lo[7]),
                        make_float4(hi[0], hi[1], hi[2], hi[3]), make_float4(hi[4], hi[5], hi[6], hi[7])};
  if (lane == 0) {
    float4 *box = db ? o.tbox : o.gbox;
    const int tile = pos / kOrdTile;
    if (pos < n)
#pragma unroll
      for (int k = 0; k < 4; ++k) box[4 * (size_t)tile + k] = bx[k];
#pragma unroll
    for (int k = 0; k < 4; ++k) sb[w][k] = bx[k];
  }
  __syncthreads();
  float4 *leaf_box = db ? o.lbox : o.qbox;
  if (threadIdx.x < 4) {
    const int k = threadIdx.x;
    float4 r = sb[0][k];
    for (int t = 1; t < kOrdLeaf / kOrdTile; ++t) {
      const float4 x = sb[t][k];
      if (k < 2)
        r = make_float4(fminf(r.x, x.x), fminf(r.y, x.y), fminf(r.z, x.z), fminf(r.w, x.w));
      else
        r = make_float4(fmaxf(r.x, x.x), fmaxf(r.y, x.y), fmaxf(r.z, x.z), fmaxf(r.w, x.w));
    }
    leaf_box[4 * (size_t)leaf + k] = r;
  }
}

}  // namespace

LSR_CHECK_READER(order)

size_t desc_order_layout(char *base, int nP, int nQ, DescOrder &o) {
  const size_t n = (size_t)nP + (size_t)nQ, nt = (size_t)lsr_div_up(nQ, kOrdTile), nl = (size_t)lsr_div_up(nQ, kOrdLeaf);
  const size_t ng = (size_t)lsr_div_up(nP, kOrdTile), nql = (size_t)lsr_div_up(nP, kOrdLeaf);
  size_t off = 0;
  auto take = [&](auto *&p, size_t count) {
    using T = std::remove_reference_t<decltype(*p)>;
    p = reinterpret_cast<T *>(base ? base + off : nullptr);
    off += (sizeof(T) * (count > 0 ? count : 1) + 255) / 256 * 256;
  };
  take(o.pp, 1);
  take(o.pq, 2 * n);
  take(o.pe, n);
  take(o.slot, n);
  take(o.rank, n);
  take(o.counts, n + 1);
  take(o.start, n + 1);
  take(o.order1, n);
  take(o.order, n);
  take(o.scan, (size_t)scan_scratch_ints((int64_t)n));
  // whole tiles: chunk c of the last tile's rows lies at c * 32 within it
  take(o.FQs, kDS * kOrdTile * nt);
  take(o.dorig, (size_t)nQ);
  take(o.tbox, 4 * nt);
  take(o.lbox, 4 * nl);
  take(o.FPs, kDS * (size_t)nP);
  take(o.qorig, (size_t)nP);
  take(o.qp, 2 * (size_t)nP);
  take(o.qe, (size_t)nP);
  take(o.gbox, 4 * ng);
  take(o.qbox, 4 * nql);
  return off;
}

cudaError_t launch_desc_order(const float *FP, int nP, const float *FQ, int nQ, const DescOrder &o, cudaStream_t s) {
  const int n = nP + nQ, eb = (int)lsr_div_up(n, 256);
  constexpr int kAxSmem = kAxSamples * kD * (int)sizeof(float);
  constexpr int kKdSmem = kOrdSlab * (int)(sizeof(float4) + sizeof(unsigned));
  LSR_CUDA_TRY(cudaMemsetAsync(o.counts, 0, sizeof(int) * ((size_t)n + 1), s));
  LSR_CUDA_TRY(cudaFuncSetAttribute(k_axes, cudaFuncAttributeMaxDynamicSharedMemorySize, kAxSmem));
  LSR_CUDA_TRY(cudaFuncSetAttribute(k_kd, cudaFuncAttributeMaxDynamicSharedMemorySize, kKdSmem));
  LSR_LAUNCH(k_axes<<<1, kAxThreads, kAxSmem, s>>>(FQ, nQ, n, o.pp));
  LSR_LAUNCH(k_proj<<<eb, 256, 0, s>>>(FP, nP, FQ, nQ, o.pp, o.pq, o.pe));
  LSR_LAUNCH(k_bucket<<<eb, 256, 0, s>>>(o.pq, nQ, nP, o.pp, o.slot, o.rank, o.counts));
  LSR_CUDA_TRY(scan_exclusive(o.counts, o.start, &o.pp->ntot, n, o.scan, s));
  LSR_LAUNCH(k_bucket_scatter<<<eb, 256, 0, s>>>(n, o.slot, o.rank, o.start, o.order1));
  const int slabs_db = (int)lsr_div_up(nQ, kOrdSlab), slabs_q = (int)lsr_div_up(nP, kOrdSlab);
  LSR_LAUNCH(k_kd<<<slabs_db + slabs_q, kKdThreads, kKdSmem, s>>>(o.pq, o.order1, nQ, nP, slabs_db, o.order));
  const int leaves_db = (int)lsr_div_up(nQ, kOrdLeaf), leaves_q = (int)lsr_div_up(nP, kOrdLeaf);
  LSR_LAUNCH(k_gather<true><<<leaves_db + leaves_q, kGatherThreads, 0, s>>>(FP, nP, FQ, nQ, leaves_db, o));
  return cudaGetLastError();
}

cudaError_t launch_desc_rows(const float *FP, int nP, const float *FQ, int nQ, const DescOrder &o, cudaStream_t s) {
  const int leaves_db = (int)lsr_div_up(nQ, kOrdLeaf), leaves_q = (int)lsr_div_up(nP, kOrdLeaf);
  LSR_LAUNCH(k_gather<false><<<leaves_db + leaves_q, kGatherThreads, 0, s>>>(FP, nP, FQ, nQ, leaves_db, o));
  return cudaGetLastError();
}

}  // namespace lsr
