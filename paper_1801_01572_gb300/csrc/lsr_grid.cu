// lsr_grid.cu -- bounding boxes, the uniform 3D grid of eq. (1) and its
// construction by a deterministic counting sort.
//
// The grid replaces a k-d tree for neighbour search (Sec. IV: O(1) cell
// lookup, no data-dependent branching on the search path). Cells are stored
// densely over the bounding box; points are sorted by cell so that the three
// x-adjacent cells of a row form one contiguous range, and a radius query
// reads at most nine contiguous ranges.
#include <float.h>

#include <algorithm>

#include "lsr_internal.cuh"

namespace lsr {

namespace {

constexpr int kBoxThreads = 256;
constexpr int kBoxItems = 8;

__device__ __forceinline__ float3 load_xyz(const float *xyz, int i) {
  return make_float3(xyz[3 * i], xyz[3 * i + 1], xyz[3 * i + 2]);
}

// The partial of one block of points: min (3), max (3), non-finite flag, count
// and coordinate sums (3) of the finite ones, as kBoxPart doubles.
__device__ __forceinline__ void bbox_partial(const float *__restrict__ xyz, int n, int block, double *out) {
  float lo[3] = {FLT_MAX, FLT_MAX, FLT_MAX}, hi[3] = {-FLT_MAX, -FLT_MAX, -FLT_MAX};
  float bad = 0.f, cnt = 0.f;
  float sum[3] = {0.f, 0.f, 0.f};
  int base = block * kBoxThreads * kBoxItems;
  for (int k = 0; k < kBoxItems; ++k) {
    int i = base + k * kBoxThreads + threadIdx.x;
    if (i >= n) break;
    const float3 p = load_xyz(xyz, i);
    if (!(isfinite(p.x) && isfinite(p.y) && isfinite(p.z))) {
      bad = 1.f;
      continue;
    }
    lo[0] = fminf(lo[0], p.x), lo[1] = fminf(lo[1], p.y), lo[2] = fminf(lo[2], p.z);
    hi[0] = fmaxf(hi[0], p.x), hi[1] = fmaxf(hi[1], p.y), hi[2] = fmaxf(hi[2], p.z);
    sum[0] += p.x, sum[1] += p.y, sum[2] += p.z;
    cnt += 1.f;
  }
  for (int off = 16; off > 0; off >>= 1) {
    for (int d = 0; d < 3; ++d) {
      lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], off));
      hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], off));
      sum[d] += __shfl_xor_sync(0xffffffffu, sum[d], off);
    }
    bad = fmaxf(bad, __shfl_xor_sync(0xffffffffu, bad, off));
    cnt += __shfl_xor_sync(0xffffffffu, cnt, off);
  }
  __shared__ float sm[kBoxThreads / 32][kBoxPart];
  int w = threadIdx.x / 32, l = threadIdx.x % 32;
  if (l == 0) {
    for (int d = 0; d < 3; ++d) sm[w][d] = lo[d], sm[w][3 + d] = hi[d], sm[w][8 + d] = sum[d];
    sm[w][6] = bad;
    sm[w][7] = cnt;
  }
  __syncthreads();
  if (threadIdx.x < kBoxPart) {
    int t = threadIdx.x;
    double v = sm[0][t];
    for (int k = 1; k < kBoxThreads / 32; ++k) {
      double u = sm[k][t];
      v = t < 3 ? fmin(v, u) : (t < 7 ? fmax(v, u) : v + u);
    }
    out[t] = v;
  }
}

// box from the nblk partials, combined in block order (a block of kBoxThreads
// stages them in shared memory; combining straight from global memory was a
// chain of 74 loads at 150k points, 14 to 25 us): min (3), max (3), non-finite
// flag, number of finite points, centroid (3). Ends with a barrier.
__device__ __forceinline__ void bbox_combine(const double *partials, int nblk, float *box) {
  constexpr int kStage = 64;
  __shared__ double st[kStage * kBoxPart], acc[kBoxPart];
  const int t = threadIdx.x;
  double v = 0.0;
  for (int b0 = 0; b0 < nblk; b0 += kStage) {
    const int nb = min(kStage, nblk - b0);
    for (int k = t; k < nb * kBoxPart; k += kBoxThreads) st[k] = __ldcg(partials + (size_t)b0 * kBoxPart + k);
    __syncthreads();
    if (t < kBoxPart) {
      if (b0 == 0) v = st[t];
      for (int b = b0 == 0 ? 1 : 0; b < nb; ++b) {
        const double u = st[b * kBoxPart + t];
        v = t < 3 ? fmin(v, u) : (t < 7 ? fmax(v, u) : v + u);
      }
    }
    __syncthreads();
  }
  if (t < kBoxPart) acc[t] = v;
  __syncthreads();
  if (t < 8) box[t] = (float)acc[t];
  if (t >= 8 && t < 11) box[t] = acc[7] > 0.0 ? (float)(acc[t] / acc[7]) : 0.f;
  if (t == 11) box[t] = 0.f;
  __threadfence_block();
  __syncthreads();
}

__global__ void __launch_bounds__(kBoxThreads) k_bbox_partial(const float *xyz, int n, double *partials) {
  bbox_partial(xyz, n, blockIdx.x, partials + (size_t)kBoxPart * blockIdx.x);
}

__global__ void __launch_bounds__(kBoxThreads) k_bbox_final(const double *partials, int nblk, float *box) {
  bbox_combine(partials, nblk, box);
}

__device__ void grid_params(const float *box, float radius, int npts, int cap, const unsigned *mask, GridParams *g) {
  GridParams q;
  float ext[3] = {box[3] - box[0], box[4] - box[1], box[5] - box[2]};
  // Cell coordinates (x - origin) / cell are computed in FP32 with a relative
  // error of a few units of 2^-24 of the box extent; the cell is enlarged by
  // that margin (at least 1e-4) so that two points within the radius never
  // land more than one cell apart.
  float emax = fmaxf(fmaxf(ext[0], ext[1]), ext[2]);
  if (!(emax >= 0.f) || !isfinite(emax)) emax = 0.f;
  float delta = fmaxf(1e-4f, 8.f * 5.9604645e-8f * emax / radius);
  float cell = radius * (1.f + delta);
  q.cell = cell;
  q.inv_cell = 1.0f / cell;
  q.ox = box[0], q.oy = box[1], q.oz = box[2];
  int nn[3];
  for (int d = 0; d < 3; ++d) {
    float e = ext[d] * q.inv_cell;
    if (!(e >= 0.f)) e = 0.f;            // empty or non-finite input
    if (e > 1073741824.f) e = 1073741824.f;
    nn[d] = (int)floorf(e) + 1;
  }
  q.nx = nn[0], q.ny = nn[1], q.nz = nn[2];
  long long cx = nn[0], cy = nn[1], cz = nn[2];
  long long wx = cx, wy = cy, wz = cz;
  if (wx * wy * wz > cap) {
    if (wx * wy <= cap) {
      wz = cap / (wx * wy);
    } else {
      wz = 1;
      if (wx <= cap) {
        wy = cap / wx;
      } else {
        wy = 1;
        wx = cap;
      }
    }
    if (wz < 1) wz = 1;
    if (wy < 1) wy = 1;
  }
  q.wx = (int)wx, q.wy = (int)wy, q.wz = (int)wz;
  q.ncells = (int)(wx * wy * wz);
  q.npts = npts;
  q.margin = grid_margin(q.cell, q.nx, q.ny, q.nz);
  q.nbmask = mask;
  *g = q;
}

// Dilate the occupied storage cell c into its 3 x 3 x 3 neighbourhood
// (neighbourhoods are symmetric, so a query cell's bit is set iff some point
// lies in the block around it; wrapped axes dilate modulo the stored extent,
// which can only add bits). The x-adjacent bits of a row are set at once.
__device__ __forceinline__ void dilate_cell(const GridParams &g, int c, unsigned *mask) {
  const bool wx = g.wx != g.nx, wy = g.wy != g.ny, wz = g.wz != g.nz;
  const int sx = c % g.wx, sy = (c / g.wx) % g.wy, sz = c / (g.wx * g.wy);
  for (int dz = -1; dz <= 1; ++dz) {
    int z = sz + dz;
    if (z < 0 || z >= g.wz) {
      if (!wz) continue;
      z = (z + g.wz) % g.wz;
    }
    for (int dy = -1; dy <= 1; ++dy) {
      int y = sy + dy;
      if (y < 0 || y >= g.wy) {
        if (!wy) continue;
        y = (y + g.wy) % g.wy;
      }
      const int row = (z * g.wy + y) * g.wx;
      int word = -1;
      unsigned bits = 0u;
      for (int dx = -1; dx <= 1; ++dx) {
        int x = sx + dx;
        if (x < 0 || x >= g.wx) {
          if (!wx) continue;
          x = (x + g.wx) % g.wx;
        }
        const int t = row + x;
        if ((t >> 5) != word) {
          if (bits) atomicOr(mask + word, bits);
          word = t >> 5, bits = 0u;
        }
        bits |= 1u << (t & 31);
      }
      if (bits) atomicOr(mask + word, bits);
    }
  }
}

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

__device__ __forceinline__ int cell_slot(const GridParams &g, float x, float y, float z) {
  int cx = clampi(__float2int_rd((x - g.ox) * g.inv_cell), 0, g.nx - 1);
  int cy = clampi(__float2int_rd((y - g.oy) * g.inv_cell), 0, g.ny - 1);
  int cz = clampi(__float2int_rd((z - g.oz) * g.inv_cell), 0, g.nz - 1);
  return ((cz % g.wz) * g.wy + (cy % g.wy)) * g.wx + (cx % g.wx);
}

// Grids are built for up to kGridJobs clouds at once: blockIdx.y is the job.
// At the library's sizes (5k to 200k points) every step is a launch of a few
// microseconds, so what a build costs is the number of launches: six for any
// number of grids, seven with a bounding box to find, where each grid used to
// take twelve kernels and three memsets of its own.
struct GridJobs {
  GridJob j[kGridJobs];
};

// Clears the counts, the neighbourhood mask and the caller's array, and fills
// the grid's parameters from a known box.
__global__ void k_grid_begin(const __grid_constant__ GridJobs J) {
  const GridJob &job = J.j[blockIdx.y];
  const int t = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
  auto zero = [&](void *p, int64_t words) {
    if (!p) return;
    int *w = static_cast<int *>(p);
    // word by word up to a 16-byte boundary (a caller's array may start anywhere), then vectors
    const int64_t head = min(words, (int64_t)(((16 - ((uintptr_t)p & 15)) & 15) >> 2)), vec = (words - head) / 4;
    for (int64_t k = t; k < vec; k += step) reinterpret_cast<int4 *>(w + head)[k] = make_int4(0, 0, 0, 0);
    for (int64_t k = t; k < words - 4 * vec; k += step) w[k < head ? k : k + 4 * vec] = 0;
  };
  zero(job.sc.counts, (int64_t)job.cap + 1);
  zero(job.mask, job.mask ? job.cap / 32 + 2 : 0);
  zero(job.zero, job.zero_words);
  if (t == 0 && !job.box_part && !job.params_ready) grid_params(job.box, job.radius, job.n, job.cap, job.mask, job.g);
}

// Bounding box of the jobs that need one; the last block of a job to finish
// (a ticket in the spare word after the counts) combines the partials in
// block order and fills the grid's parameters.
__global__ void __launch_bounds__(kBoxThreads) k_grid_bbox(const __grid_constant__ GridJobs J) {
  const GridJob &job = J.j[blockIdx.y];
  const int nblk = (job.n + kBoxThreads * kBoxItems - 1) / (kBoxThreads * kBoxItems);
  if (!job.box_part || (int)blockIdx.x >= nblk) return;
  __shared__ int s_last;
  bbox_partial(job.xyz, job.n, blockIdx.x, job.box_part + (size_t)kBoxPart * blockIdx.x);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(job.sc.counts + job.cap, 1) == nblk - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  bbox_combine(job.box_part, nblk, job.box);
  if (threadIdx.x == 0 && job.g) grid_params(job.box, job.radius, job.n, job.cap, job.mask, job.g);
}

// The cell of every point and its arrival number there.
__global__ void k_grid_slots(const __grid_constant__ GridJobs J) {
  const GridJob &job = J.j[blockIdx.y];
  if (!job.out) return;
  const GridParams g = *job.g;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < job.n; i += gridDim.x * blockDim.x) {
    float3 p;
    if (job.x4) {
      const float4 q = job.x4[i];
      p = make_float3(q.x, q.y, q.z);
    } else {
      p = load_xyz(job.xyz, i * job.stride);
    }
    const int s = cell_slot(g, p.x, p.y, p.z);
    job.sc.slot[i] = s;
    job.sc.rank[i] = atomicAdd(job.sc.counts + s, 1);
  }
}

__global__ void k_grid_scatter(const __grid_constant__ GridJobs J) {
  const GridJob &job = J.j[blockIdx.y];
  if (!job.out) return;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < job.n; i += gridDim.x * blockDim.x)
    job.sc.tmp[job.start[job.sc.slot[i]] + job.sc.rank[i]] = i;
}

// A thread per point, in cell order: its place among the cell's points by
// source index (the arrival order is arbitrary, the result is not), and, once
// per occupied cell, the neighbourhood mask. (A warp per cell walked mostly
// empty cells: two dependent loads for each of up to 400k cells.)
__global__ void k_grid_order(const __grid_constant__ GridJobs J) {
  const GridJob &job = J.j[blockIdx.y];
  if (!job.out) return;
  const int *__restrict__ tmp = job.sc.tmp;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < job.n; t += gridDim.x * blockDim.x) {
    const int v = tmp[t];
    const int c = job.sc.slot[v];
    const int b = job.start[c], e = job.start[c + 1];
    float4 o;
    if (job.x4) {
      o = job.x4[v];
    } else {
      const float3 p = load_xyz(job.xyz, v * job.stride);
      o = make_float4(p.x, p.y, p.z, 0.f);
    }
    int rank = 0;
#pragma unroll 4
    for (int u = b; u < e; ++u) rank += tmp[u] < v;
    o.w = __int_as_float(job.carry_pos ? b + rank : v);
    job.out[b + rank] = o;
    if (job.inv) job.inv[v] = b + rank;
    if (job.mask && t == b) dilate_cell(*job.g, c, job.mask);
  }
}

// ---------------------------------------------------------------- scan
constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ int block_exclusive_scan(int v, int *sm_warp, int *total) {
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int x = v;
  for (int off = 1; off < 32; off <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) sm_warp[w] = x;
  __syncthreads();
  if (w == 0) {
    int s = lane < (kScanThreads / 32) ? sm_warp[lane] : 0;
    for (int off = 1; off < 32; off <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, s, off);
      if (lane >= off) s += y;
    }
    if (lane < (kScanThreads / 32)) sm_warp[lane] = s;
  }
  __syncthreads();
  int warp_off = w > 0 ? sm_warp[w - 1] : 0;
  *total = sm_warp[kScanThreads / 32 - 1];
  __syncthreads();
  return warp_off + x - v;
}

// Exclusive scans in two launches: the sum of every tile, then each tile adds
// up the sums before its own (at most kScanTiles of them) and scans itself.
// Tiles grow with the capacity so that there are never more.
constexpr int kScanTiles = 1024;
__host__ __device__ __forceinline__ int64_t scan_tile_size(int64_t cap) {
  const int64_t parts = (cap + kScanTile) / kScanTile;  // of kScanTile entries, cap + 1 in all
  return (parts + kScanTiles - 1) / kScanTiles * kScanTile;
}

__device__ __forceinline__ int block_sum(int v, int *sm_warp) {
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  if ((threadIdx.x & 31) == 0) sm_warp[threadIdx.x >> 5] = v;
  __syncthreads();
  int t = 0;
  for (int w = 0; w < kScanThreads / 32; ++w) t += sm_warp[w];
  __syncthreads();
  return t;
}

// in (256-byte aligned): n entries; sums[tile] for the tiles that begin before n.
__device__ __forceinline__ void scan_tile_sum(const int *__restrict__ in, int n, int64_t tile, int *__restrict__ sums) {
  __shared__ int sm[kScanThreads / 32];
  const int64_t base = (int64_t)blockIdx.x * tile;
  if (base >= n) return;
  const int64_t end = base + tile < n ? base + tile : n;
  int sum = 0;
  for (int64_t i = base + 4 * (int)threadIdx.x; i < end; i += 4 * kScanThreads) {
    if (i + 3 < end) {
      const int4 q = *reinterpret_cast<const int4 *>(in + i);
      sum += q.x + q.y + q.z + q.w;
    } else {
      for (int64_t k = i; k < end; ++k) sum += in[k];
    }
  }
  sum = block_sum(sum, sm);
  if (threadIdx.x == 0) sums[blockIdx.x] = sum;
}

// out[0..n] = exclusive scan of in[0..n), out[n] = the total.
__device__ __forceinline__ void scan_tile_write(const int *__restrict__ in, int n, int64_t tile,
                                                const int *__restrict__ sums, int *__restrict__ out) {
  __shared__ int sm[kScanThreads / 32];
  const int64_t base = (int64_t)blockIdx.x * tile;
  if (base > n) return;
  int carry = 0;
  for (int k = threadIdx.x; k < (int)blockIdx.x; k += kScanThreads) carry += sums[k];
  carry = block_sum(carry, sm);
  const int64_t end = base + tile < (int64_t)n + 1 ? base + tile : (int64_t)n + 1;
  for (int64_t b = base; b < end; b += kScanTile) {
    const int64_t i0 = b + threadIdx.x * kScanItems;
    int v[kScanItems];
    int sum = 0;
    if (i0 + kScanItems <= n) {
      const int4 q0 = reinterpret_cast<const int4 *>(in + i0)[0], q1 = reinterpret_cast<const int4 *>(in + i0)[1];
      v[0] = q0.x, v[1] = q0.y, v[2] = q0.z, v[3] = q0.w, v[4] = q1.x, v[5] = q1.y, v[6] = q1.z, v[7] = q1.w;
    } else {
#pragma unroll
      for (int k = 0; k < kScanItems; ++k) v[k] = i0 + k < n ? in[i0 + k] : 0;
    }
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) sum += v[k];
    int total;
    int pre = carry + block_exclusive_scan(sum, sm, &total);
    carry += total;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
      const int c = v[k];
      v[k] = pre;
      pre += c;
    }
    if (i0 + kScanItems <= end) {
      reinterpret_cast<int4 *>(out + i0)[0] = make_int4(v[0], v[1], v[2], v[3]);
      reinterpret_cast<int4 *>(out + i0)[1] = make_int4(v[4], v[5], v[6], v[7]);
    } else {
#pragma unroll
      for (int k = 0; k < kScanItems; ++k)
        if (i0 + k < end) out[i0 + k] = v[k];
    }
  }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_sums(const int *in, const int *n_dev, int64_t tile, int *sums) {
  scan_tile_sum(in, *n_dev, tile, sums);
}
__global__ void __launch_bounds__(kScanThreads) k_scan_write(const int *in, const int *n_dev, int64_t tile,
                                                             const int *sums, int *out) {
  scan_tile_write(in, *n_dev, tile, sums, out);
}
__global__ void __launch_bounds__(kScanThreads) k_grid_sums(const __grid_constant__ GridJobs J) {
  const GridJob &job = J.j[blockIdx.y];
  if (job.out) scan_tile_sum(job.sc.counts, job.g->ncells, scan_tile_size(job.cap), job.sc.scan);
}
__global__ void __launch_bounds__(kScanThreads) k_grid_starts(const __grid_constant__ GridJobs J) {
  const GridJob &job = J.j[blockIdx.y];
  if (job.out) scan_tile_write(job.sc.counts, job.g->ncells, scan_tile_size(job.cap), job.sc.scan, job.start);
}

}  // namespace

int bbox_blocks(int n) { return (int)lsr_div_up(n > 0 ? n : 1, kBoxThreads * kBoxItems); }

cudaError_t launch_bbox_xyz(const float *xyz, int n, double *partials, int nblk_cap, float *box, cudaStream_t s) {
  int nb = bbox_blocks(n);
  if (nb > nblk_cap) return cudaErrorInvalidValue;
  LSR_LAUNCH(k_bbox_partial<<<nb, kBoxThreads, 0, s>>>(xyz, n, partials));
  LSR_LAUNCH(k_bbox_final<<<1, kBoxThreads, 0, s>>>(partials, nb, box));
  return cudaGetLastError();
}

int64_t nbmask_words(int cap_cells) { return cap_cells / 32 + 2; }

int64_t scan_scratch_ints(int64_t n) { return lsr_div_up(n + 1, kScanTile) + 64; }

cudaError_t scan_exclusive(const int *in, int *out, const int *n_dev, int cap, int *scratch, cudaStream_t s) {
  const int64_t tile = scan_tile_size(cap);
  const int nb = (int)lsr_div_up((int64_t)cap + 1, tile);
  LSR_LAUNCH(k_scan_sums<<<nb, kScanThreads, 0, s>>>(in, n_dev, tile, scratch));
  LSR_LAUNCH(k_scan_write<<<nb, kScanThreads, 0, s>>>(in, n_dev, tile, scratch, out));
  return cudaGetLastError();
}

cudaError_t build_grids(const GridJob *jobs, int count, cudaStream_t s) {
  for (int j0 = 0; j0 < count; j0 += kGridJobs) {
    GridJobs J{};
    const int nj = count - j0 < kGridJobs ? count - j0 : kGridJobs;
    int64_t words = 1, npts = 1, tiles = 1;
    int boxes = 0, grids = 0;
    for (int j = 0; j < nj; ++j) {
      const GridJob &q = J.j[j] = jobs[j0 + j];
      words = std::max(words, std::max((int64_t)q.cap + 1, q.zero_words));
      if (q.box_part) boxes = std::max(boxes, bbox_blocks(q.n));
      if (!q.out) continue;
      ++grids;
      npts = std::max(npts, (int64_t)q.n);
      tiles = std::max(tiles, lsr_div_up((int64_t)q.cap + 1, scan_tile_size(q.cap)));
    }
    const int zb = (int)std::min<int64_t>(lsr_div_up(words, 4 * 256), kSms * 8);
    const int pb = (int)lsr_div_up(npts, 256);
    LSR_LAUNCH(k_grid_begin<<<dim3(zb, nj), 256, 0, s>>>(J));
    if (boxes) LSR_LAUNCH(k_grid_bbox<<<dim3(boxes, nj), kBoxThreads, 0, s>>>(J));
    if (!grids) continue;
    LSR_LAUNCH(k_grid_slots<<<dim3(pb, nj), 256, 0, s>>>(J));
    LSR_LAUNCH(k_grid_sums<<<dim3((int)tiles, nj), kScanThreads, 0, s>>>(J));
    LSR_LAUNCH(k_grid_starts<<<dim3((int)tiles, nj), kScanThreads, 0, s>>>(J));
    LSR_LAUNCH(k_grid_scatter<<<dim3(pb, nj), 256, 0, s>>>(J));
    LSR_LAUNCH(k_grid_order<<<dim3(pb, nj), 256, 0, s>>>(J));
  }
  return cudaGetLastError();
}

}  // namespace lsr
