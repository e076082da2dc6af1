// lsr_surfel.cu -- dense model correction after a loop closure (eq. (7)).
//
// Every surfel moves with the keyframes that observe it: with F the keyframes
// f whose time stamp lies strictly between the surfel's initialisation and
// last-update stamps and whose camera (before the correction) sees the
// surfel -- in front of it, no farther than the maximum depth, projecting
// inside the image --
//   p' = (1/k) sum_f T_f_new T_f_old^-1 p,   n' = normalize(sum_f R_f_new R_f_old^-1 n),
// k = |F|; a surfel no keyframe observes is removed. Surfels do not interact.
// A keyframe's two 3 x 4 transforms are precomputed on the host in FP64 and
// stored in FP32; the time window is found by binary search over the sorted
// keyframe stamps. Up to kSurfTileKf keyframes fit in shared memory beside a
// tile of surfels (k_surfel_tile); with more, a thread per surfel reads the
// transforms through the read-only cache (k_surfel_correct), half as fast. Both
// give the same bits.
#include "lsr_internal.cuh"

namespace lsr {

namespace {

constexpr int kSurfThreads = 256;
constexpr int kSurfTileThreads = 512;
constexpr int kSurfTileKf = 600;  // keyframes of the tile kernel's table: 3 blocks an SM at 300, 2 at 600

__device__ __forceinline__ void xf34(const float *__restrict__ T, float x, float y, float z, float &ox, float &oy,
                                     float &oz) {
  ox = fmaf(__ldg(T + 0), x, fmaf(__ldg(T + 1), y, fmaf(__ldg(T + 2), z, __ldg(T + 3))));
  oy = fmaf(__ldg(T + 4), x, fmaf(__ldg(T + 5), y, fmaf(__ldg(T + 6), z, __ldg(T + 7))));
  oz = fmaf(__ldg(T + 8), x, fmaf(__ldg(T + 9), y, fmaf(__ldg(T + 10), z, __ldg(T + 11))));
}

__global__ void __launch_bounds__(kSurfThreads) k_surfel_correct(int64_t n, const float *__restrict__ pos,
                                                                 const float *__restrict__ nrm,
                                                                 const float *__restrict__ t0,
                                                                 const float *__restrict__ tu, int m,
                                                                 const KfPose *__restrict__ kf,
                                                                 const float *__restrict__ t_kf, SurfelCam cam,
                                                                 float *__restrict__ pos_out,
                                                                 float *__restrict__ nrm_out,
                                                                 uint8_t *__restrict__ keep,
                                                                 unsigned long long *__restrict__ n_keep) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float px = pos[3 * i], py = pos[3 * i + 1], pz = pos[3 * i + 2];
    const float nx = nrm[3 * i], ny = nrm[3 * i + 1], nz = nrm[3 * i + 2];
    const float a = t0[i], b = tu[i];
    // first keyframe with t_f > t0
    int lo = 0, hi = m;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (__ldg(t_kf + mid) > a) hi = mid; else lo = mid + 1;
    }
    int k = 0;
    float sx = 0.f, sy = 0.f, sz = 0.f, qx = 0.f, qy = 0.f, qz = 0.f;
    for (int f = lo; f < m && __ldg(t_kf + f) < b; ++f) {
      float cx, cy, cz;
      xf34(kf[f].A, px, py, pz, cx, cy, cz);
      if (!(cz > 0.f && cz <= cam.dmax)) continue;
      const float u = cam.fx * cx / cz + cam.cx, v = cam.fy * cy / cz + cam.cy;
      if (!(u >= 0.f && u < cam.w && v >= 0.f && v < cam.h)) continue;
      float ox, oy, oz;
      xf34(kf[f].M, px, py, pz, ox, oy, oz);
      sx += ox, sy += oy, sz += oz;
      const float *R = kf[f].M;
      qx += fmaf(__ldg(R + 0), nx, fmaf(__ldg(R + 1), ny, __ldg(R + 2) * nz));
      qy += fmaf(__ldg(R + 4), nx, fmaf(__ldg(R + 5), ny, __ldg(R + 6) * nz));
      qz += fmaf(__ldg(R + 8), nx, fmaf(__ldg(R + 9), ny, __ldg(R + 10) * nz));
      ++k;
    }
    const bool kept = k > 0;
    float op[3] = {px, py, pz}, on[3] = {nx, ny, nz};
    if (kept) {
      const float ik = 1.f / (float)k;
      op[0] = sx * ik, op[1] = sy * ik, op[2] = sz * ik;
      const float il = rsqrtf(fmaxf(qx * qx + qy * qy + qz * qz, 1e-30f));
      on[0] = qx * il, on[1] = qy * il, on[2] = qz * il;
    }
    for (int d = 0; d < 3; ++d) pos_out[3 * i + d] = op[d], nrm_out[3 * i + d] = on[d];
    keep[i] = kept ? 1 : 0;
    const unsigned ballot = __ballot_sync(__activemask(), kept);
    if (ballot && (threadIdx.x & 31) == __ffs(__activemask()) - 1) atomicAdd(n_keep, (unsigned long long)__popc(ballot));
  }
}

// The same correction for a keyframe table that fits in shared memory. The
// kernel above reads 12 to 24 scalars per (surfel, keyframe) through L1 with a
// different keyframe on every lane (map order says nothing about time), and
// that gather bound it: 869 us for 2M surfels and 300 keyframes, L1 at 88%,
// 114 MB of traffic worth 17 us (the whole call 967 us, 412 with this kernel).
// Here a block takes a tile of surfels, sorts the tile by first keyframe (a
// counting sort in shared memory), and a warp walks 32 neighbours of that order through the union of their windows one
// keyframe at a time: the keyframe is the same on every lane, so its rows are
// broadcasts. A window is 20 keyframes and the union about 50 (the spread of
// 32 of 1024 first keyframes, and the longest window), so half the lanes idle;
// they cost less than the gathers. Positions and normals pass through shared
// memory so that the tile is read and written in whole lines. Every surfel
// still adds its keyframes in ascending order: the same sums.
template <int kItems>
__global__ void __launch_bounds__(kSurfTileThreads, 3) k_surfel_tile(int64_t n, const float *__restrict__ pos,
                                                                  const float *__restrict__ nrm,
                                                                  const float *__restrict__ t0,
                                                                  const float *__restrict__ tu, int m,
                                                                  const KfPose *__restrict__ kf,
                                                                  const float *__restrict__ t_kf, SurfelCam cam,
                                                                  float *__restrict__ pos_out,
                                                                  float *__restrict__ nrm_out,
                                                                  uint8_t *__restrict__ keep,
                                                                  unsigned long long *__restrict__ n_keep) {
  constexpr int kTile = kSurfTileThreads * kItems;
  extern __shared__ float4 sf_smem[];
  float4 *tab = sf_smem;                                        // m x (A, M), three float4 each
  float *sp = reinterpret_cast<float *>(tab + 6 * (size_t)m);   // kTile positions, then normals, in place
  float *sn = sp + 3 * kTile;
  float *st = sn + 3 * kTile;                                   // m stamps
  int *hist = reinterpret_cast<int *>(st + m);                  // m + 1 buckets
  int *win = hist + m + 1;                                      // kTile windows: first keyframe | end << 16
  uint16_t *order = reinterpret_cast<uint16_t *>(win + kTile);
  uint8_t *sk = reinterpret_cast<uint8_t *>(order + kTile);
  __shared__ int s_warp[kSurfTileThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int k = tid; k < 6 * m; k += kSurfTileThreads) tab[k] = __ldg(reinterpret_cast<const float4 *>(kf) + k);
  for (int k = tid; k < m; k += kSurfTileThreads) st[k] = __ldg(t_kf + k);
  int kept_sum = 0;
  for (int64_t base = (int64_t)blockIdx.x * kTile; base < n; base += (int64_t)gridDim.x * kTile) {
    const int cnt = (int)(n - base < kTile ? n - base : kTile);
    __syncthreads();  // the previous tile has left; the table is in
    for (int k = tid; k <= m; k += kSurfTileThreads) hist[k] = 0;
    for (int k = tid; k < 3 * cnt; k += kSurfTileThreads) sp[k] = pos[3 * base + k], sn[k] = nrm[3 * base + k];
    __syncthreads();
    int key[kItems], rank[kItems];
#pragma unroll
    for (int u = 0; u < kItems; ++u) {
      const int j = u * kSurfTileThreads + tid;
      key[u] = m;
      rank[u] = 0;
      if (j < cnt) {
        const float a = t0[base + j], b = tu[base + j];
        // the window: from the first keyframe with t_f > t0 to the first with t_f >= tu
        int lo = 0, hi = m;
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (st[mid] > a) hi = mid; else lo = mid + 1;
        }
        int e = lo, eh = m;
        while (e < eh) {
          const int mid = (e + eh) >> 1;
          if (!(st[mid] < b)) eh = mid; else e = mid + 1;
        }
        key[u] = e > lo ? lo : m;  // surfels without a window come last
        win[j] = e > lo ? lo | (e << 16) : 0;
        rank[u] = atomicAdd(hist + key[u], 1);
      }
    }
    __syncthreads();
    // exclusive scan of the m + 1 buckets, a run per thread
    {
      const int per = (m + kSurfTileThreads) / kSurfTileThreads;
      const int k0 = min(tid * per, m + 1), k1 = min(k0 + per, m + 1);
      int s = 0;
      for (int k = k0; k < k1; ++k) s += hist[k];
      int x = s;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (lane == 31) s_warp[warp] = x;
      __syncthreads();
      int run = x - s;
      for (int w = 0; w < warp; ++w) run += s_warp[w];
      for (int k = k0; k < k1; ++k) {
        const int c = hist[k];
        hist[k] = run;
        run += c;
      }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kItems; ++u) {
      const int j = u * kSurfTileThreads + tid;
      if (j < cnt) order[hist[key[u]] + rank[u]] = (uint16_t)j;
    }
    __syncthreads();
    for (int g = 32 * warp; g < cnt; g += kSurfTileThreads) {
      const bool in = g + lane < cnt;
      const int j = in ? order[g + lane] : 0;
      const int w = in ? win[j] : 0;
      const int lo = w & 0xffff, hi = w >> 16;
      const float px = sp[3 * j], py = sp[3 * j + 1], pz = sp[3 * j + 2];
      const float nx = sn[3 * j], ny = sn[3 * j + 1], nz = sn[3 * j + 2];
      int k = 0;
      float sx = 0.f, sy = 0.f, sz = 0.f, qx = 0.f, qy = 0.f, qz = 0.f;
      const int f0 = __reduce_min_sync(0xffffffffu, hi > lo ? lo : m), f1 = __reduce_max_sync(0xffffffffu, hi);
      for (int f = f0; f < f1; ++f) {
        const float4 *T = tab + 6 * f;
        const float4 a2 = T[2];
        const float cz = fmaf(a2.x, px, fmaf(a2.y, py, fmaf(a2.z, pz, a2.w)));
        bool see = f >= lo && f < hi && cz > 0.f && cz <= cam.dmax;
        if (!__any_sync(0xffffffffu, see)) continue;
        const float4 a0 = T[0], a1 = T[1];
        const float cx = fmaf(a0.x, px, fmaf(a0.y, py, fmaf(a0.z, pz, a0.w)));
        const float cy = fmaf(a1.x, px, fmaf(a1.y, py, fmaf(a1.z, pz, a1.w)));
        if (see) {
          const float u = cam.fx * cx / cz + cam.cx, v = cam.fy * cy / cz + cam.cy;
          see = u >= 0.f && u < cam.w && v >= 0.f && v < cam.h;
        }
        if (!__any_sync(0xffffffffu, see)) continue;
        const float4 m0 = T[3], m1 = T[4], m2 = T[5];
        if (see) {
          sx += fmaf(m0.x, px, fmaf(m0.y, py, fmaf(m0.z, pz, m0.w)));
          sy += fmaf(m1.x, px, fmaf(m1.y, py, fmaf(m1.z, pz, m1.w)));
          sz += fmaf(m2.x, px, fmaf(m2.y, py, fmaf(m2.z, pz, m2.w)));
          qx += fmaf(m0.x, nx, fmaf(m0.y, ny, m0.z * nz));
          qy += fmaf(m1.x, nx, fmaf(m1.y, ny, m1.z * nz));
          qz += fmaf(m2.x, nx, fmaf(m2.y, ny, m2.z * nz));
          ++k;
        }
      }
      if (in) {
        if (k > 0) {
          const float ik = 1.f / (float)k;
          sp[3 * j] = sx * ik, sp[3 * j + 1] = sy * ik, sp[3 * j + 2] = sz * ik;
          const float il = rsqrtf(fmaxf(qx * qx + qy * qy + qz * qz, 1e-30f));
          sn[3 * j] = qx * il, sn[3 * j + 1] = qy * il, sn[3 * j + 2] = qz * il;
          ++kept_sum;
        }
        sk[j] = k > 0 ? 1 : 0;
      }
    }
    __syncthreads();
    for (int k = tid; k < 3 * cnt; k += kSurfTileThreads) pos_out[3 * base + k] = sp[k], nrm_out[3 * base + k] = sn[k];
    for (int k = tid; k < cnt; k += kSurfTileThreads) keep[base + k] = sk[k];
  }
  kept_sum = warp_sum(kept_sum);
  if (lane == 0 && kept_sum) atomicAdd(n_keep, (unsigned long long)kept_sum);
}

template <int kItems>
size_t surfel_tile_smem(int m) {
  constexpr size_t kTile = (size_t)kSurfTileThreads * kItems;
  return 96 * (size_t)m + 24 * kTile + 4 * (size_t)m + 4 * (size_t)(m + 1) + 4 * kTile + 2 * kTile + kTile;
}

}  // namespace

cudaError_t launch_surfel_correct(int64_t n, const float *pos, const float *nrm, const float *t0, const float *tu,
                                  int m, const KfPose *kf, const float *t_kf, const SurfelCam &cam, float *pos_out,
                                  float *nrm_out, uint8_t *keep, unsigned long long *n_keep, cudaStream_t s) {
  LSR_CUDA_TRY(cudaMemsetAsync(n_keep, 0, sizeof(unsigned long long), s));
  if (m <= kSurfTileKf) {
    // tiles of 1024 surfels; of 512 while those of 1024 would not fill the GPU three blocks deep
    const bool big = n >= (int64_t)kSms * 3 * 1024;
    const size_t smem = big ? surfel_tile_smem<2>(m) : surfel_tile_smem<1>(m);
    const int64_t tiles = lsr_div_up(n, big ? 1024 : 512);
    const int grid = (int)(tiles < kSms * 3 ? tiles : kSms * 3);
    auto kern = big ? k_surfel_tile<2> : k_surfel_tile<1>;
    // the limit belongs to the function on the device, which contexts on other
    // threads launch too: always the one for the largest table, never the call's own
    const size_t limit = big ? surfel_tile_smem<2>(kSurfTileKf) : surfel_tile_smem<1>(kSurfTileKf);
    LSR_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit));
    LSR_LAUNCH(kern<<<grid, kSurfTileThreads, smem, s>>>(n, pos, nrm, t0, tu, m, kf, t_kf, cam, pos_out, nrm_out, keep,
                                                         n_keep));
    return cudaGetLastError();
  }
  const int64_t nb = lsr_div_up(n, kSurfThreads);
  const int blocks = (int)(nb < 1 ? 1 : (nb > kSms * 16 ? kSms * 16 : nb));
  LSR_LAUNCH(k_surfel_correct<<<blocks, kSurfThreads, 0, s>>>(n, pos, nrm, t0, tu, m, kf, t_kf, cam, pos_out, nrm_out,
                                                               keep, n_keep));
  return cudaGetLastError();
}

}  // namespace lsr
