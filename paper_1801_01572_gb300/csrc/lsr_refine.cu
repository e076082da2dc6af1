// lsr_refine.cu -- robust pose refinement and the robust alignment objective.
//
// The cost is the line-process objective of eq. (3)-(4) with the line process
// eliminated: for a residual r, min_l l r^2 + mu (sqrt(l) - 1)^2 is reached at
// l* = (mu / (mu + r^2))^2 and equals the Geman-McClure rho(r^2) = mu r^2 /
// (mu + r^2). Refinement iterates reweighted Gauss-Newton with the Jacobian
// G_p = [-[p]_x | I] of eq. (5), taken about a linearisation centre c (the
// weighted centroid of the current correspondences, so that FP32 stays exact
// to the micrometre whatever the clouds' offset): FP32 per-thread and
// per-block sums, then one launch-closing block sums the block partials in
// FP64 in a fixed order, solves the 6x6 system (Schur complement of its
// translation block, then a 3x3 adjugate) and updates the
// FP64 pose -- one kernel launch per iteration, no host round trip.
#include "lsr_internal.cuh"

namespace lsr {

namespace {

constexpr int kRefThreads = 256;
constexpr int kRefG = 4;   // lanes per nearest-neighbour query in refinement (4 measured fastest of 4/8/16)
constexpr int kRefBlocksPerSm = 4;  // resident refinement blocks per SM (64 registers a thread; 3 measured slower)
constexpr int kRefMaxBlocks = kSms * kRefBlocksPerSm;  // refine_blocks' cap
constexpr int kRefGroup = 16;                           // blocks summed together when a step closes
constexpr int kRefMaxGroups = (kRefMaxBlocks + kRefGroup - 1) / kRefGroup;
constexpr int kRefAtOnce = 8;                           // groups summed by the last block alone
static_assert(kRefAtOnce <= kRefThreads / 17, "a segment per group");
// 21 (upper triangle of A) + 6 (b) + count + sum w + sum w x (3)
constexpr int kNAcc = kRefAcc;
static_assert(kNAcc == 32, "refinement partial layout");

template <int N>
__device__ __forceinline__ void block_reduce_to(float (&v)[N], double *out) {
  __shared__ float sm[kRefThreads / 32][N];
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < N; ++k) v[k] = warp_sum(v[k]);
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < N; ++k) sm[w][k] = v[k];
  __syncthreads();
  if (threadIdx.x < N) {
    double s = 0.0;
    for (int k = 0; k < kRefThreads / 32; ++k) s += (double)sm[k][threadIdx.x];
    out[threadIdx.x] = s;
  }
}

// Per-step sums of the IRLS normal equations. With J = [-[xc]_x | I] (xc the
// moved point about the step's centre c), w the line-process weight of eq. (4)
// and r the residual, J^T W J and J^T W r need only these 17 sums:
//   [0] count  [1] sum w  [2..4] sum w xc  [5..10] sum w xc_a xc_b (00 01 02 11 12 22)
//   [11..16] b = sum w J^T r = (sum w xc x r, sum w r)
constexpr int kNSum = 17;
static_assert(kNSum <= kNAcc, "refinement partial layout");

// The state one step reads, copied to shared memory by the closing block
// while it sums the partials (its loads then overlap instead of queueing
// behind each other in the single solving thread).
struct StepState {
  double T[12];
  double center[3];
  int iters_done;
  int level_iters;
};

// 1 / x in FP64 for a positive x: the FP32 reciprocal refined by two Newton-
// Raphson steps r <- r + r (1 - x r) (each doubles the correct bits: 24 ->
// 48 -> 96, so the result is within an ulp of 1 / x); outside the FP32 range
// the FP64 division. A division costs far more FP64 latency on this part
// than the four fused multiply-adds.
__device__ __forceinline__ double recip_pos(double x) {
  if (!(x > 1e-30 && x < 1e30)) return 1.0 / x;
  double r = (double)__frcp_rn((float)x);
  r = fma(r, fma(-x, r, 1.0), r);
  r = fma(r, fma(-x, r, 1.0), r);
  return r;
}

// Solve A d = -b in FP64 from the summed partials and left-multiply the pose
// by the update about the centre c used for this step: x' = Exp(d_w)(x - c) +
// c + d_v. The next step's centre is the weighted centroid of this step's
// correspondences. Reads the state from ss, writes it to st.
//
// With J = [-[xc]_x | I], A = [[M, [s]_x], [[s]_x^T, sw I]] where M is the
// rotation block, s = sum w xc and sw = sum w. The translation block is a
// multiple of I, so it is eliminated in closed form (Schur complement):
//   M' = M - (|s|^2 I - s s^T) / sw,
//   M' d_w = -b_w + (s x b_v) / sw,   d_v = -(b_v - s x d_w) / sw,
// and the 3x3 system is solved by its adjugate (one reciprocal). A is
// positive definite iff sw > 0 and M' is (its leading minors positive).
//
// Bound by the latency of its chain of FP64 operations (a warp instruction
// every 16 clocks at best, one lane or all): both sides of the 3x3 system are
// multiplied by sw (times a power of two that brings it to [1, 2), so that the
// determinant stays in range) instead of waiting for 1 / sw, the terms of each
// stage are computed a lane each and exchanged by shuffles, and the series of
// Exp are Horner chains: about 30 dependent operations; with one lane
// computing all of it in 47 the solve took 4.9 us (now 2.9). Run by one warp; every value is
// computed in a fixed order. S[kNSum] is 0.
__device__ __forceinline__ double lane_of(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ int field(unsigned long long packed, int lane) { return (int)(packed >> (5 * lane)) & 31; }
// Nine five-bit fields.
__host__ __device__ constexpr unsigned long long fields(int a, int b, int c, int d, int e, int f, int g = 0, int h = 0,
                                                        int i = 0) {
  const int v[9] = {a, b, c, d, e, f, g, h, i};
  unsigned long long p = 0;
  for (int k = 0; k < 9; ++k) p |= (unsigned long long)v[k] << (5 * k);
  return p;
}

__device__ void refine_solve(const double *S, const StepState &ss, RansacState *st, int max_iters, double tol) {
  const int lane = threadIdx.x & 31, j = lane < 9 ? lane : 0;
  const double sw = S[1];
  if (!(S[0] >= 3.0 && sw > 0.0)) {
    if (lane == 0) st->active = 0;
    return;
  }
  // lanes 0..5: M' (00 01 02 11 12 22), 6..8: the right-hand side, times sw f:
  // sw f (base) + f (S S + S S)
  constexpr int Z = kNSum;  // S[Z] = 0
  constexpr unsigned long long kBase = fields(8, 6, 7, 5, 9, 5, 11, 12, 13), kMore = fields(10, Z, Z, 10, Z, 8, Z, Z, Z);
  constexpr unsigned long long kP = fields(3, 2, 2, 2, 3, 2, 3, 4, 2), kQ = fields(3, 3, 4, 2, 4, 2, 16, 14, 15);
  constexpr unsigned long long kU = fields(4, Z, Z, 4, Z, 3, 4, 2, 3), kV = fields(4, Z, Z, 4, Z, 3, 15, 16, 14);
  const bool diag = j == 0 || j == 3 || j == 5;
  // f = 2^-e for sw in [2^e, 2^(e + 1))
  const double f = __longlong_as_double((long long)(2046 - ((__double_as_longlong(sw) >> 52) & 2047)) << 52);
  const double base = S[field(kBase, j)] + S[field(kMore, j)];
  const double P = S[field(kP, j)] * (diag ? -f : f), U = S[field(kU, j)] * -f;
  const double e = fma(diag ? base : -base, sw * f, fma(P, S[field(kQ, j)], U * S[field(kV, j)]));
  const double iw = recip_pos(sw);
  // lanes 0..5: cofactors (00 01 02 11 12 22)
  constexpr unsigned long long kA = fields(3, 2, 1, 0, 1, 0), kB = fields(5, 4, 4, 5, 2, 3);
  constexpr unsigned long long kC = fields(4, 1, 2, 2, 0, 1), kD4 = fields(4, 5, 3, 2, 4, 1);
  const double cof = fma(lane_of(e, field(kA, j)), lane_of(e, field(kB, j)), -(lane_of(e, field(kC, j)) * lane_of(e, field(kD4, j))));
  // lanes 0..2: rows of the adjugate times the right-hand side; 3: the determinant
  constexpr unsigned long long kR0 = fields(0, 1, 2, 0, 0, 0), kR1 = fields(1, 3, 4, 1, 0, 0), kR2 = fields(2, 4, 5, 2, 0, 0);
  const int v = j == 3 ? 0 : 6;  // what the row meets: M' or the right-hand side
  const double num = fma(lane_of(cof, field(kR2, j)), lane_of(e, v + 2),
                         fma(lane_of(cof, field(kR1, j)), lane_of(e, v + 1), lane_of(cof, field(kR0, j)) * lane_of(e, v)));
  const double det = lane_of(num, 3);
  if (!(lane_of(e, 0) > 0.0 && lane_of(cof, 5) > 0.0 && det > 0.0)) {
    if (lane == 0) st->active = 0;
    return;
  }
  const double wl = num * recip_pos(det);
  const double w0 = lane_of(wl, 0), w1 = lane_of(wl, 1), w2 = lane_of(wl, 2);
  // Exp of the rotation part: the series of sin(t)/t and (1 - cos t)/t^2 to
  // the t^8 term below t = 0.01 (the next term is below 1e-21), else sin/cos
  const double t2 = fma(w2, w2, fma(w1, w1, w0 * w0));
  double ea, eb;
  if (t2 < 1e-4) {
    ea = fma(t2, fma(t2, fma(t2, fma(t2, 1.0 / 362880.0, -1.0 / 5040.0), 1.0 / 120.0), -1.0 / 6.0), 1.0);
    eb = fma(t2, fma(t2, fma(t2, fma(t2, 1.0 / 3628800.0, -1.0 / 40320.0), 1.0 / 720.0), -1.0 / 24.0), 0.5);
  } else {
    const double th = sqrt(t2);
    ea = sin(th) / th;
    eb = (1.0 - cos(th)) / t2;
  }
  // lane 4 r + q < 12: pose entry (r, q); p, o: the two axes after r
  const int r = lane < 12 ? lane >> 2 : 0, q = lane & 3, p = r == 2 ? 0 : r + 1, o = p == 2 ? 0 : p + 1;
  const double wr = r == 0 ? w0 : r == 1 ? w1 : w2, wp = r == 0 ? w1 : r == 1 ? w2 : w0, wo = r == 0 ? w2 : r == 1 ? w0 : w1;
  // row r of Rd = I + a [w]_x + b [w]_x^2, and of d_v
  const double Rr = fma(-eb, fma(wp, wp, wo * wo), 1.0), Rp = fma(eb, wr * wp, -(ea * wo)), Ro = fma(eb, wr * wo, ea * wp);
  const double dv = -(S[14 + r] - (S[2 + p] * wo - S[2 + o] * wp)) * iw;
  const double *c = ss.center;
  const double vr = c[r] - fma(Ro, c[o], fma(Rp, c[p], Rr * c[r])) + dv;
  if (lane < 12) st->T[lane] = fma(Ro, ss.T[4 * o + q], fma(Rp, ss.T[4 * p + q], fma(Rr, ss.T[4 * r + q], q == 3 ? vr : 0.0)));
  if (lane < 12 && q == 0) st->center[r] = fma(S[2 + r], iw, c[r]);
  const double dv1 = lane_of(dv, 4), dv2 = lane_of(dv, 8);
  if (lane == 0) {
    const double nd2 = t2 + fma(dv2, dv2, fma(dv1, dv1, dv * dv));
    st->iters_done = ss.iters_done + 1;
    st->level_iters = ss.level_iters + 1;
    if (nd2 < tol * tol || ss.level_iters + 1 >= max_iters) st->active = 0;
  }
}

// A distance that no point outside the 3 x 3 x 3 block of cells around the cell
// coordinates (fx, fy, fz) is closer than: at least a cell beyond the query's
// own; for a query outside the box (where nothing is visited) the distance to it.
__device__ __forceinline__ float nn_border(const GridParams &g, float fx, float fy, float fz) {
  const float ux = fx - floorf(fx), uy = fy - floorf(fy), uz = fz - floorf(fz);
  const float in = fminf(fminf(fminf(ux, 1.f - ux), fminf(uy, 1.f - uy)), fminf(uz, 1.f - uz));
  const float out = fmaxf(fmaxf(fmaxf(-fx, fx - (float)g.nx), fmaxf(-fy, fy - (float)g.ny)), fmaxf(-fz, fz - (float)g.nz));
  return fmaxf(1.f + in, out) * g.cell - 2.f * g.margin;
}

// The result of group_nn (at: the position in Xe, -1 if none), and a distance
// that no other point is closer than (no point at all, if at = -1): the second
// smallest distance seen, the bound up to which cells were visited (the seed's
// or eps plus guard) and the distance to the border of the 3 x 3 x 3 block,
// whichever is least, less a margin of 4e-6 of it (above the FP32 rounding of
// the distances).
struct Found {
  int at;
  float apart;
};

// Half a warp a query (grids without wrapped storage). Its lanes read the mask
// and the nine rows' ranges at once and then walk the candidates of all rows
// together, four a lane in flight, so a search is two to four dependent loads
// long (1.5 us) instead of two or more for each row. seed2: the squared distance
// of the seed (below eps2), which the walk meets again; none: eps2 and -1. Not
// inlined: the registers that the caller holds for its point were spilled
// around the loads, and a search took 9 us.
constexpr int kRefH = 16;
__device__ __noinline__ Found half_nn(const GridParams &g, const int *__restrict__ start,
                                      const float4 *__restrict__ Xe, float x, float y, float z, float seed2, int seed,
                                      float guard) {
  const int sub = threadIdx.x & (kRefH - 1);
  float best = seed2, m1 = 3e38f, m2 = 3e38f, reach2 = 3e38f;
  int bidx = 0x7fffffff, bt = seed;
  const float mg = g.margin;
  const float fx = (x - g.ox) * g.inv_cell, fy = (y - g.oy) * g.inv_cell, fz = (z - g.oz) * g.inv_cell;
  bool go = fx >= -1.f && fx < (float)g.nx + 1.f && fy >= -1.f && fy < (float)g.ny + 1.f && fz >= -1.f &&
            fz < (float)g.nz + 1.f;
  const int cx = go ? __float2int_rd(fx) : 0, cy = go ? __float2int_rd(fy) : 0, cz = go ? __float2int_rd(fz) : 0;
  const int x0 = cx - 1 < 0 ? 0 : cx - 1, x1 = cx + 1 > g.nx - 1 ? g.nx - 1 : cx + 1;
  go = go && x0 <= x1;
  unsigned mask = 0xffffffffu;
  if (go && g.nbmask && cx >= 0 && cx < g.nx && cy >= 0 && cy < g.ny && cz >= 0 && cz < g.nz) {
    const int slot = (cz * g.wy + cy) * g.wx + cx;
    mask = __ldg(g.nbmask + (slot >> 5)) >> (slot & 31);
  }
  constexpr float kShrink = 1.f - 1e-6f;  // the FP32 rounding of d^2 itself
  // lane sub < 9: a row of cells and the part of it within reach
  int b = 0, len = 0;
  if (go) {
    const float r = sqrtf(best) + guard, gb = r * r;
    const int dy = sub % 3 - 1, dz = sub / 3 - 1, iy = cy + dy, iz = cz + dz;
    if (sub < 9 && iy >= 0 && iy < g.ny && iz >= 0 && iz < g.nz) {
      auto gsq = [&](float d) {
        const float t = fmaxf(d - mg, 0.f);
        return t * t;
      };
      const float ux = fx - (float)cx, uy = fy - (float)cy, uz = fz - (float)cz;
      const float r2 = (dy < 0 ? gsq(uy * g.cell) : dy > 0 ? gsq((1.f - uy) * g.cell) : 0.f) +
                       (dz < 0 ? gsq(uz * g.cell) : dz > 0 ? gsq((1.f - uz) * g.cell) : 0.f);
      int a = x0, e = x1;
      if (a < cx && (r2 + gsq(ux * g.cell)) * kShrink > gb) a = cx;
      if (e > cx && (r2 + gsq((1.f - ux) * g.cell)) * kShrink > gb) e = cx;
      const int row = (iz * g.wy + iy) * g.wx;
      if (!(r2 * kShrink > gb) && a <= e && LSR_IN_BOUNDS(row + e + 1, g.ncells + 1, kSiteGridRow) &&
          LSR_IN_BOUNDS(row + a, g.ncells + 1, kSiteGridRow)) {
        b = start[row + a], len = start[row + e + 1] - b;
        if (len > 0 && (!LSR_IN_BOUNDS(b + len - 1, g.npts, kSiteGridPoint) || !LSR_IN_BOUNDS(b, g.npts, kSiteGridPoint)))
          len = 0;
      }
    }
    if (mask & 1u) reach2 = gb * kShrink;
    else len = 0;  // nothing in the block
  }
  // the rows' candidates numbered through: row k's end at its lane's end
  int end = len;
#pragma unroll
  for (int off = 1; off < kRefH; off <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, end, off, kRefH);
    if (sub >= off) end += o;
  }
  const int total = __shfl_sync(0xffffffffu, end, kRefH - 1, kRefH), shift = b - (end - len);
  const int most = max(total, __shfl_xor_sync(0xffffffffu, total, kRefH));
  int ends[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) ends[k] = __shfl_sync(0xffffffffu, end, k, kRefH);
#pragma unroll 1
  for (int t0 = sub; t0 - sub < most; t0 += 4 * kRefH) {
    int at[4];
    float4 q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int t = t0 + u * kRefH;
      int row = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) row += t >= ends[k];
      at[u] = t + __shfl_sync(0xffffffffu, shift, row, kRefH);
      q[u] = make_float4(3e18f, 0.f, 0.f, 0.f);  // out of everyone's reach
      if (t < total) q[u] = Xe[at[u]];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float d2 = nn_d2(q[u], x, y, z);
      m2 = fminf(m2, fmaxf(m1, d2)), m1 = fminf(m1, d2);
      const int qi = __float_as_int(q[u].w);
      if (d2 < best || (d2 == best && qi < bidx)) best = d2, bt = at[u], bidx = qi;
    }
  }
#pragma unroll
  for (int off = kRefH / 2; off > 0; off >>= 1) {
    const float ob = __shfl_xor_sync(0xffffffffu, best, off);
    const int ot = __shfl_xor_sync(0xffffffffu, bt, off);
    const int oi = __shfl_xor_sync(0xffffffffu, bidx, off);
    if (ob < best || (ob == best && oi < bidx)) best = ob, bt = ot, bidx = oi;
    const float o1 = __shfl_xor_sync(0xffffffffu, m1, off), o2 = __shfl_xor_sync(0xffffffffu, m2, off);
    m2 = fminf(fmaxf(m1, o1), fminf(m2, o2)), m1 = fminf(m1, o1);
  }
  const float other = bt >= 0 && m1 <= best ? m2 : m1;  // (m1 is the best itself)
  return {bt, fminf(sqrtf(fminf(other, reach2)), nn_border(g, fx, fy, fz)) * (1.f - 4e-6f)};
}

// Wrapped storage: the general walk, which vouches for nothing.
__device__ __noinline__ Found group_nn_wrapped(const GridParams &g, const int *__restrict__ start,
                                               const float4 *__restrict__ Xe, float x, float y, float z, float eps2,
                                               int seed) {
  float best;
  int bt, bidx;
  group_nn<kRefH>(g, &g.margin, start, Xe, x, y, z, eps2, best, bt, bidx, seed);
  return {bt, 0.f};
}

// One IRLS step. Every block accumulates its points; the last block to
// finish (atomic ticket, no waiting) sums all block partials and solves.
//
// Most steps move the points by far less than the gap between their nearest
// and second nearest Q point, so most searches would find what the last one
// found. A search therefore also leaves where it was made and a distance that
// no other point is closer than (Found); by the triangle inequality
// the neighbour stands while its distance now is below that distance less the
// way moved since, and there is still none while eps is. A block first decides
// that with a point per thread, lists the points that need a search, searches
// those with half a warp each, and a point per thread then lays out the values
// whose products the sums take. The neighbours are those of a search of every
// point. With a search of every point each step was bound by the latency of
// the grid walks (42 us of 55 at 150k points).
// Bound by a chain of latencies now, whatever the points: a settled step of 50k
// takes 17.5 us from its first load (pose and values 2.5, searches 3.5, sums 1.5,
// the two tickets 3, closing sums 2.7, solve 2.9; 12.6 for 4k points).
// near[i]: the neighbour and its position in Xe, or kSeedNone or kSeedFresh (no
// search yet at this level) there; certs[i]: where the search was made and the
// distance. Neither needs a gather, and the loads of a point's values do not
// wait for the pose.
//
// A block's points are the runs of kRefSlots points numbered blockIdx.x,
// + gridDim.x, ..., kRefRuns of them at a time; the 17 sums of each slot go
// through the runs in order (four lanes a slot, every fourth sum each), then
// over the slots.
constexpr int kSeedFresh = -1, kSeedNone = -2;
// Cells are visited up to this part of eps beyond the nearest point (half of it or
// twice it: 2 and 6% slower at 50k points).
constexpr float kRefGuard = 0.125f;
constexpr int kRefSlots = 64, kRefRuns = kRefThreads / kRefSlots;
// The values of a point: 1, w, w xc (3), xc (3), xc x e (3), e (3), or all 0
// without a neighbour; sum k takes the products of kTermA[k] and kTermB[k].
constexpr int kNVal = 14;
__constant__ const unsigned char kTermA[20] = {0, 1, 2, 3, 4, 2, 2, 2, 3, 3, 4, 1, 1, 1, 1, 1, 1, 0, 0, 0};
__constant__ const unsigned char kTermB[20] = {0, 0, 0, 0, 0, 5, 6, 7, 6, 7, 7, 8, 9, 10, 11, 12, 13, 0, 0, 0};

__global__ void __launch_bounds__(kRefThreads, kRefBlocksPerSm) k_refine_step(const float4 *__restrict__ XP, int nP,
                                                             const GridParams *gep, const int *__restrict__ start,
                                                             const float4 *__restrict__ Xe, float eps, float mu,
                                                             RansacState *st, double *partials, int max_iters,
                                                             double tol, float4 *__restrict__ near,
                                                             float4 *__restrict__ certs) {
  __shared__ int s_last, s_need;
  __shared__ double tot[kNSum + 1];  // the last is 0 (refine_solve)
  __shared__ GridParams s_grid;
  __shared__ float s_pose[15];  // rotation, centre, translation less the centre
  __shared__ float4 s_query[kRefThreads];  // the points to search: position, thread
  __shared__ int s_found[kRefThreads];     // per thread: its seed, then its neighbour
  __shared__ float s_seed2[kRefThreads];   // the seed's squared distance
  __shared__ float s_val[kNVal][kRefThreads + 8];
  // the next step may be scheduled now (launched as a programmatic dependent,
  // it waits below for this one to finish); this step reads the pose, the
  // state and the neighbours the previous step wrote
  asm volatile("griddepcontrol.launch_dependents;");
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int run = gridDim.x * kRefSlots;  // points from one run of this block to its next
  const int own = (threadIdx.x / kRefSlots) * run + (threadIdx.x % kRefSlots);
  float4 p = make_float4(0.f, 0.f, 0.f, 0.f), at = p, nr = p;
  int i = blockIdx.x * kRefSlots + own;
  if (i < nP) p = XP[i];
  static_assert(sizeof(GridParams) % 4 == 0 && sizeof(GridParams) <= 128, "a lane per word");
  if (threadIdx.x < sizeof(GridParams) / 4)
    reinterpret_cast<int *>(&s_grid)[threadIdx.x] = reinterpret_cast<const int *>(gep)[threadIdx.x];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (i < nP) at = certs[i], nr = near[i];
  // a lane per entry of the pose: the FP64 unit takes a warp instruction every
  // 16 clocks, and eighteen of them in each of an SM's 32 warps took 4.8 us
  if (threadIdx.x < 15) {
    const int k = threadIdx.x, r = k < 9 ? k / 3 : (k - 9) % 3;
    const double c = __ldcg(st->center + r);
    s_pose[k] = (float)(k < 9 ? __ldcg(st->T + 4 * r + k % 3) : k < 12 ? c : __ldcg(st->T + 4 * r + 3) - c);
  }
  if (threadIdx.x == 0) s_need = 0;
  if (!st->active) return;
  const float eps2 = eps * eps;
  __syncthreads();
  const bool wrapped = (s_grid.wx != s_grid.nx) | (s_grid.wy != s_grid.ny) | (s_grid.wz != s_grid.nz);
  // sums lane % 4, + 4, ... of the slot threadIdx.x / 4
  constexpr int kMine = (kNSum + 3) / 4;
  float acc[kMine];
#pragma unroll
  for (int u = 0; u < kMine; ++u) acc[u] = 0.f;
  for (int r0 = blockIdx.x * kRefSlots; r0 < nP; r0 += kRefRuns * run) {
    i = r0 + own;
    const bool valid = i < nP;
    float xc0 = 0.f, xc1 = 0.f, xc2 = 0.f, x = 0.f, y = 0.f, z = 0.f;
    int bt = kSeedNone;
    bool search = false;
    float seed2 = eps2;
    __syncthreads();  // s_need is 0; the previous round's s_found and s_val have been read
    if (valid) {
      if (r0 >= run) p = XP[i], at = certs[i], nr = near[i];  // (the first round's are here)
      const float *R = s_pose, *c = s_pose + 9, *tc = s_pose + 12;
      xc0 = fmaf(R[0], p.x, fmaf(R[1], p.y, fmaf(R[2], p.z, tc[0])));
      xc1 = fmaf(R[3], p.x, fmaf(R[4], p.y, fmaf(R[5], p.z, tc[1])));
      xc2 = fmaf(R[6], p.x, fmaf(R[7], p.y, fmaf(R[8], p.z, tc[2])));
      x = xc0 + c[0], y = xc1 + c[1], z = xc2 + c[2];
      bt = __float_as_int(nr.w);
      search = true;
      if (bt != kSeedFresh) {
        const float d2 = bt >= 0 ? nn_d2(nr, x, y, z) : eps2, d = bt >= 0 ? sqrtf(d2) : eps;
        if (d2 < eps2) seed2 = d2;
        // (4e-6: above the FP32 rounding of both distances; a NaN searches)
        search = !((d + sqrtf(nn_d2(at, x, y, z))) * (1.f + 4e-6f) < at.w);
      }
    }
    const unsigned m = __ballot_sync(0xffffffffu, search);
    if (m) {
      int base = 0;
      if (lane == 0) base = atomicAdd(&s_need, __popc(m));
      base = __shfl_sync(0xffffffffu, base, 0);
      if (search) {
        s_query[base + __popc(m & ((1u << lane) - 1u))] = make_float4(x, y, z, __int_as_float(threadIdx.x));
        s_found[threadIdx.x] = bt;
        s_seed2[threadIdx.x] = seed2;
      }
    }
    __syncthreads();
    const int need = s_need;
    if (need) {
      constexpr int kWarps = kRefThreads / 32;
      // consecutive queries go to different warps; whole warps reach the shuffles
      for (int q0 = wp; q0 < need; q0 += kRefThreads / kRefH) {
        const int k = q0 + kWarps * (lane / kRefH);
        float4 w = make_float4(__int_as_float(0x7fc00000), 0.f, 0.f, 0.f);  // NaN: the query visits no cell
        int thread = 0, seed = -1;
        float seed2 = eps2;
        if (k < need) {
          w = s_query[k], thread = __float_as_int(w.w);
          if (s_seed2[thread] < eps2) seed = s_found[thread], seed2 = s_seed2[thread];
        }
        const Found f = wrapped ? group_nn_wrapped(s_grid, start, Xe, w.x, w.y, w.z, eps2, seed)
                                : half_nn(s_grid, start, Xe, w.x, w.y, w.z, seed2, seed, kRefGuard * eps);
        if (k < need && (lane & (kRefH - 1)) == 0) {
          s_found[thread] = f.at < 0 ? kSeedNone : f.at;
          certs[r0 + (thread / kRefSlots) * run + (thread % kRefSlots)] = make_float4(w.x, w.y, w.z, f.apart);
        }
      }
      __syncthreads();
      if (threadIdx.x == 0) s_need = 0;
      if (search) {
        bt = s_found[threadIdx.x];
        if (bt >= 0) nr = Xe[bt];
        nr.w = __int_as_float(bt);
        near[i] = nr;
      }
    }
    const float4 q = bt >= 0 ? nr : make_float4(__int_as_float(0x7fc00000), 0.f, 0.f, 0.f);
    float v[kNVal];
#pragma unroll
    for (int u = 0; u < kNVal; ++u) v[u] = 0.f;
    if (nn_d2(q, x, y, z) < eps2) {
      const float e0 = x - q.x, e1 = y - q.y, e2 = z - q.z;  // the residual
      const float s = e0 * e0 + e1 * e1 + e2 * e2;
      const float l = mu / (mu + s);
      const float w = l * l;
      v[0] = 1.f, v[1] = w;
      v[2] = w * xc0, v[3] = w * xc1, v[4] = w * xc2;
      v[5] = xc0, v[6] = xc1, v[7] = xc2;
      v[8] = xc1 * e2 - xc2 * e1;
      v[9] = xc2 * e0 - xc0 * e2;
      v[10] = xc0 * e1 - xc1 * e0;
      v[11] = e0, v[12] = e1, v[13] = e2;
    }
#pragma unroll
    for (int u = 0; u < kNVal; ++u) s_val[u][threadIdx.x] = v[u];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kMine; ++u) {
      const float *A = s_val[kTermA[4 * u + (lane & 3)]], *B = s_val[kTermB[4 * u + (lane & 3)]];
#pragma unroll
      for (int k = 0; k < kRefRuns; ++k) {
        const int t = k * kRefSlots + threadIdx.x / 4;
        acc[u] = fmaf(A[t], B[t], acc[u]);
      }
    }
  }
  {
    __shared__ float sm[kRefThreads / 32][4 * kMine];
#pragma unroll
    for (int u = 0; u < kMine; ++u) {
      // over the warp's eight slots
#pragma unroll
      for (int off = 16; off >= 4; off >>= 1) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], off);
      if (lane < 4) sm[wp][4 * u + lane] = acc[u];
    }
    __syncthreads();
    if (threadIdx.x < kNSum) {
      double t = 0.0;
      for (int k = 0; k < kRefThreads / 32; ++k) t += (double)sm[k][threadIdx.x];
      partials[(size_t)blockIdx.x * kNAcc + threadIdx.x] = t;
    }
  }
  // The last block to finish sums the partials: those of each kRefGroup blocks in
  // block order, sum k = t % 17 over the groups t / 17, t / 17 + 15, ..., then
  // the 15 segments in order (a fixed order: the sums are deterministic). With
  // more than kRefAtOnce groups the last block of each group sums its group
  // first: another fence, atomic and load one after the other (1.7 us), but the
  // 17 x 608 FP64 additions of a full grid alone keep one SM's unit (two lanes a
  // clock) busy for 2.7 us.
  const unsigned nb = gridDim.x, ng = (nb + kRefGroup - 1) / kRefGroup;
  const bool grouped = ng > kRefAtOnce;
  double *gpart = partials + (size_t)kRefMaxBlocks * kNAcc;
  const auto group_sum = [&](unsigned g, int k) {
    const unsigned g0 = g * kRefGroup;
    double v[kRefGroup];
#pragma unroll
    for (unsigned u = 0; u < kRefGroup; ++u)
      v[u] = g0 + u < nb ? __ldcg(partials + (size_t)(g0 + u) * kNAcc + k) : 0.0;
    double t = 0.0;
#pragma unroll
    for (unsigned u = 0; u < kRefGroup; ++u) t += v[u];
    return t;
  };
  if (grouped) {
    unsigned *gticket = reinterpret_cast<unsigned *>(gpart + (size_t)kRefMaxGroups * kNAcc);
    const unsigned cgrp = blockIdx.x / kRefGroup, gsz = min((unsigned)kRefGroup, nb - cgrp * kRefGroup);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(gticket + cgrp, 1u) == gsz - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (threadIdx.x < kNSum) gpart[(size_t)cgrp * kNAcc + threadIdx.x] = group_sum(cgrp, threadIdx.x);
    if (threadIdx.x == 0) gticket[cgrp] = 0u;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&st->ticket, 1u) == (grouped ? ng : nb) - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  __shared__ StepState ss;
  if (threadIdx.x < 12) ss.T[threadIdx.x] = __ldcg(st->T + threadIdx.x);
  else if (threadIdx.x < 15) ss.center[threadIdx.x - 12] = __ldcg(st->center + threadIdx.x - 12);
  else if (threadIdx.x == 15) ss.iters_done = __ldcg(&st->iters_done);
  else if (threadIdx.x == 16) ss.level_iters = __ldcg(&st->level_iters);
  else if (threadIdx.x == 17) tot[kNSum] = 0.0, st->ticket = 0u;
  {
    constexpr int kSeg = kRefThreads / kNSum;
    __shared__ double seg[kSeg][kNSum];
    const int k = threadIdx.x % kNSum, sg = threadIdx.x / kNSum;
    if (sg < kSeg) {
      double sum = 0.0;
      if (grouped)
        for (unsigned g = sg; g < ng; g += kSeg) sum += __ldcg(gpart + (size_t)g * kNAcc + k);
      else if (sg < ng)
        sum += group_sum(sg, k);
      seg[sg][k] = sum;
    }
    __syncthreads();
    if (threadIdx.x < kNSum) {
      double t = 0.0;
      for (int q = 0; q < kSeg; ++q) t += seg[q][threadIdx.x];
      tot[threadIdx.x] = t;
    }
    __syncwarp();
  }
  if (threadIdx.x < 32) refine_solve(tot, ss, st, max_iters, tol);
}

__global__ void k_refine_level_begin(RansacState *st) {
  if (threadIdx.x == 0) {
    st->active = st->status == 0 ? 1 : 0;
    st->level_iters = 0;
    st->ticket = 0u;
  }
}

__global__ void k_subsample(const float *xyz, int n, int stride, float4 *out) {
  int m_n = (n + stride - 1) / stride;
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < m_n; m += gridDim.x * blockDim.x) {
    int i = m * stride;
    out[m] = make_float4(xyz[3 * i], xyz[3 * i + 1], xyz[3 * i + 2], __int_as_float(m));
  }
}

// Starting pose (T_in, or the selected hypothesis already in st) and the
// first linearisation centre: the centroid of P moved by that pose.
__global__ void k_refine_init(RansacState *st, const float *boxP, const double *T_in) {
  if (threadIdx.x != 0) return;
  if (T_in) {
    for (int i = 0; i < 16; ++i) st->T[i] = st->T_hyp[i] = T_in[i];
    st->active = 1;
    st->status = 0;
    st->iters_done = 0;
  }
  const double *T = st->T;
  double m[3] = {boxP[8], boxP[9], boxP[10]};
  for (int r = 0; r < 3; ++r) st->center[r] = T[4 * r] * m[0] + T[4 * r + 1] * m[1] + T[4 * r + 2] * m[2] + T[4 * r + 3];
  st->ticket = 0u;
}

__global__ void k_final_pose(const RansacState *st, float *pose) {
  if (threadIdx.x < 12) {
    int r = threadIdx.x / 4, c = threadIdx.x % 4;
    pose[threadIdx.x] = (float)st->T[4 * r + c];
  }
}

__global__ void k_final_count(const int *count, const unsigned long long *sum, RansacState *st) {
  if (threadIdx.x == 0) {
    st->final_count = count[0];
    st->final_sumd2 = (double)sum[0] / kFixScale;
  }
}

// ---------------------------------------------------------------- information matrix
// Loop verification (eq. (5)-(6)): Lambda = sum over K of G_p^T G_p with
// G_p = [-[p]_x | I], K the moved points p = R p' + t whose nearest Q point
// lies within eps. Written out, G_p^T G_p = [[|p|^2 I - p p^T, [p]_x],
// [-[p]_x, I]], so Lambda needs only |K|, sum p and sum p p^T. Each group of
// kRefG lanes searches one point; its first lane adds 1, d and d d^T with
// d = p - c (c: the centre of Q's box, which keeps the FP32 sums small) to ten
// per-thread sums; blocks reduce them to FP64 partials, and one thread adds
// the partials in block order and expands them about c.
struct InfoArgs {
  float R[9], t[3];
  float eps2;
};

__global__ void __launch_bounds__(kRefThreads) k_info_sums(const float *__restrict__ P, int nP, const GridParams *gep,
                                                           const int *__restrict__ start, const float4 *__restrict__ Xe,
                                                           const float *__restrict__ boxQ, InfoArgs a,
                                                           double *__restrict__ partials) {
  constexpr int G = kRefG, GPB = kRefThreads / G;
  const GridParams g = *gep;
  const float c0 = 0.5f * (boxQ[0] + boxQ[3]), c1 = 0.5f * (boxQ[1] + boxQ[4]), c2 = 0.5f * (boxQ[2] + boxQ[5]);
  const int grp = threadIdx.x / G, sub = threadIdx.x & (G - 1);
  float acc[10];
#pragma unroll
  for (int k = 0; k < 10; ++k) acc[k] = 0.f;
  // block-uniform trip count: every lane reaches the group shuffles
  for (int r0 = blockIdx.x * GPB; r0 < nP; r0 += gridDim.x * GPB) {
    const int i = r0 + grp;
    const bool valid = i < nP;
    float px = valid ? P[3 * i] : __int_as_float(0x7fc00000), py = valid ? P[3 * i + 1] : 0.f,
          pz = valid ? P[3 * i + 2] : 0.f;  // NaN: the query visits no cell
    const float x = fmaf(a.R[0], px, fmaf(a.R[1], py, fmaf(a.R[2], pz, a.t[0])));
    const float y = fmaf(a.R[3], px, fmaf(a.R[4], py, fmaf(a.R[5], pz, a.t[1])));
    const float z = fmaf(a.R[6], px, fmaf(a.R[7], py, fmaf(a.R[8], pz, a.t[2])));
    float best;
    int bt, bidx;
    group_nn<G>(g, &g.margin, start, Xe, x, y, z, a.eps2, best, bt, bidx);
    if (!valid || bt < 0 || sub != 0) continue;
    const float dx = x - c0, dy = y - c1, dz = z - c2;
    acc[0] += 1.f;
    acc[1] += dx, acc[2] += dy, acc[3] += dz;
    acc[4] += dx * dx, acc[5] += dx * dy, acc[6] += dx * dz;
    acc[7] += dy * dy, acc[8] += dy * dz, acc[9] += dz * dz;
  }
  block_reduce_to<10>(acc, partials + (size_t)blockIdx.x * 10);
}

__global__ void k_info_final(const double *__restrict__ partials, int nb, const float *__restrict__ boxQ,
                             double *__restrict__ out) {
  __shared__ double seg[256], tot[10];
  block_sum_partials(partials, nb, 10, 10, seg, tot);
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double S[10];
  for (int k = 0; k < 10; ++k) S[k] = tot[k];
  const double c[3] = {0.5 * ((double)boxQ[0] + (double)boxQ[3]), 0.5 * ((double)boxQ[1] + (double)boxQ[4]),
                       0.5 * ((double)boxQ[2] + (double)boxQ[5])};
  const double n = S[0];
  // sum p = sum d + n c; sum p p^T = sum d d^T + c (sum d)^T + (sum d) c^T + n c c^T
  double sp[3], spp[3][3];
  const double sdd[3][3] = {{S[4], S[5], S[6]}, {S[5], S[7], S[8]}, {S[6], S[8], S[9]}};
  for (int r = 0; r < 3; ++r) sp[r] = S[1 + r] + n * c[r];
  for (int r = 0; r < 3; ++r)
    for (int q = r; q < 3; ++q)  // upper triangle, mirrored: Lambda is exactly symmetric
      spp[r][q] = spp[q][r] = sdd[r][q] + c[r] * S[1 + q] + S[1 + r] * c[q] + n * c[r] * c[q];
  const double tr = spp[0][0] + spp[1][1] + spp[2][2];
  // [sp]_x
  const double K[3][3] = {{0.0, -sp[2], sp[1]}, {sp[2], 0.0, -sp[0]}, {-sp[1], sp[0], 0.0}};
  for (int r = 0; r < 3; ++r)
    for (int q = 0; q < 3; ++q) {
      out[6 * r + q] = (r == q ? tr : 0.0) - spp[r][q];
      out[6 * r + 3 + q] = K[r][q];
      out[6 * (3 + r) + q] = -K[r][q];
      out[6 * (3 + r) + 3 + q] = r == q ? n : 0.0;
    }
  out[36] = n;
}

// ---------------------------------------------------------------- neighbours under a pose
// The nearest Q point of every moved point of P, for the kernels that then
// evaluate their terms in FP64: nn[i] = its position in the sorted array, -1
// if none lies within eps. Searching and evaluating in one kernel left the
// FP64 unit (2 lanes a clock on an SM, a warp instruction every 16 clocks
// however many of its lanes live) to the one lane in four or eight that held a
// point: 59 to 75% of its cycles for an eighth to a quarter of the work, and
// the registers of the FP64 terms kept the search at 16 warps an SM. As a pass
// of its own it runs at full occupancy, writes 4 bytes a point, and the terms
// run a point per lane.
struct PoseNnJobs {
  PoseNnJob j[kPoseJobs];
};
constexpr int kPoseNnG = 4;  // lanes per query

__global__ void __launch_bounds__(kRefThreads, 5) k_pose_nn(const __grid_constant__ PoseNnJobs J) {
  const PoseNnJob &a = J.j[blockIdx.y];
  constexpr int GPB = kRefThreads / kPoseNnG;
  const int i = blockIdx.x * GPB + threadIdx.x / kPoseNnG;
  if ((int)blockIdx.x * GPB >= a.nP) return;
  const bool valid = i < a.nP;
  const GridParams g = *a.g;
  const float px = valid ? a.P[3 * i] : __int_as_float(0x7fc00000), py = valid ? a.P[3 * i + 1] : 0.f,
              pz = valid ? a.P[3 * i + 2] : 0.f;  // NaN: the query visits no cell
  const float x = fmaf(a.R[0], px, fmaf(a.R[1], py, fmaf(a.R[2], pz, a.t[0])));
  const float y = fmaf(a.R[3], px, fmaf(a.R[4], py, fmaf(a.R[5], pz, a.t[1])));
  const float z = fmaf(a.R[6], px, fmaf(a.R[7], py, fmaf(a.R[8], pz, a.t[2])));
  float best;
  int bt, bidx;
  group_nn<kPoseNnG>(g, &g.margin, a.start, a.Xe, x, y, z, a.eps2, best, bt, bidx);
  if (valid && (threadIdx.x & (kPoseNnG - 1)) == 0) a.nn[i] = bt;
}

// ---------------------------------------------------------------- objective
// E = sum_i rho(s_i) - rho(eps^2) over points with an NN closer than eps.
// Forward and backward share this kernel; the backward also writes
// dP_i = 2 rho'(s) R^T r_i, scatters dQ_j -= 2 rho'(s) r_i, and reduces
// g_v = sum 2 rho' r_i and g_w = sum z_i x (2 rho' r_i) with z_i = x_i - v.
// dxi = (J_l(w)^T g_w, g_v) is finished on the host. The nearest neighbour is
// found in FP32 (k_pose_nn, the pose rounded to FP32); the residual of the pair, the
// terms and their sums are evaluated in FP64 from the FP32 coordinates: a
// residual of a few millimetres between points metres from the origin would
// otherwise carry the 2^-24 rounding of the coordinates (about 1e-7 m).
// A thread per point; blockIdx.y is the pair. Bound by FP64 issue (about 110
// instructions a point backward); 8 pairs of 50k points took 8 x 57 us.
struct ObjJobs {
  ObjJob j[kPoseJobs];
};
constexpr int kObjThreads = 128;

__global__ void __launch_bounds__(kObjThreads) k_objective(const __grid_constant__ ObjJobs J, int want_grad) {
  const ObjJob &a = J.j[blockIdx.y];
  if ((int)blockIdx.x >= objective_blocks(a.nP)) return;
  const int nblk = objective_blocks(a.nP);
  double acc[7] = {0, 0, 0, 0, 0, 0, 0};  // E, g_v (3), g_w (3)
  for (int i = blockIdx.x * kObjThreads + threadIdx.x; i < a.nP; i += nblk * kObjThreads) {
    const int bt = a.nn[i];
    if (bt < 0) {
      if (want_grad) a.dP[3 * i] = a.dP[3 * i + 1] = a.dP[3 * i + 2] = 0.f;
      continue;
    }
    const float4 q = a.Xe[bt];
    const double p[3] = {a.P[3 * i], a.P[3 * i + 1], a.P[3 * i + 2]};
    double zd[3], r[3];
    for (int k = 0; k < 3; ++k) {
      zd[k] = a.R[3 * k] * p[0] + a.R[3 * k + 1] * p[1] + a.R[3 * k + 2] * p[2] + a.t[k];
      r[k] = zd[k] - (double)(k == 0 ? q.x : (k == 1 ? q.y : q.z));
    }
    const double s = r[0] * r[0] + r[1] * r[1] + r[2] * r[2];
    const double den = a.mu + s;
    acc[0] += a.mu * s / den - a.rho_eps;
    if (want_grad) {
      const double k2 = 2.0 * a.mu * a.mu / (den * den);
      const double g0 = k2 * r[0], g1 = k2 * r[1], g2 = k2 * r[2];
      a.dP[3 * i + 0] = (float)(a.scale * (a.R[0] * g0 + a.R[3] * g1 + a.R[6] * g2));
      a.dP[3 * i + 1] = (float)(a.scale * (a.R[1] * g0 + a.R[4] * g1 + a.R[7] * g2));
      a.dP[3 * i + 2] = (float)(a.scale * (a.R[2] * g0 + a.R[5] * g1 + a.R[8] * g2));
      const int j = __float_as_int(q.w);
      atomicAdd(&a.dQ[3 * j + 0], (float)(-a.scale * g0));
      atomicAdd(&a.dQ[3 * j + 1], (float)(-a.scale * g1));
      atomicAdd(&a.dQ[3 * j + 2], (float)(-a.scale * g2));
      const double zx = zd[0] - a.v[0], zy = zd[1] - a.v[1], zz = zd[2] - a.v[2];
      acc[1] += g0, acc[2] += g1, acc[3] += g2;
      acc[4] += zy * g2 - zz * g1;
      acc[5] += zz * g0 - zx * g2;
      acc[6] += zx * g1 - zy * g0;
    }
  }
  block_sum_rows<7, kObjThreads>(acc, a.partials + (size_t)blockIdx.x * 7);
}

__global__ void k_objective_sum(const __grid_constant__ ObjJobs J) {
  const ObjJob &a = J.j[blockIdx.y];
  __shared__ double seg[256], tot[7];
  block_sum_partials(a.partials, objective_blocks(a.nP), 7, 7, seg, tot);
  if (threadIdx.x < 7) a.out[threadIdx.x] = tot[threadIdx.x];
}

}  // namespace

int64_t refine_partial_doubles() { return (int64_t)kNAcc * (kRefMaxBlocks + kRefMaxGroups) + kRefMaxGroups; }

cudaError_t refine_reset_tickets(double *partials, cudaStream_t s) {
  return cudaMemsetAsync(partials + (size_t)kNAcc * (kRefMaxBlocks + kRefMaxGroups), 0,
                         sizeof(unsigned) * kRefMaxGroups, s);
}

int refine_blocks(int nP) {
  int64_t b = lsr_div_up((int64_t)(nP > 0 ? nP : 1) * kRefG, kRefThreads);
  return (int)(b < 1 ? 1 : (b > kSms * kRefBlocksPerSm ? kSms * kRefBlocksPerSm : b));  // all blocks resident
}

int gnc_stride(int64_t n, int level, int levels) {
  int64_t f = 1;
  for (int k = 0; k < levels - 1 - level; ++k) f *= 4;
  int64_t cap = n / 4096;
  if (f > cap) f = cap;
  return (int)(f < 1 ? 1 : f);
}

cudaError_t launch_refine_init(RansacState *st, const float *boxP, const double *T_in, cudaStream_t s) {
  LSR_LAUNCH(k_refine_init<<<1, 32, 0, s>>>(st, boxP, T_in));
  return cudaGetLastError();
}

cudaError_t launch_refine_level_begin(RansacState *st, cudaStream_t s) {
  LSR_LAUNCH(k_refine_level_begin<<<1, 32, 0, s>>>(st));
  return cudaGetLastError();
}

cudaError_t launch_subsample(const float *xyz, int n, int stride, float4 *out, cudaStream_t s) {
  int m = (n + stride - 1) / stride;
  int b = (int)lsr_div_up(m > 0 ? m : 1, 256);
  LSR_LAUNCH(k_subsample<<<b < 4096 ? b : 4096, 256, 0, s>>>(xyz, n, stride, out));
  return cudaGetLastError();
}

cudaError_t launch_refine_step(const float4 *XP, int nP, const GridParams *ge, const int *start_e, const float4 *Xe,
                               float eps_r, float mu, int max_iters, RansacState *st, double *partials, float4 *near,
                               float4 *certs, bool chained, cudaStream_t s) {
  const int nb = refine_blocks(nP);
  if (chained) {
    // directly after the previous step: scheduled while it closes
    cudaError_t e = cudaSuccess;
    LSR_LAUNCH(e = pdl_launch(k_refine_step, dim3(nb), dim3(kRefThreads), s, XP, nP, ge, start_e, Xe, eps_r, mu, st,
                              partials, max_iters, 1e-6, near, certs));
    LSR_CUDA_TRY(e);
  } else {
    LSR_LAUNCH(k_refine_step<<<nb, kRefThreads, 0, s>>>(XP, nP, ge, start_e, Xe, eps_r, mu, st, partials, max_iters,
                                                        1e-6, near, certs));
  }
  return cudaGetLastError();
}

cudaError_t launch_final_pose(RansacState *st, float *pose, cudaStream_t s) {
  LSR_LAUNCH(k_final_pose<<<1, 32, 0, s>>>(st, pose));
  return cudaGetLastError();
}

cudaError_t launch_final_count(const int *count, const unsigned long long *sum, RansacState *st, cudaStream_t s) {
  LSR_LAUNCH(k_final_count<<<1, 32, 0, s>>>(count, sum, st));
  return cudaGetLastError();
}

int information_blocks(int nP) {
  int64_t b = lsr_div_up((int64_t)(nP > 0 ? nP : 1) * kRefG, kRefThreads);
  return (int)(b < 1 ? 1 : (b > kSms * 4 ? kSms * 4 : b));
}

cudaError_t launch_information(const float *P, int nP, const GridParams *ge, const int *start_e, const float4 *Xe,
                               const float *boxQ, const float R[9], const float t[3], float eps, double *partials,
                               double *out, cudaStream_t s) {
  InfoArgs a;
  for (int k = 0; k < 9; ++k) a.R[k] = R[k];
  for (int k = 0; k < 3; ++k) a.t[k] = t[k];
  a.eps2 = eps * eps;
  const int nb = information_blocks(nP);
  LSR_LAUNCH(k_info_sums<<<nb, kRefThreads, 0, s>>>(P, nP, ge, start_e, Xe, boxQ, a, partials));
  LSR_LAUNCH(k_info_final<<<1, 256, 0, s>>>(partials, nb, boxQ, out));
  return cudaGetLastError();
}

cudaError_t launch_pose_nn(const PoseNnJob *jobs, int n, cudaStream_t s) {
  if (n < 1 || n > kPoseJobs) return cudaErrorInvalidValue;
  PoseNnJobs J{};
  int64_t most = 1;
  for (int k = 0; k < n; ++k) J.j[k] = jobs[k], most = jobs[k].nP > most ? jobs[k].nP : most;
  const int nb = (int)lsr_div_up(most * kPoseNnG, kRefThreads);
  LSR_LAUNCH(k_pose_nn<<<dim3(nb, n), kRefThreads, 0, s>>>(J));
  return cudaGetLastError();
}

cudaError_t launch_objective(const ObjJob *jobs, int n, int want_grad, cudaStream_t s) {
  if (n < 1 || n > kPoseJobs) return cudaErrorInvalidValue;
  ObjJobs J{};
  int most = 1;
  for (int k = 0; k < n; ++k) {
    J.j[k] = jobs[k];
    const int nb = objective_blocks(jobs[k].nP);
    most = nb > most ? nb : most;
  }
  LSR_LAUNCH(k_objective<<<dim3(most, n), kObjThreads, 0, s>>>(J, want_grad));
  LSR_LAUNCH(k_objective_sum<<<dim3(1, n), 256, 0, s>>>(J));
  return cudaGetLastError();
}

LSR_CHECK_READER(refine)

}  // namespace lsr
