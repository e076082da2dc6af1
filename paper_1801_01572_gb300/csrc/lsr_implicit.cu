// lsr_implicit.cu -- gradient of the refined pose with respect to the points
// (implicit differentiation of the robust alignment at its optimum).
//
// The refinement ends at T* minimising E(xi) = sum_i rho(|T(xi) p_i - q_i|^2)
// over the pairs it holds at convergence (eq. (3)-(4) with the line process
// eliminated, rho(s) = mu s / (mu + s); T(xi) = [Exp(w) | v] T*, the left
// perturbation whose Jacobian is G_p = [-[p]_x | I] of eq. (5)). The
// first-order condition g(xi = 0) = 0 defines T* as a function of the points,
// so for a loss L with gradient dL/dxi in that perturbation,
//   lambda = H^-1 dL/dxi,   dL/dp_i = -R^T dphi_i/dz_i,   dL/dq_i = -dphi_i/dq_i,
// with phi_i = lambda . g_i = 2 rho'(s_i) a_i . r_i, a_i = w_l x z_i + v_l,
// z_i = R p_i + t, r_i = z_i - q_i, and H the exact Hessian of E in xi:
//   H = sum 4 rho''(s) (J^T r)(J^T r)^T + 2 rho'(s) (J^T J + S),
// J^T r = (z x r, r), J^T J = [[|z|^2 I - z z^T, [z]_x], [-[z]_x, I]], and S
// (rotation block only) = (r z^T + z r^T) / 2 - (r . z) I, the second
// derivative of r . Exp(w) z at w = 0, which does not vanish for a robust
// kernel away from a zero residual.
//
// After the neighbours under T* (k_pose_nn), three launches: (1) every point
// with a neighbour within eps adds its terms of g and H, evaluated in FP64, to
// FP64 per-block partials; (2) one block sums the partials in a fixed order and
// a warp solves H lambda = dL/dxi by Gaussian elimination with partial
// pivoting in FP64, a row per lane; (3) every point writes dL/dp_i and
// scatters dL/dq_j into its neighbour's row. (1) and (3) are bound by FP64
// issue (a warp instruction every 16 clocks on an SM), so they run a point per
// lane; with the search inside, one lane in four held a point and (1) took
// 121 us for 50k points, and the solve on one lane 24 us.
#include "lsr_internal.cuh"

namespace lsr {

namespace {

constexpr int kImpThreads = 128;
constexpr int kImpSums = 28;    // g (6), H upper triangle (21), count

struct ImpArgs {
  double R[9], t[3];
  double mu;
};

__device__ __forceinline__ void imp_point(const ImpArgs &a, float px, float py, float pz, float4 q, double z[3],
                                          double r[3], double &s, double &d1, double &d2) {
  const double p[3] = {px, py, pz};
  for (int k = 0; k < 3; ++k) z[k] = a.R[3 * k] * p[0] + a.R[3 * k + 1] * p[1] + a.R[3 * k + 2] * p[2] + a.t[k];
  r[0] = z[0] - (double)q.x, r[1] = z[1] - (double)q.y, r[2] = z[2] - (double)q.z;
  s = r[0] * r[0] + r[1] * r[1] + r[2] * r[2];
  const double den = a.mu + s;
  d1 = a.mu * a.mu / (den * den);            // rho'(s)
  d2 = -2.0 * a.mu * a.mu / (den * den * den);  // rho''(s)
}

__global__ void __launch_bounds__(kImpThreads) k_implicit_sums(const float *__restrict__ P, int nP,
                                                               const int *__restrict__ nn,
                                                               const float4 *__restrict__ Xe, ImpArgs a,
                                                               double *__restrict__ partials) {
  double acc[kImpSums];
#pragma unroll
  for (int k = 0; k < kImpSums; ++k) acc[k] = 0.0;
  for (int i = blockIdx.x * kImpThreads + threadIdx.x; i < nP; i += gridDim.x * kImpThreads) {
    const int bt = nn[i];
    if (bt < 0) continue;
    double z[3], r[3], s, d1, d2;
    imp_point(a, P[3 * i], P[3 * i + 1], P[3 * i + 2], Xe[bt], z, r, s, d1, d2);
    const double jr[6] = {z[1] * r[2] - z[2] * r[1], z[2] * r[0] - z[0] * r[2], z[0] * r[1] - z[1] * r[0],
                          r[0], r[1], r[2]};
    const double zz = z[0] * z[0] + z[1] * z[1] + z[2] * z[2], rz = r[0] * z[0] + r[1] * z[1] + r[2] * z[2];
    const double c1 = 2.0 * d1, c2 = 4.0 * d2, diag = zz - rz;
#pragma unroll
    for (int u = 0; u < 6; ++u) acc[u] += c1 * jr[u];
    // H: c2 jr jr^T + c1 (J^T J + S), upper triangle, row-major over (w, v)
    int k = 6;
#pragma unroll
    for (int u = 0; u < 6; ++u) {
      const double cu = c2 * jr[u];
#pragma unroll
      for (int v = u; v < 6; ++v, ++k) {
        acc[k] = fma(cu, jr[v], acc[k]);
        if (v < 3)
          acc[k] += c1 * ((u == v ? diag : 0.0) - z[u] * z[v] + 0.5 * (r[u] * z[v] + z[u] * r[v]));
        else if (u >= 3 && u == v)
          acc[k] += c1;
        else if (u < 3 && v == 3 + (u + 1) % 3)  // [z]_x: entry (u, u + 1) is -z of the third axis
          acc[k] -= c1 * z[(u + 2) % 3];
        else if (u < 3 && v == 3 + (u + 2) % 3)
          acc[k] += c1 * z[(u + 1) % 3];
      }
    }
    acc[27] += 1.0;
  }
  block_sum_rows<kImpSums, kImpThreads>(acc, partials + (size_t)blockIdx.x * kImpSums);
}

// out: g (6), H (36, row-major), lambda (6), count, singular flag.
__global__ void k_implicit_solve(const double *__restrict__ partials, int nb, const double *__restrict__ dl,
                                 double *__restrict__ out) {
  __shared__ double seg[256], tot[kImpSums];
  block_sum_partials(partials, nb, kImpSums, kImpSums, seg, tot);
  if (threadIdx.x >= 32) return;
  // a row of [H | dl] per lane (lanes 6 and up repeat row 5, unused)
  const int lane = threadIdx.x, row = lane < 6 ? lane : 5;
  constexpr unsigned kAll = 0xffffffffu;
  double A[7];
#pragma unroll
  for (int v = 0; v < 6; ++v) {
    const int u0 = row < v ? row : v, v0 = row < v ? v : row;  // the upper triangle's entry (u0, v0)
    A[v] = tot[6 + u0 * 6 - u0 * (u0 - 1) / 2 + v0 - u0];
  }
  A[6] = dl[row];
  double diag = 0.0;
#pragma unroll
  for (int v = 0; v < 6; ++v)
    if (v == row) diag = A[v];
  if (lane < 6) {
    out[lane] = tot[lane];
#pragma unroll
    for (int v = 0; v < 6; ++v) out[6 + 6 * lane + v] = A[v];
  }
  // Gaussian elimination with partial pivoting
  double scale = lane < 6 ? fabs(diag) : 0.0;
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) scale = fmax(scale, __shfl_xor_sync(kAll, scale, o));
  scale = __shfl_sync(kAll, scale, 0);
  int singular = !(scale > 0.0);
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    if (singular) break;
    // the row of the largest entry of column c, the first of equal ones
    double big = lane >= c && lane < 6 ? fabs(A[c]) : -1.0;
    int piv = lane;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      const double ob = __shfl_xor_sync(kAll, big, o);
      const int op = __shfl_xor_sync(kAll, piv, o);
      if (ob > big || (ob == big && op < piv)) big = ob, piv = op;
    }
    big = __shfl_sync(kAll, big, 0), piv = __shfl_sync(kAll, piv, 0);
    if (!(big > 1e-14 * scale)) {
      singular = 1;
      break;
    }
    const int src = lane == c ? piv : (lane == piv ? c : lane);
    double head[7];
#pragma unroll
    for (int q = 0; q < 7; ++q) {
      A[q] = __shfl_sync(kAll, A[q], src);
      head[q] = __shfl_sync(kAll, A[q], c);
    }
    if (lane > c) {
      const double f = A[c] / head[c];
#pragma unroll
      for (int q = c; q < 7; ++q) A[q] -= f * head[q];
    }
  }
  double lam[6] = {0, 0, 0, 0, 0, 0};
  if (!singular) {
#pragma unroll
    for (int c = 5; c >= 0; --c) {
      double v = A[6];
#pragma unroll
      for (int q = 5; q > 0; --q)
        if (q > c) v -= A[q] * lam[q];
      lam[c] = __shfl_sync(kAll, v / A[c], c);
    }
  }
  if (lane == 0) {
    for (int u = 0; u < 6; ++u) out[42 + u] = lam[u];
    out[48] = tot[27];
    out[49] = singular;
  }
}

__global__ void __launch_bounds__(kImpThreads) k_implicit_grad(const float *__restrict__ P, int nP,
                                                               const int *__restrict__ nn,
                                                               const float4 *__restrict__ Xe, ImpArgs a,
                                                               const double *__restrict__ solved, int nQ,
                                                               float *__restrict__ dP, float *__restrict__ dQ) {
  const double wl[3] = {solved[42], solved[43], solved[44]}, vl[3] = {solved[45], solved[46], solved[47]};
  for (int i = blockIdx.x * kImpThreads + threadIdx.x; i < nP; i += gridDim.x * kImpThreads) {
    const int bt = nn[i];
    if (bt < 0) {
      dP[3 * i] = dP[3 * i + 1] = dP[3 * i + 2] = 0.f;
      continue;
    }
    const float4 q = Xe[bt];
    double z[3], r[3], s, d1, d2;
    imp_point(a, P[3 * i], P[3 * i + 1], P[3 * i + 2], q, z, r, s, d1, d2);
    // a_i = w_l x z + v_l
    const double A[3] = {wl[1] * z[2] - wl[2] * z[1] + vl[0], wl[2] * z[0] - wl[0] * z[2] + vl[1],
                         wl[0] * z[1] - wl[1] * z[0] + vl[2]};
    const double ar = A[0] * r[0] + A[1] * r[1] + A[2] * r[2];
    // r x w_l
    const double rw[3] = {r[1] * wl[2] - r[2] * wl[1], r[2] * wl[0] - r[0] * wl[2], r[0] * wl[1] - r[1] * wl[0]};
    double dz[3], gq[3];
    for (int k = 0; k < 3; ++k) {
      dz[k] = 4.0 * d2 * ar * r[k] + 2.0 * d1 * (A[k] + rw[k]);
      gq[k] = 4.0 * d2 * ar * r[k] + 2.0 * d1 * A[k];  // -dphi/dq
    }
    // dL/dp = -R^T dphi/dz
    for (int c = 0; c < 3; ++c)
      dP[3 * i + c] = (float)(-(a.R[c] * dz[0] + a.R[3 + c] * dz[1] + a.R[6 + c] * dz[2]));
    const int j = __float_as_int(q.w);
    if (LSR_IN_BOUNDS(j, nQ, kSiteGridPoint))
      for (int c = 0; c < 3; ++c) atomicAdd(&dQ[3 * j + c], (float)gq[c]);
  }
}

}  // namespace

int implicit_blocks(int nP) {
  const int64_t b = lsr_div_up(nP > 0 ? nP : 1, kImpThreads);
  return (int)(b > kSms * 2 ? kSms * 2 : b);
}
int implicit_partials(int nP) { return implicit_blocks(nP) * kImpSums; }

cudaError_t launch_implicit(const float *P, int nP, const int *nn, const float4 *Xe, int nQ, const double T[16],
                            double mu, const double *dl_dev, double *partials, double *out, float *dP, float *dQ,
                            cudaStream_t s) {
  ImpArgs a;
  for (int r = 0; r < 3; ++r) {
    for (int q = 0; q < 3; ++q) a.R[3 * r + q] = T[4 * r + q];
    a.t[r] = T[4 * r + 3];
  }
  a.mu = mu;
  const int nb = implicit_blocks(nP);
  LSR_LAUNCH(k_implicit_sums<<<nb, kImpThreads, 0, s>>>(P, nP, nn, Xe, a, partials));
  LSR_LAUNCH(k_implicit_solve<<<1, 256, 0, s>>>(partials, nb, dl_dev, out));
  LSR_LAUNCH(k_implicit_grad<<<(int)lsr_div_up(nP > 0 ? nP : 1, kImpThreads), kImpThreads, 0, s>>>(
      P, nP, nn, Xe, a, out, nQ, dP, dQ));
  return cudaGetLastError();
}

LSR_CHECK_READER(implicit)

}  // namespace lsr
