// The fused time step for small D2Q9 lattices in FP64: one thread per site and component.
//
// A 64 x 64 lattice in tiles of 32 x 4 sites is 32 blocks of four warps: the FP64 pipe of 32 SMs (one warp
// instruction per 16 cycles) is the bound, 120 SMs have nothing to do, and tiles of one row leave a single warp a
// chain of 200 dependent FP64 instructions of 50-90 cycles each.  Here a block owns 32 x 1 sites and has eight
// warps: the sums of its sites and of the halo, per component, are one round of 204 threads, and two warps collide,
// one per component, exchanging only the half momenta.  Operation by operation the arithmetic is sc_step_kernel's,
// so the stored bits are the same.
// Measured, 64 x 64: 9.1 -> 5.1 us a step (96 x 96: 9.2 -> 6.2).  The halo costs two thirds of the sums, so the rule is two blocks
// per SM at most (96 x 96); beyond that the FP64 pipes are full either way.
#pragma once

#include "sc_step_kernel.cuh"

namespace scgb {

constexpr int kLaneThreads = 256;

template <bool T1>
__global__ void __launch_bounds__(kLaneThreads) sc_step_lanes(const StepArgs<double> a) {
  using L = Lattice<kD2Q9>;
  using SN = Stencil<kD2Q9, kE4>;
  constexpr int Q = L::Q, SX = 34;
  __shared__ double s_dn[2][3][SX], s_psi[2][3][SX], s_h[2][2][32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nx = a.nx, ny = a.ny, x0 = blockIdx.x * 32, y0 = blockIdx.y;
  // warp 0: component A of the block's sites, warp 1: component B; then 70 halo sites of A, 70 of B
  int J, px, py;
  bool on = true;
  if (warp < 2) {
    J = warp;
    px = lane;
    py = 0;
  } else {
    const int h = tid - 64;
    J = h >= 70 ? 1 : 0;
    const int k = h - 70 * J;
    on = h < 140;
    py = k < SX ? -1 : (k < 2 * SX ? 1 : 0);
    px = k < SX ? k - 1 : (k < 2 * SX ? k - SX - 1 : (k == 2 * SX ? -1 : 32));
  }
  const double nbar = J ? a.nbar.y : a.nbar.x, gself = J ? a.gself.y : a.gself.x, psibar = J ? a.psibar.y : a.psibar.x;
  const int gx = ((x0 + px) % nx + nx) % nx, gy = ((y0 + py) % ny + ny) % ny;
  pass_begin();
  double g[Q], dn = 0.0;
  if (on) {
    const double *src = static_cast<const double *>(a.src);
    const int X[3] = {wrapi(gx + 1, nx), gx, wrapi(gx - 1, nx)};
    const int Y[3] = {wrapi(gy + 1, ny) * nx, gy * nx, wrapi(gy - 1, ny) * nx};
#pragma unroll
    for (int i = 0; i < Q; ++i) g[i] = src[((int64_t)i * a.N + X[L::c(i, 0) + 1] + Y[L::c(i, 1) + 1]) * 2 + J];
#pragma unroll
    for (int i = 0; i < Q; ++i) dn = radd(dn, g[i]);
    s_dn[J][py + 1][px + 1] = dn;
    if (a.self_on) {
      double p = dn;
      if (a.psi_exp) {
        const double n = radd(nbar, dn);
        p = rmul(psibar, gself != 0.0 ? expm1(rdiv(dn, rmul(n, nbar))) : 0.0);
      }
      s_psi[J][py + 1][px + 1] = p;
    }
  }
  __syncthreads();
  const int c = lane + 1;  // ring column of the site
  double F[2], n = 0.0, nA = 0.0, nB = 0.0;
  if (warp < 2) {
    nA = radd(a.nbar.x, s_dn[0][1][c]);
    nB = radd(a.nbar.y, s_dn[1][1][c]);
    n = J ? nB : nA;
    double S[2] = {0.0, 0.0}, T[2] = {0.0, 0.0};
#pragma unroll
    for (int k = 0; k < SN::NH; ++k) {
      const int vx = SN::v(k, 0), vy = SN::v(k, 1);
      const double d = rsub(s_dn[1 - J][1 + vy][c + vx], s_dn[1 - J][1 - vy][c - vx]);  // the other component's
      if (vx) S[0] = rfma(SN::W(k) * vx, d, S[0]);
      if (vy) S[1] = rfma(SN::W(k) * vy, d, S[1]);
      if (a.self_on) {
        const double e = rsub(s_psi[J][1 + vy][c + vx], s_psi[J][1 - vy][c - vx]);
        if (vx) T[0] = rfma(SN::W(k) * vx, e, T[0]);
        if (vy) T[1] = rfma(SN::W(k) * vy, e, T[1]);
      }
    }
    const double psi = a.self_on ? radd(psibar, s_psi[J][1][c]) : 0.0;
    const double cn = rmul(a.gcross, n), cp = rmul(gself, psi);
    double d[Q];
#pragma unroll
    for (int i = 1; i < Q; i += 2) d[i] = rsub(g[i], g[i + 1]);
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      F[m] = rfma(cp, T[m], rmul(cn, S[m]));
      double j = 0.0;
#pragma unroll
      for (int i = 1; i < Q; i += 2) {
        if (L::c(i, m) > 0) j = radd(j, d[i]);
        if (L::c(i, m) < 0) j = rsub(j, d[i]);
      }
      s_h[J][m][lane] = rfma(0.5, F[m], j);
    }
  }
  __syncthreads();
  if (warp >= 2 || x0 + lane >= nx) return;
  const double inv_n = rdiv(1.0, radd(nA, nB));
  double u[2];
#pragma unroll
  for (int m = 0; m < 2; ++m) u[m] = rmul(radd(s_h[0][m][lane], s_h[1][m][lane]), inv_n);
  // collide_pair's factored form for this component
  const double om = T1 ? 1.0 : (J ? a.omega.y : a.omega.x), ga = T1 ? 0.5 : (J ? a.guo.y : a.guo.x);
  const double uu = rfma(u[1], u[1], rmul(u[0], u[0])), uF = rfma(u[1], F[1], rmul(u[0], F[0]));
  const double a0 = rfma(rmul(-3.0, ga), uF, rfma(rmul(rmul(-1.5, om), n), uu, rmul(om, dn)));
  const double a1 = rmul(rmul(3.0, om), n), a4 = rmul(3.0, ga), keep = rsub(1.0, om);
  const double K[2] = {rmul(a4, F[0]), rmul(a4, F[1])};
  double *dst = static_cast<double *>(a.dst) + ((int64_t)y0 * nx + x0 + lane) * 2 + J;
  const int64_t stride = 2 * a.N;
  dst[0] = T1 ? rmul(L::w(0), a0) : rfma(keep, g[0], rmul(L::w(0), a0));
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    const double w = L::w(i);
    double cu = 0.0, q = 0.0;
    bool first = true;
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      if (L::c(i, m) == 0) continue;
      cu = first ? u[m] : (L::c(i, m) > 0 ? radd(cu, u[m]) : rsub(cu, u[m]));
      q = first ? K[m] : (L::c(i, m) > 0 ? radd(q, K[m]) : rsub(q, K[m]));
      first = false;
    }
    const double O = rfma(a1, cu, q);
    const double E = rfma(rmul(rmul(1.5, w), cu), radd(O, q), rmul(w, a0));
    dst[i * stride] = T1 ? rfma(w, O, E) : rfma(keep, g[i], rfma(w, O, E));
    dst[(i + 1) * stride] = T1 ? rfma(rmul(-1.0, w), O, E) : rfma(keep, g[i + 1], rfma(rmul(-1.0, w), O, E));
  }
  if (J == 0) check_density<double>(a, make_double2(nA, nB));
}

}  // namespace scgb
