// Kernels around the time step: initial state, population access, FP64
// density / pseudopotential fields, the common velocity, the lattice pressure
// tensor with its profiles, the sigma[R] minimum and conserved totals.
// Analysis results are FP64 (arXiv:2112.02574, sections 2 and 3): sums of stored values are three-term FP32 expansions
// of FP64 accuracy (PairSum3), the sigma[R] grid is screened in FP32, everything else is FP64 arithmetic.
#pragma once

#include "sc_common.cuh"
#include "sc_profile.cuh"

namespace scgb {

// Storage read / write in FP64 (natural populations f = g / scale + w nbar).
// Populations are component-interleaved: element (i * N + s) * 2 + J.
__device__ __forceinline__ double to_double(float v) { return v; }
__device__ __forceinline__ double to_double(double v) { return v; }
__device__ __forceinline__ double to_double(__half v) { return __half2float(v); }
__device__ __forceinline__ double to_double(__nv_bfloat16 v) { return __bfloat162float(v); }
template <class ST>
__device__ __forceinline__ ST from_double(double v);
template <>
__device__ __forceinline__ float from_double<float>(double v) { return float(v); }
template <>
__device__ __forceinline__ double from_double<double>(double v) { return v; }
template <>
__device__ __forceinline__ __half from_double<__half>(double v) { return __float2half_rn(float(v)); }
template <>
__device__ __forceinline__ __nv_bfloat16 from_double<__nv_bfloat16>(double v) {
  return __float2bfloat16_rn(float(v));
}
template <class ST>
__device__ __forceinline__ double load_dev(const ST *p, double inv_scale) {
  return to_double(*p) * inv_scale;
}
template <class ST>
__device__ __forceinline__ void store_dev(ST *p, double v, double scale) {
  *p = from_double<ST>(v * scale);
}

struct PopArgs {
  void *buf;         // stored populations [Q][N][2]
  float2 *nref;      // local reference density deviations n_ref - nbar [N] (16-bit storage; nullptr otherwise)
  int nx, ny, nz;
  int64_t N;
  SiteDiv div;
  double nbar[2];
  double scale[2][19];
  double inv_scale[2][19];
};

// Natural FP64 population of direction i, component J stored at site s.
template <int LAT, class ST>
__device__ __forceinline__ double pop_value(const PopArgs &a, const ST *buf, int i, int J, int64_t s) {
  const double g = load_dev<ST>(buf + ((int64_t)i * a.N + s) * 2 + J, a.inv_scale[J][i]);
  const double ref = a.nbar[J] + (local_ref<ST>() ? double(J == 0 ? a.nref[s].x : a.nref[s].y) : 0.0);
  return g + Lattice<LAT>::w(i) * ref;
}

// mode 0: initial rest equilibrium from densities n0 (FP64 [2][N]): the value
//         stored at y for direction i is w_i n0_J(y + xi_i), so that the first
//         pull delivers f_i(x) = w_i n0_J(x);
// mode 1: natural populations f (FP64 [2][Q][N]) -> storage (inverse pull);
// mode 2: storage -> natural populations f.
// Stored values are relative to w_i nbar_J, or with a local reference to
// w_i nref_J(y) where nref(y) is the sum of the values stored at y.
template <int LAT, class ST>
__global__ void pop_kernel(PopArgs a, int mode, const double *n0A, const double *n0B, double *f) {
  using L = Lattice<LAT>;
  ST *buf = static_cast<ST *>(a.buf);
  const int64_t N = a.N;
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < N; s += (int64_t)gridDim.x * blockDim.x) {
    int x, y, z;
    coords(s, a.nx, a.ny, x, y, z);
    if (mode == 2) {
#pragma unroll
      for (int J = 0; J < 2; ++J)
#pragma unroll
        for (int i = 0; i < L::Q; ++i) {
          const int64_t bwd = site_at(x - L::c(i, 0), y - L::c(i, 1), z - L::c(i, 2), a.nx, a.ny, a.nz);
          f[((int64_t)J * L::Q + i) * N + s] = pop_value<LAT, ST>(a, buf, i, J, bwd);
        }
      continue;
    }
    double ref[2];
#pragma unroll
    for (int J = 0; J < 2; ++J) {
      if constexpr (local_ref<ST>()) {
        double sum = 0.0;
        if (mode == 0) {
          sum = (J == 0 ? n0A : n0B)[s];
        } else {
#pragma unroll
          for (int i = 0; i < L::Q; ++i)
            sum += f[((int64_t)J * L::Q + i) * N + site_at(x + L::c(i, 0), y + L::c(i, 1), z + L::c(i, 2), a.nx, a.ny, a.nz)];
        }
        ref[J] = a.nbar[J] + double(float(sum - a.nbar[J]));  // the deviation is kept in FP32
      } else {
        ref[J] = a.nbar[J];
      }
    }
    if constexpr (local_ref<ST>())
      a.nref[s] = make_float2(float(ref[0] - a.nbar[0]), float(ref[1] - a.nbar[1]));
#pragma unroll
    for (int J = 0; J < 2; ++J)
#pragma unroll
      for (int i = 0; i < L::Q; ++i) {
        const double w = L::w(i);
        const int64_t fwd = site_at(x + L::c(i, 0), y + L::c(i, 1), z + L::c(i, 2), a.nx, a.ny, a.nz);
        const double v = mode == 0 ? w * (J == 0 ? n0A : n0B)[fwd] : f[((int64_t)J * L::Q + i) * N + fwd];
        store_dev<ST>(buf + ((int64_t)i * N + s) * 2 + J, v - w * ref[J], a.scale[J][i]);
      }
  }
}

// Sums of FP32 pairs to FP64 accuracy.  GB300 issues one FP64 warp instruction per 16 cycles and SM but four FP32
// ones per cycle, so sums of values that are stored in FP32 (or fewer bits) are kept as three FP32 terms: each
// addition is Knuth's TwoSum (an error-free transformation) with the error passed down, and only the result is
// converted.  Nothing is lost but the roundings of the third term: for n terms at most n^3 2^-72 of the sum of their
// magnitudes, 2^-59 for the 19 of a density, against the 2^-53 of each FP64 addition.  A sum beyond the FP32 range is infinite.
// Against FP64 sums of the 38 populations of a site (38 conversions, 38 additions): density fields of 128^3 FP32
// 647 -> 88 us, BF16 with one psi 1062 -> 197 us, velocity BF16 1929 -> 683 us (its force stays FP64).
struct PairSum3 {
  float2 a = {0.0f, 0.0f}, b = {0.0f, 0.0f}, c = {0.0f, 0.0f};
  __device__ __forceinline__ static float2 neg_add(float2 x, float2 y) {  // x - y
    return __ffma2_rn(y, make_float2(-1.0f, -1.0f), x);
  }
  __device__ __forceinline__ static float2 two_sum(float2 &s, float2 v) {  // s += v, returns the error
    const float2 t = __fadd2_rn(s, v), bb = neg_add(t, s);
    const float2 e = __fadd2_rn(neg_add(s, neg_add(t, bb)), neg_add(v, bb));
    s = t;
    return e;
  }
  __device__ __forceinline__ void add(float2 v) { c = __fadd2_rn(c, two_sum(b, two_sum(a, v))); }
  __device__ __forceinline__ void sub(float2 v) { add(make_float2(-v.x, -v.y)); }
  // An infinite or NaN term leaves inf - inf in the errors, so the leading term, once it is not finite, is the sum.
  __device__ __forceinline__ static double total(float a, float b, float c) {
    const double s = ((double)c + (double)b) + (double)a;
    return (__float_as_uint(a) & 0x7f800000u) == 0x7f800000u ? (double)a : s;
  }
  __device__ __forceinline__ double2 value() const { return make_double2(total(a.x, b.x, c.x), total(a.y, b.y, c.y)); }
};
struct PairSumD {
  double2 s = {0.0, 0.0};
  __device__ __forceinline__ void add(double2 v) { s = padd(s, v); }
  __device__ __forceinline__ void sub(double2 v) { s = psub(s, v); }
  __device__ __forceinline__ double2 value() const { return s; }
};
template <class ST>
using PairSum = std::conditional_t<std::is_same<ST, double>::value, PairSumD, PairSum3>;
template <class ST>
using PairOf = std::conditional_t<std::is_same<ST, double>::value, double, float>;

__device__ __forceinline__ float2 stored_pair(const float *p) { return *reinterpret_cast<const float2 *>(p); }
__device__ __forceinline__ double2 stored_pair(const double *p) { return *reinterpret_cast<const double2 *>(p); }
__device__ __forceinline__ float2 stored_pair(const __half *p) {
  return __half22float2(*reinterpret_cast<const __half2 *>(p));
}
__device__ __forceinline__ float2 stored_pair(const __nv_bfloat16 *p) {
  return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(p));
}

// 36 w_i: an integer times every density deviation of a local reference, added exactly (12 as 8 + 4).
template <int LAT>
__device__ __forceinline__ constexpr int weight36(int i) {
  return LAT == kD3Q19 ? (i == 0 ? 12 : (i < 7 ? 2 : 1)) : (i == 0 ? 16 : (i < 5 ? 4 : 1));
}

// Densities n_J and, with MOM, momentum sums j_J of the populations arriving at site s (pull), in FP64.
template <int LAT, class ST, bool MOM>
__device__ __forceinline__ void arriving_sums(const PopArgs &a, int s, int x, int y, int z, double2 &n,
                                              double2 (&j)[3]) {
  using L = Lattice<LAT>;
  const ST *buf = static_cast<const ST *>(a.buf);
  int X[3], Y[3], Z[3];
  axis_offsets<1>(x, a.nx, 1, X);
  axis_offsets<1>(y, a.ny, a.nx, Y);
  axis_offsets<1>(z, a.nz, a.nx * a.ny, Z);
  PairSum<ST> sum, mom[3];
  PairSum3 ref, rmom[3];
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    const int src = s + X[1 - L::c(i, 0)] + Y[1 - L::c(i, 1)] + Z[1 - L::c(i, 2)];
    const auto g = stored_pair(buf + ((int64_t)i * a.N + src) * 2);
    sum.add(g);
    if constexpr (MOM) {
#pragma unroll
      for (int m = 0; m < L::DIM; ++m) {
        if (L::c(i, m) > 0) mom[m].add(g);
        if (L::c(i, m) < 0) mom[m].sub(g);
      }
    }
    if constexpr (local_ref<ST>()) {
      const float2 r = a.nref[src];
      constexpr float w8 = 8.0f, w4 = 4.0f;
      const int w = weight36<LAT>(i);
      if (w == 12) {
        ref.add(make_float2(w8 * r.x, w8 * r.y));
        ref.add(make_float2(w4 * r.x, w4 * r.y));
      } else {
        const float2 wr = make_float2(float(w) * r.x, float(w) * r.y);
        ref.add(wr);
        if constexpr (MOM) {
#pragma unroll
          for (int m = 0; m < L::DIM; ++m) {
            if (L::c(i, m) > 0) rmom[m].add(wr);
            if (L::c(i, m) < 0) rmom[m].sub(wr);
          }
        }
      }
    }
  }
  const double2 inv = make_double2(a.inv_scale[0][0], a.inv_scale[1][0]), nb = make_double2(a.nbar[0], a.nbar[1]);
  n = pfma(inv, sum.value(), nb);
  if constexpr (local_ref<ST>()) n = pfma(pbc(1.0 / 36.0), ref.value(), n);
  if constexpr (MOM) {
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      j[m] = m < L::DIM ? pmul(inv, mom[m].value()) : pbc(0.0);
      if constexpr (local_ref<ST>())
        if (m < L::DIM) j[m] = pfma(pbc(1.0 / 36.0), rmom[m].value(), j[m]);
    }
  }
}

// FP64 density fields n_J (and psi_J) from the stored state (pull + sum).
// fields: [4][N] = n_A, n_B, psi_A, psi_B; psi_J is written only for a component with a self coupling
// (self bit J): psi enters the force and the pressure times G_JJ only.
template <int LAT, class ST>
__global__ void __launch_bounds__(128) fields_kernel(PopArgs a, int psi_exp, int self, double *fields) {
  const int64_t N = a.N;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < N; q += (int64_t)gridDim.x * blockDim.x) {
    const int s = (int)q;
    int x, y, z;
    a.div.coords(s, a.nx, a.ny, x, y, z);
    double2 n, j[3];
    arriving_sums<LAT, ST, false>(a, s, x, y, z, n, j);
    fields[s] = n.x;
    fields[N + s] = n.y;
    if (self & 1) fields[2 * N + s] = psi_exp ? exp(-1.0 / n.x) : n.x;
    if (self & 2) fields[3 * N + s] = psi_exp ? exp(-1.0 / n.y) : n.y;
  }
}

// Gradient sum_a W v_a f(x + v_a) of an FP64 plane, +/- pairs first.
template <int STEN_LAT, int STEN>
__device__ __forceinline__ void gradient64(const double *f, int s, const int *X, const int *Y, const int *Z,
                                           double (&S)[3]) {
  using SN = Stencil<STEN_LAT, STEN>;
  constexpr int H = SN::HALO;
  S[0] = S[1] = S[2] = 0.0;
#pragma unroll
  for (int k = 0; k < SN::NH; ++k) {
    const int v0 = SN::v(k, 0), v1 = SN::v(k, 1), v2 = SN::v(k, 2);
    const double d = f[s + X[H + v0] + Y[H + v1] + Z[H + v2]] - f[s + X[H - v0] + Y[H - v1] + Z[H - v2]];
    if (v0) S[0] += SN::W(k) * v0 * d;
    if (v1) S[1] += SN::W(k) * v1 * d;
    if (v2) S[2] += SN::W(k) * v2 * d;
  }
}

// Common velocity of Eq. u (force of Eq. sc_force included) at site s, FP64.  With both self couplings the four
// fields' differences across a stencil pair, each with its own factor, add up before they meet the pair's vector:
// 87 FP64 instructions instead of 108 for four gradients (convergence check of 14 droplets 1430 -> 1333 us).  With
// three fields the longer chain costs more than the 12 instructions it saves (fields and diagnostics at 128^3
// 2690 -> 2745 us), so each has its own gradient there.
template <int LAT, int STEN, class ST>
__device__ __forceinline__ void site_velocity(const PopArgs &a, const ForceParams &fp, const double *fields, int s,
                                              double u[3]) {
  using SN = Stencil<LAT, STEN>;
  constexpr int H = SN::HALO;
  const int64_t N = a.N;
  int x, y, z;
  a.div.coords(s, a.nx, a.ny, x, y, z);
  double2 n, j[3];
  arriving_sums<LAT, ST, true>(a, s, x, y, z, n, j);
  int X[2 * H + 1], Y[2 * H + 1], Z[2 * H + 1];
  axis_offsets<H>(x, a.nx, 1, X);
  axis_offsets<H>(y, a.ny, a.nx, Y);
  axis_offsets<H>(z, a.nz, a.nx * a.ny, Z);
  const double *fA = fields, *fB = fields + N, *gA = fields + 2 * N, *gB = fields + 3 * N;
  const double nA = fA[s], nB = fB[s], h = -0.5 / 3.0;
  // half the force: component A feels the gradient of n_B and the other way round, each its own psi's
  const double cA = fp.G * h * nB, cB = fp.G * h * nA;
  double F[3] = {0.0, 0.0, 0.0}, S[3];
  if (fp.G_self[0] != 0.0 && fp.G_self[1] != 0.0) {
    const double pA = fp.G_self[0] * h * gA[s], pB = fp.G_self[1] * h * gB[s];
#pragma unroll
    for (int k = 0; k < SN::NH; ++k) {
      const int v0 = SN::v(k, 0), v1 = SN::v(k, 1), v2 = SN::v(k, 2);
      const int ip = s + X[H + v0] + Y[H + v1] + Z[H + v2], im = s + X[H - v0] + Y[H - v1] + Z[H - v2];
      const double d = cA * (fA[ip] - fA[im]) + cB * (fB[ip] - fB[im]) + pA * (gA[ip] - gA[im]) + pB * (gB[ip] - gB[im]);
      if (v0) F[0] += SN::W(k) * v0 * d;
      if (v1) F[1] += SN::W(k) * v1 * d;
      if (v2) F[2] += SN::W(k) * v2 * d;
    }
  } else {
    gradient64<LAT, STEN>(fA, s, X, Y, Z, S);
#pragma unroll
    for (int m = 0; m < 3; ++m) F[m] += cA * S[m];
    gradient64<LAT, STEN>(fB, s, X, Y, Z, S);
#pragma unroll
    for (int m = 0; m < 3; ++m) F[m] += cB * S[m];
    if (fp.G_self[0] != 0.0 || fp.G_self[1] != 0.0) {
      const int J = fp.G_self[0] != 0.0 ? 0 : 1;
      const double *g = J ? gB : gA, p = fp.G_self[J] * h * g[s];
      gradient64<LAT, STEN>(g, s, X, Y, Z, S);
#pragma unroll
      for (int m = 0; m < 3; ++m) F[m] += p * S[m];
    }
  }
  const double inv = 1.0 / (nA + nB);
#pragma unroll
  for (int m = 0; m < 3; ++m) u[m] = ((j[m].x + j[m].y) + F[m]) * inv;
}

template <int LAT, int STEN, class ST>
__global__ void __launch_bounds__(128, 4) velocity_kernel(PopArgs a, ForceParams fp, const double *fields, double *u) {
  const int64_t N = a.N;
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < N; s += (int64_t)gridDim.x * blockDim.x) {
    double v[3];
    site_velocity<LAT, STEN, ST>(a, fp, fields, (int)s, v);
#pragma unroll
    for (int m = 0; m < 3; ++m) u[m * N + s] = v[m];
  }
}

// Convergence measure of section 4 (criterion on the velocity field): per-block
// partial sums of sum_alpha |u_alpha(x) - u_prev_alpha(x)| over the sites (fixed
// grid-stride order, fixed tree); u_prev is overwritten with u.
template <int LAT, int STEN, class ST>
__global__ void __launch_bounds__(256, 2) velocity_change_partial_kernel(PopArgs a, ForceParams fp, const double *fields,
                                                                      double *u_prev, double *partial) {
  const int64_t N = a.N;
  double acc = 0.0;
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < N; s += (int64_t)gridDim.x * blockDim.x) {
    double v[3];
    site_velocity<LAT, STEN, ST>(a, fp, fields, (int)s, v);
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      acc += fabs(v[m] - u_prev[m * N + s]);
      u_prev[m * N + s] = v[m];
    }
  }
  __shared__ double red[256];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

// Centre of mass of one density field's excess over a background value, partial
// sums (w x, w y, w z, w) with w = n(x) - background, in lattice coordinates.
__global__ void __launch_bounds__(256) com_partial_kernel(const double *n, int nx, int ny, SiteDiv div, int64_t N,
                                                          double bg, double *partial) {
  double acc[4] = {0, 0, 0, 0};
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < N; s += (int64_t)gridDim.x * blockDim.x) {
    int x, y, z;
    div.coords((int)s, nx, ny, x, y, z);
    const double w = n[s] - bg;
    acc[0] += w * x;
    acc[1] += w * y;
    acc[2] += w * z;
    acc[3] += w;
  }
  __shared__ double red[4][256];
#pragma unroll
  for (int c = 0; c < 4; ++c) red[c][threadIdx.x] = acc[c];
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w)
#pragma unroll
      for (int c = 0; c < 4; ++c) red[c][threadIdx.x] += red[c][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0)
#pragma unroll
    for (int c = 0; c < 4; ++c) partial[blockIdx.x * 4 + c] = red[c][0];
}

// First stride of a tree over the first n of a block's 256 values (the others do not change the result: zeros of a
// sum): the largest power of two below n, at most 128.
__device__ __forceinline__ int tree_top(int n) {
  return n > 128 ? 128 : (n > 1 ? 1 << (31 - __clz(n - 1)) : 0);
}

// Sum of nblocks rows of NC values in a fixed order by one block of 256 threads: a strided sum per thread, then a
// tree over the threads that have a row (all 256: centre of mass of 8^3, two rows, 10.3 -> 12.4 us); the sums are
// returned to thread 0.
template <int NC>
__device__ __forceinline__ void block_rows_sum(const double *partial, int nblocks, double (&out)[NC]) {
  __shared__ double red[NC][256];
  double acc[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) acc[c] = 0.0;
  for (int k = threadIdx.x; k < nblocks; k += 256)
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] += partial[k * NC + c];
#pragma unroll
  for (int c = 0; c < NC; ++c) red[c][threadIdx.x] = acc[c];
  __syncthreads();
  auto halve = [&](int w) {
    if (threadIdx.x < w)
#pragma unroll
      for (int c = 0; c < NC; ++c) red[c][threadIdx.x] += red[c][threadIdx.x + w];
    __syncthreads();
  };
  if (nblocks > 128) {
#pragma unroll
    for (int w = 128; w > 0; w >>= 1) halve(w);
  } else {
    for (int w = tree_top(nblocks); w > 0; w >>= 1) halve(w);
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) out[c] = red[c][0];
}

// out[c] = scale * sum of component c of the partial rows (one thread used to add the rows one after another:
// 63 us for 1024 rows of one component, 230 us of four; 5 and 7 us now).
template <int NC>
__global__ void __launch_bounds__(256) finalize_sum_kernel(const double *partial, int nblocks, double scale,
                                                           double *out) {
  double s[NC];
  block_rows_sum<NC>(partial, nblocks, s);
  if (threadIdx.x == 0)
#pragma unroll
    for (int c = 0; c < NC; ++c) out[c] = scale * s[c];
}

// out = (X, Y, Z, M) with M the summed weight and X = sum w x / M.
__global__ void __launch_bounds__(256) finalize_com_kernel(const double *partial, int nblocks, double *out) {
  double s[4];
  block_rows_sum<4>(partial, nblocks, s);
  if (threadIdx.x == 0) {
    for (int c = 0; c < 3; ++c) out[c] = s[c] / s[3];
    out[3] = s[3];
  }
}

// Bulk pressure of Eq. bulkp (e_2 = 1) at nodes s0 (out[0]) and, with s1 >= 0, s1 (out[1]).
__global__ void bulk_pressure_kernel(ForceParams fp, const double *fields, int64_t s0, int64_t s1, double *out) {
  const int64_t s = threadIdx.x == 0 ? s0 : s1;
  if (threadIdx.x > 1 || s < 0) return;
  const double cs2 = 1.0 / 3.0;
  const double nA = fields[s], nB = fields[fp.N + s];
  double P = (nA + nB) * cs2 + fp.G * cs2 * nA * nB;
  for (int J = 0; J < 2; ++J) {
    if (fp.G_self[J] == 0.0) continue;
    const double ps = fields[(2 + J) * fp.N + s];
    P += 0.5 * fp.G_self[J] * cs2 * ps * ps;
  }
  out[threadIdx.x] = P;
}

// sigma[R] minimum (section 3) on one block of 256 threads (one warp for at most 32 rows and samples); see sc_sigma_minimum in sc.h.
//  * The trapezoid of r^(dim-1) P_T: rows come 256 at a time into shared memory, every thread forms the term of its
//    row with the last non-empty row before it, and the terms are added in a fixed tree.
//  * The grid search needs sigma[R] in FP64 only where it can be the minimum: FP32 values of all samples leave those
//    whose lower bound is below every upper bound.  Their margin is 1e-5 of the sizes of the two terms; R = lo + k step
//    (k < 2^24 exact, both summands positive) and the two terms take at most ten roundings of 2^-24 each, 6e-7.
// One warp did both one after another before: 212 us at 128 rows and 6400 samples, now 18 us.  The trees and the
// search for a chunk's last row span the rows and samples there are: 2 rows and 5 samples 18.9 -> 11.3 us (9.8 in the
// one warp).
constexpr int kSigmaThreads = 256;
__global__ void __launch_bounds__(kSigmaThreads) sigma_kernel(const double *rows, int nbins, const double *pio, int dim,
                                                              double R_lo, double R_hi, double R_step, double *out) {
  const int tid = threadIdx.x, nt = blockDim.x;
  __shared__ double s_r[kSigmaThreads], s_f[kSigmaThreads], s_t[kSigmaThreads];
  __shared__ int s_on[kSigmaThreads];
  __shared__ int s_i[kSigmaThreads];
  __shared__ float s_u[kSigmaThreads];
  double T = 0.0, rp = 0.0, fp = 0.0;  // rp, fp: the last non-empty row of the chunks before
  bool any = false;
  for (int b0 = 0; b0 < nbins; b0 += nt) {
    const int b = b0 + tid, rows_here = min(nt, nbins - b0);
    const bool on = b < nbins && rows[b * 6 + 5] > 0.0;
    const double r = on ? rows[b * 6 + 0] : 0.0, pt = on ? rows[b * 6 + 2] : 0.0;
    const double f = (dim == 3 ? r * r : r) * pt;
    s_on[tid] = on;
    s_r[tid] = r;
    s_f[tid] = f;
    __syncthreads();
    double term = 0.0;
    if (on) {
      int q = tid - 1;
      while (q >= 0 && !s_on[q]) --q;
      if (q >= 0)
        term = 0.5 * (f + s_f[q]) * (r - s_r[q]);
      else if (any)
        term = 0.5 * (f + fp) * (r - rp);
    }
    s_t[tid] = term;
    int last = rows_here - 1;
    while (last >= 0 && !s_on[last]) --last;
    if (last >= 0) {
      rp = s_r[last];
      fp = s_f[last];
      any = true;
    }
    __syncthreads();
    for (int w = tree_top(rows_here); w > 0; w >>= 1) {
      if (tid < w) s_t[tid] += s_t[tid + w];
      __syncthreads();
    }
    T += s_t[0];
    __syncthreads();
  }
  const double Pin = pio[0], Pout = pio[1], dP = Pin - Pout;
  const double C = Pout * (dim == 3 ? rp * rp * rp / 3.0 : rp * rp / 2.0) - T;
  auto sigma = [&](double R) { return dim == 3 ? dP * R / 3.0 + C / (R * R) : dP * R / 2.0 + C / R; };
  // the grid: lowest index on ties
  const int ng = int(floor((R_hi - R_lo) / R_step + 0.5)) + 1;
  const float c1 = float(dim == 3 ? dP / 3.0 : dP / 2.0), c2 = float(C), lo = float(R_lo), st = float(R_step);
  auto bounds = [&](int k, float &down, float &up) {
    const float R = fmaf(float(k), st, lo), u = c1 * R, v = dim == 3 ? c2 / (R * R) : c2 / R, m = 1e-5f * (fabsf(u) + fabsf(v));
    down = u + v - m;
    up = u + v + m;
  };
  float best_up = INFINITY;
  // a warp's worth of samples, or sizes outside FP32's comfortable range: every sample in FP64
  const double big = fmax(fabs(dP), fabs(C)), small = fmin(fabs(dP), fabs(C));
  if (ng > 32 && big < 1e25 && small > 1e-25 && R_lo > 1e-4 && R_hi < 1e8) {
    for (int k = tid; k < ng; k += nt) {
      float down, up;
      bounds(k, down, up);
      best_up = fminf(best_up, up);  // a NaN bound is ignored here and its sample kept below
    }
    s_u[tid] = best_up;
    __syncthreads();
    for (int w = tree_top(min(ng, nt)); w > 0; w >>= 1) {
      if (tid < w) s_u[tid] = fminf(s_u[tid], s_u[tid + w]);
      __syncthreads();
    }
    best_up = s_u[0];
  }
  double best = INFINITY;
  int bi = -1;
  for (int k = tid; k < ng; k += nt) {
    float down, up;
    bounds(k, down, up);
    if (down > best_up && down < INFINITY) continue;
    const double v = sigma(R_lo + k * R_step);
    if (v < best) {
      best = v;
      bi = k;
    }
  }
  s_t[tid] = best;
  s_i[tid] = bi;
  __syncthreads();
  for (int w = tree_top(min(ng, nt)); w > 0; w >>= 1) {
    if (tid < w) {
      const double ob = s_t[tid + w];
      const int oi = s_i[tid + w];
      if (oi >= 0 && (ob < s_t[tid] || (ob == s_t[tid] && (s_i[tid] < 0 || oi < s_i[tid])))) {
        s_t[tid] = ob;
        s_i[tid] = oi;
      }
    }
    __syncthreads();
  }
  if (tid == 0) {
    bi = s_i[0];
    const double Rs = dim == 3 ? cbrt(6.0 * C / dP) : sqrt(2.0 * C / dP);
    out[0] = dP;
    out[1] = C;
    out[2] = Rs;
    out[3] = dim == 3 ? 0.5 * dP * Rs : dP * Rs;
    int k = bi < 1 ? 1 : (bi > ng - 2 ? ng - 2 : bi);
    double Rg = NAN, sg = NAN;
    if (ng >= 3) {
      const double y0 = sigma(R_lo + (k - 1) * R_step), y1 = sigma(R_lo + k * R_step),
                   y2 = sigma(R_lo + (k + 1) * R_step);
      const double den = y0 - 2.0 * y1 + y2;
      const double off = den != 0.0 ? 0.5 * (y0 - y2) / den : 0.0;
      Rg = R_lo + (k + off) * R_step;
      sg = y1 - 0.25 * (y0 - y2) * off;
    }
    out[4] = Rg;
    out[5] = sg;
    out[6] = Pin;
    out[7] = Pout;
  }
}

// Flat-interface tension (section 4): sigma_0 = sum over the planes z >= nbins / 2 of
// P_N(z) - P_T(z) from planar profile rows; one warp, lane-strided sums and a fixed
// shuffle tree (deterministic).
__global__ void __launch_bounds__(32) sigma0_kernel(const double *rows, int nbins, double *out) {
  const int lane = threadIdx.x;
  double acc = 0.0;
  for (int z = nbins / 2 + lane; z < nbins; z += 32) acc += rows[z * 6 + 1] - rows[z * 6 + 2];
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if (lane == 0) out[0] = acc;
}

// Curvature expansion of the surface tension (Eq. sigma_c),
// sigma_s = sigma_0 (1 - 2 delta x + c x^2), x = 1 / R_s, by least squares over n
// droplets: sigma_0 fitted (columns 1, x, x^2) or held at *sigma0 (columns x, x^2 on
// sigma_s / sigma_0 - 1); order 1 drops the x^2 column.  The normal equations are
// formed in x scaled by 1 / max|x| and solved by Gaussian elimination with partial
// pivoting; one thread, fixed order.  out = (sigma_0, delta, c (NaN for order 1), rms
// residual of sigma_s).
__global__ void curvature_fit_kernel(const double *Rs, const double *sig, int n, int order, const double *sigma0,
                                     double *out) {
  if (threadIdx.x != 0) return;
  const bool fixed = sigma0 != nullptr;
  const double s0f = fixed ? sigma0[0] : 0.0;
  double xm = 0.0;
  for (int i = 0; i < n; ++i) xm = fmax(xm, fabs(1.0 / Rs[i]));
  const double sc = xm > 0.0 ? 1.0 / xm : 1.0;
  const int m = fixed ? order : order + 1;
  double G[3][4];
  for (int k = 0; k < 3; ++k)
    for (int l = 0; l < 4; ++l) G[k][l] = 0.0;
  for (int i = 0; i < n; ++i) {
    const double t = sc / Rs[i];
    const double col[3] = {fixed ? t : 1.0, fixed ? t * t : t, t * t};
    const double y = fixed ? sig[i] / s0f - 1.0 : sig[i];
    for (int k = 0; k < m; ++k) {
      for (int l = 0; l < m; ++l) G[k][l] += col[k] * col[l];
      G[k][3] += col[k] * y;
    }
  }
  // elimination on the augmented m x (m + 1) system
  for (int k = 0; k < m; ++k) {
    int piv = k;
    for (int r = k + 1; r < m; ++r)
      if (fabs(G[r][k]) > fabs(G[piv][k])) piv = r;
    if (piv != k)
      for (int l = 0; l < 4; ++l) {
        const double t = G[k][l];
        G[k][l] = G[piv][l];
        G[piv][l] = t;
      }
    for (int r = k + 1; r < m; ++r) {
      const double f = G[r][k] / G[k][k];
      for (int l = k; l < 4; ++l) G[r][l] -= f * G[k][l];
    }
  }
  double c[3] = {0.0, 0.0, 0.0};
  for (int k = m - 1; k >= 0; --k) {
    double v = G[k][3];
    for (int l = k + 1; l < m; ++l) v -= G[k][l] * c[l];
    c[k] = v / G[k][k];
  }
  double s0, a1, a2;  // sigma_s = s0 + a1 x + a2 x^2 in unscaled x
  if (fixed) {
    s0 = s0f;
    a1 = s0f * c[0] * sc;
    a2 = order == 2 ? s0f * c[1] * sc * sc : 0.0;
  } else {
    s0 = c[0];
    a1 = c[1] * sc;
    a2 = order == 2 ? c[2] * sc * sc : 0.0;
  }
  double rss = 0.0;
  for (int i = 0; i < n; ++i) {
    const double x = 1.0 / Rs[i];
    const double d = s0 + a1 * x + a2 * x * x - sig[i];
    rss += d * d;
  }
  out[0] = s0;
  out[1] = -a1 / (2.0 * s0);
  out[2] = order == 2 ? a2 / s0 : NAN;
  out[3] = sqrt(rss / n);
}

// FP32 value as FP64 by integer arithmetic: the conversion instruction issues at the FP64 rate, 1/64 of this.
// Zeros, denormals, infinities and NaN take the instruction.
__device__ __forceinline__ double widen(float v) {
  const unsigned b = __float_as_uint(v), e = b & 0x7f800000u;
  if (e == 0u || e == 0x7f800000u) return (double)v;
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}
__device__ __forceinline__ double widen(double v) { return v; }

// Deterministic FP64 totals: per-block partial sums (fixed grid-stride order,
// fixed tree) of mass_A, mass_B and momentum; finalised in block order.
// The total momentum is a small difference of large sums, so its terms are FP64 populations added one by one.
// FP64-bound: 142 FP64 instructions a site (conversions in integers, no product with a scale of one, no zero
// terms) against 304 before: 128^3 BF16 987 -> 757 us.
template <int LAT, class ST>
__global__ void __launch_bounds__(256) totals_partial_kernel(PopArgs a, double *partial) {
  using L = Lattice<LAT>;
  const ST *buf = static_cast<const ST *>(a.buf);
  const int64_t N = a.N;
  double acc[5] = {0, 0, 0, 0, 0};
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < N; s += (int64_t)gridDim.x * blockDim.x) {
    float2 nref = make_float2(0.0f, 0.0f);
    if constexpr (local_ref<ST>()) nref = a.nref[s];
    double g[2][L::Q];
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      // stored at the collision site: sums over all sites need no pull
      const auto v = stored_pair(buf + ((int64_t)i * N + s) * 2);
      g[0][i] = widen(v.x);
      g[1][i] = widen(v.y);
    }
#pragma unroll
    for (int J = 0; J < 2; ++J) {
      const double ref = a.nbar[J] + (local_ref<ST>() ? widen(J == 0 ? nref.x : nref.y) : 0.0);
#pragma unroll
      for (int i = 0; i < L::Q; ++i) {
        const double wr = __dmul_rn(L::w(i), ref);
        const double f = scaled_units<ST>() ? __fma_rn(g[J][i], a.inv_scale[J][0], wr) : __dadd_rn(g[J][i], wr);
        acc[J] += f;
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          if (L::c(i, m) > 0) acc[2 + m] += f;
          if (L::c(i, m) < 0) acc[2 + m] -= f;
        }
      }
    }
  }
  __shared__ double red[5][256];
#pragma unroll
  for (int c = 0; c < 5; ++c) red[c][threadIdx.x] = acc[c];
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w)
#pragma unroll
      for (int c = 0; c < 5; ++c) red[c][threadIdx.x] += red[c][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x < 5) partial[blockIdx.x * 5 + threadIdx.x] = red[threadIdx.x][0];
}

// Sums of the NC components of nblocks rows added in block order (the mean densities and the totals keep this
// order: the first fix the stored bits of every population, the others are differences).  The rows come into
// shared memory by all threads; one thread per component adds them.
template <int NC>
__global__ void __launch_bounds__(256) totals_finalize_kernel(const double *partial, int nblocks, double *out) {
  __shared__ double rows[256 * NC];
  double acc = 0.0;
  for (int k0 = 0; k0 < nblocks; k0 += 256) {
    const int n = min(256, nblocks - k0) * NC;
    for (int k = threadIdx.x; k < n; k += 256) rows[k] = partial[k0 * NC + k];
    __syncthreads();
    if (threadIdx.x < NC) {
#pragma unroll 8
      for (int k = threadIdx.x; k < n; k += NC) acc += rows[k];
    }
    __syncthreads();
  }
  if (threadIdx.x < NC) out[threadIdx.x] = acc;
}

// Deterministic FP64 sums of two fields (used for the mean initial densities).
__global__ void __launch_bounds__(256) sum2_partial_kernel(const double *a, const double *b, int64_t N,
                                                           double *partial) {
  double acc[2] = {0, 0};
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < N; s += (int64_t)gridDim.x * blockDim.x) {
    acc[0] += a[s];
    acc[1] += b[s];
  }
  __shared__ double red[2][256];
  red[0][threadIdx.x] = acc[0];
  red[1][threadIdx.x] = acc[1];
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      red[0][threadIdx.x] += red[0][threadIdx.x + w];
      red[1][threadIdx.x] += red[1][threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x < 2) partial[blockIdx.x * 2 + threadIdx.x] = red[threadIdx.x][0];
}

// max |n_J - nbar_J| of both init fields (for the F16/BF16 scales); one value per block.
__global__ void __launch_bounds__(256) maxdev_partial_kernel(const double *a, const double *b, int64_t N,
                                                             double nbarA, double nbarB, double *partial) {
  double m[2] = {0, 0};
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < N; s += (int64_t)gridDim.x * blockDim.x) {
    m[0] = fmax(m[0], fabs(a[s] - nbarA));
    m[1] = fmax(m[1], fabs(b[s] - nbarB));
  }
  __shared__ double red[2][256];
  red[0][threadIdx.x] = m[0];
  red[1][threadIdx.x] = m[1];
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      red[0][threadIdx.x] = fmax(red[0][threadIdx.x], red[0][threadIdx.x + w]);
      red[1][threadIdx.x] = fmax(red[1][threadIdx.x], red[1][threadIdx.x + w]);
    }
    __syncthreads();
  }
  if (threadIdx.x < 2) partial[blockIdx.x * 2 + threadIdx.x] = red[threadIdx.x][0];
}

// min of (n_A, n_B) over both init fields, per block (validation: densities > 0).
__global__ void __launch_bounds__(256) min2_partial_kernel(const double *a, const double *b, int64_t N,
                                                           double *partial) {
  double m = INFINITY;
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < N; s += (int64_t)gridDim.x * blockDim.x)
    m = fmin(m, fmin(a[s], b[s]));  // NaN-propagation: fmin ignores NaN, so flag it explicitly
  __shared__ double red[256];
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < N; s += (int64_t)gridDim.x * blockDim.x)
    if (!(a[s] > 0.0) || !(b[s] > 0.0) || !isfinite(a[s]) || !isfinite(b[s])) bad = 1;
  red[threadIdx.x] = m;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] = fmin(red[threadIdx.x], red[threadIdx.x + w]);
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = bad ? -1.0 : red[0];
}

}  // namespace scgb
