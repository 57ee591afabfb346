// The lattice pressure tensor of Eq. sm:pt in FP64 and its profiles (section 3,
// Eq. pt_projection: radial shells; section 4: planes of a flat interface; the
// paper's own x-axis line).  One implementation serves both profile entry points:
// the kernels are templated on where the fields come from -- the [4][N] FP64
// planes (n_A, n_B, psi_A, psi_B) a context computes from its state, or bare
// density fields with the pseudopotential evaluated on the fly.
#pragma once

#include <math.h>

#include "sc_common.cuh"

namespace scgb {

// Site offsets to the neighbours at distance -H .. H along one axis (coordinate a of n sites, `stride` sites apart).
template <int H>
__device__ __forceinline__ void axis_offsets(int a, int n, int stride, int (&o)[2 * H + 1]) {
#pragma unroll
  for (int d = -H; d <= H; ++d) o[d + H] = ((n == 1 ? 0 : wrapi(a + d, n)) - a) * stride;
}

__device__ __forceinline__ void coords(int64_t s, int nx, int ny, int &x, int &y, int &z) {
  x = int(s % nx);
  const int64_t r = s / nx;
  y = int(r % ny);
  z = int(r / ny);
}
__device__ __forceinline__ int64_t site_at(int x, int y, int z, int nx, int ny, int nz) {
  x = ((x % nx) + nx) % nx;
  y = ((y % ny) + ny) % ny;
  z = ((z % nz) + nz) % nz;
  return (int64_t)x + (int64_t)nx * (y + (int64_t)ny * z);
}

struct ForceParams {
  double G, G_self[2];
  int nx, ny, nz;
  int64_t N;
  SiteDiv div;
};

// Field f of {n_A, n_B, psi_A, psi_B} at site s from stored FP64 planes [4][N].
struct StoredFields {
  const double *f;
  int64_t N;
  __device__ __forceinline__ double operator()(int k, int64_t s) const { return f[k * N + s]; }
};

// The same four fields from two density arrays; psi = exp(-1/n) or psi = n
// (section 4), evaluated where it is needed.
struct DensityFields {
  const double *nA, *nB;
  int psi_exp;
  __device__ __forceinline__ double operator()(int k, int64_t s) const {
    const double n = (k & 1) ? nB[s] : nA[s];
    return (k < 2 || !psi_exp) ? n : exp(-1.0 / n);
  }
};

// Weighted sums of the interaction part of the pressure tensor (Eq. sm:pt) at one site: over the stencil pairs +/- v,
//   t(v) = c_s^2/2 { G [n_A(x) n_B(+/-v) + n_B(x) n_A(+/-v)] + sum_J G_JJ psi_J(x) psi_J(+/-v) },  f(+/-v) = f(x+v) + f(x-v),
// visit(v, t(v)) is called for each (W left to the caller: it is one factor per shell |v|^2); P_mu,nu = c_s^2 (n_A + n_B) delta + sum W t v_mu v_nu.  psi is read only for a
// component with a self coupling.
template <int LAT, int STEN, class FA, class F>
__device__ __forceinline__ void ptensor_terms(const ForceParams &p, const FA &fld, int x, int y, int z, int s, double nA,
                                              double nB, F &&visit) {
  using SN = Stencil<LAT, STEN>;
  constexpr int H = SN::HALO;
  const double h = 0.5 / 3.0;
  const double qA = p.G * h * nB, qB = p.G * h * nA;  // factors of n_A(+/-v), n_B(+/-v)
  const bool sA = p.G_self[0] != 0.0, sB = p.G_self[1] != 0.0;
  const double pA = sA ? p.G_self[0] * h * fld(2, s) : 0.0, pB = sB ? p.G_self[1] * h * fld(3, s) : 0.0;
  int X[2 * H + 1], Y[2 * H + 1], Z[2 * H + 1];
  axis_offsets<H>(x, p.nx, 1, X);
  axis_offsets<H>(y, p.ny, p.nx, Y);
  axis_offsets<H>(z, p.nz, p.nx * p.ny, Z);
#pragma unroll
  for (int k = 0; k < SN::NH; ++k) {
    const int v0 = SN::v(k, 0), v1 = SN::v(k, 1), v2 = SN::v(k, 2);
    const int sp = s + X[H + v0] + Y[H + v1] + Z[H + v2], sm = s + X[H - v0] + Y[H - v1] + Z[H - v2];
    double t = qA * (fld(0, sp) + fld(0, sm)) + qB * (fld(1, sp) + fld(1, sm));
    if (sA) t += pA * (fld(2, sp) + fld(2, sm));
    if (sB) t += pB * (fld(3, sp) + fld(3, sm));
    visit(k, t);
  }
}

struct ProfileArgs {
  int kind;  // sc_profile_kind
  double centre[3];
  double bin_width;
  double inv_width;  // 1 / bin_width where bin_width is a power of two (the quotient is then the product), else 0
  int nbins;
  int dim;        // 2 or 3
  int64_t chunk;  // sites per block
};

// Distance of coordinate c from the centre along one axis, minimum image.
__device__ __forceinline__ double min_image(int c, double centre, int L) {
  double d = c - centre;
  d -= L * floor(d / L + 0.5);
  return d;
}

// Per-block partial sums of a profile, rows [nbins][6] = (sum coordinate, sum P_N, sum P_T, sum n_A, sum n_B,
// count): every warp of the block adds the sites it takes (32 at a time, a fixed assignment) to bins of its own in
// shared memory in a fixed order, and the block adds its warps' bins in warp order, so the result is
// deterministic.  Every row of the block's slice of `partial` is written, so nothing left there by an earlier
// launch is ever read.
//
// Bound: FP64 arithmetic (a warp instruction per 16 cycles and SM).  So the tensor is never formed: a radial row
// needs P_N = e.P.e and the trace, two sums over the stencil pairs (Eq. pt_projection with (v.d)^2 / r^2); sites
// outside the last shell stop at their r^2; the distances to the centre come from a table per axis; four sites are
// added to the bins at a time (24 lanes) unless two of them share a bin.  Several warps a block keep the FP64 pipe
// busy.  Radial profile of 128^3 with 128 bins: 1190 -> 550 us, its
// finalisation (one thread per bin before) 500 -> 10 us.
template <int LAT, int STEN, int KIND, class FA>
__global__ void __launch_bounds__(256) profile_partial_kernel(ForceParams fp, ProfileArgs pa, FA fld, int tables,
                                                              double *partial) {
  using SN = Stencil<LAT, STEN>;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  constexpr bool RADIAL = KIND == SC_PROFILE_RADIAL;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int row = pa.nbins * 6;
  double *bins = reinterpret_cast<double *>(smem_raw) + (int64_t)warp * (row + 32 * 5);
  double *stage = bins + row;  // [5][32] values of this warp's 32 sites
  double *tab = reinterpret_cast<double *>(smem_raw) + (int64_t)nwarps * (row + 32 * 5);  // [nx + ny + nz] distances
  for (int k = lane; k < row; k += 32) bins[k] = 0.0;
  if (RADIAL && tables) {
    for (int k = threadIdx.x; k < fp.nx + fp.ny + fp.nz; k += blockDim.x) {
      const int m = k < fp.nx ? 0 : (k < fp.nx + fp.ny ? 1 : 2);
      const int c = k - (m > 0 ? fp.nx : 0) - (m > 1 ? fp.ny : 0);
      tab[k] = min_image(c, pa.centre[m], m == 0 ? fp.nx : (m == 1 ? fp.ny : fp.nz));
    }
  }
  __syncthreads();
  const double rmax = pa.nbins * pa.bin_width, r2max = rmax * rmax * (1.0 + 1e-9);
  const int64_t s0 = blockIdx.x * pa.chunk, s1 = min(fp.N, s0 + pa.chunk);
  const int cx = int(floor(pa.centre[0] + 0.5)), cy = int(floor(pa.centre[1] + 0.5)),
            cz = int(floor(pa.centre[2] + 0.5));
  for (int64_t base = s0 + 32 * warp; base < s1; base += 32 * nwarps) {
    int bin = -1;
    if (base + lane < s1) {
      const int s = int(base) + lane;
      int x, y, z;
      fp.div.coords(s, fp.nx, fp.ny, x, y, z);
      double coord = 0.0, d0 = 0.0, d1 = 0.0, d2 = 0.0, r2 = 0.0;
      if constexpr (RADIAL) {
        d0 = tables ? tab[x] : min_image(x, pa.centre[0], fp.nx);
        d1 = tables ? tab[fp.nx + y] : min_image(y, pa.centre[1], fp.ny);
        d2 = tables ? tab[fp.nx + fp.ny + z] : min_image(z, pa.centre[2], fp.nz);
        r2 = d0 * d0;
        r2 += d1 * d1;
        r2 += d2 * d2;
        if (r2 <= r2max) {
          coord = sqrt(r2);
          bin = int(floor(pa.inv_width != 0.0 ? coord * pa.inv_width : coord / pa.bin_width));
        }
      } else if constexpr (KIND == SC_PROFILE_PLANAR_Z) {
        coord = z;
        bin = z;
      } else {
        // the x axis through the centre node: row k is the site (cx + k, cy, cz); the
        // entry points accept nbins <= nx only, so each row holds exactly one site
        if (y == ((cy % fp.ny) + fp.ny) % fp.ny && z == ((cz % fp.nz) + fp.nz) % fp.nz) {
          bin = ((x - cx) % fp.nx + fp.nx) % fp.nx;
          coord = bin;
        }
      }
      if (bin >= pa.nbins) bin = -1;
      if (bin >= 0) {
        const double nA = fld(0, s), nB = fld(1, s), ideal = (nA + nB) * (1.0 / 3.0);
        // P_N's sum; the trace's (radial) or P_T's: per shell, then weighted
        double shN[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, shT[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, sN = 0.0, sT = 0.0;
        ptensor_terms<LAT, STEN>(fp, fld, x, y, z, s, nA, nB, [&](int k, double t) {
          const int v0 = SN::v(k, 0), v1 = SN::v(k, 1), v2 = SN::v(k, 2), sh = v0 * v0 + v1 * v1 + v2 * v2;
          if constexpr (RADIAL) {
            // v.d without the terms of a zero component
            const double a0 = v0 < 0 ? -d0 : d0, a1 = v1 < 0 ? -d1 : d1, a2 = v2 < 0 ? -d2 : d2;
            double q = v0 ? a0 : (v1 ? a1 : a2);
            if (v0 && v1) q += a1;
            if ((v0 || v1) && v2) q += a2;
            if (sh == 4) q *= 2.0;  // (2, 0, 0)
            shN[sh] += q * q * t;
            if (pa.dim == 3 || v2 == 0)
              shT[sh] += t;
            else
              shT[0] += SN::W(k) * (v0 * v0 + v1 * v1) * t;  // two dimensions: the trace has no zz
          } else if constexpr (KIND == SC_PROFILE_PLANAR_Z) {
            if (v2) sN += SN::W(k) * (v2 * v2) * t;
            if (v0 || v1) sT += SN::W(k) * (v0 * v0 + v1 * v1) * t;
          } else {
            if (v0) sN += SN::W(k) * (v0 * v0) * t;
            if (v1) sT += SN::W(k) * (v1 * v1) * t;
          }
        });
        if constexpr (RADIAL) {
          sT = shT[0];
#pragma unroll
          for (int sh = 1; sh <= 4; ++sh) {
            double W = 0.0;
#pragma unroll
            for (int k = 0; k < SN::NH; ++k)
              if (SN::v(k, 0) * SN::v(k, 0) + SN::v(k, 1) * SN::v(k, 1) + SN::v(k, 2) * SN::v(k, 2) == sh) W = SN::W(k);
            if (W == 0.0) continue;  // no such shell
            sN += W * shN[sh];
            sT += W * sh * shT[sh];
          }
        }
        double PN, PT;
        if constexpr (RADIAL) {
          const double tr = pa.dim * ideal + sT;
          if (coord == 0.0) {
            PN = PT = tr / pa.dim;
          } else {
            PN = ideal + sN / r2;
            PT = pa.dim == 3 ? 0.5 * (tr - PN) : tr - PN;
          }
        } else if constexpr (KIND == SC_PROFILE_PLANAR_Z) {
          PN = ideal + sN;
          PT = ideal + 0.5 * sT;
        } else {
          PN = ideal + sN;
          PT = ideal + sT;
        }
        stage[lane] = coord;
        stage[32 + lane] = PN;
        stage[64 + lane] = PT;
        stage[96 + lane] = nA;
        stage[128 + lane] = nB;
      }
    }
    __syncwarp();
    if (!__any_sync(0xffffffffu, bin >= 0)) continue;
    // sites l, l + 8, l + 16, l + 24 at a time: lane 8 q + c adds component c (5: the count) of site l + 8 q
    const int q = lane >> 3, c = lane & 7;
    if (__all_sync(0xffffffffu, bin == __shfl_sync(0xffffffffu, bin, 0))) {  // one bin (a plane): add the 32 first
      double acc = 0.0;
      for (int l = 0; l < 8; ++l) acc += c < 5 ? stage[32 * c + l + 8 * q] : 1.0;
      acc += __shfl_xor_sync(0xffffffffu, acc, 8);
      acc += __shfl_xor_sync(0xffffffffu, acc, 16);
      if (lane < 6) bins[bin * 6 + lane] += acc;
      __syncwarp();
      continue;
    }
    for (int l = 0; l < 8; ++l) {
      const int b = __shfl_sync(0xffffffffu, bin, l + 8 * q);
      const int b0 = __shfl_sync(0xffffffffu, b, 0), b1 = __shfl_sync(0xffffffffu, b, 8),
                b2 = __shfl_sync(0xffffffffu, b, 16), b3 = __shfl_sync(0xffffffffu, b, 24);
      const bool clash = (b0 >= 0 && (b0 == b1 || b0 == b2 || b0 == b3)) || (b1 >= 0 && (b1 == b2 || b1 == b3)) ||
                         (b2 >= 0 && b2 == b3);
      const double v = c < 5 ? stage[32 * c + l + 8 * q] : 1.0;
      if (!clash) {
        if (b >= 0 && c < 6) bins[b * 6 + c] += v;
        __syncwarp();
      } else {
        for (int w = 0; w < 4; ++w) {
          if (q == w && b >= 0 && c < 6) bins[b * 6 + c] += v;
          __syncwarp();
        }
      }
    }
  }
  __syncthreads();
  double *out = partial + (int64_t)blockIdx.x * row;
  const double *all = reinterpret_cast<const double *>(smem_raw);
  if constexpr (RADIAL) {
    if (nwarps == 1 && pa.nbins >= 1024) {  // a plain copy, whose loads the loop overlaps
#pragma unroll 8
      for (int k = lane; k < row; k += 32) out[k] = all[k];
      return;
    }
  }
  for (int k = threadIdx.x; k < row; k += blockDim.x) {
    double acc = all[k];
    for (int w = 1; w < nwarps; ++w) acc += all[(int64_t)w * (row + 32 * 5) + k];
    out[k] = acc;
  }
}

// Sum the per-block partials of one bin (a block of 32 x 6 threads) in a fixed order and turn sums into means.
template <class T>
__global__ void __launch_bounds__(192) profile_finalize_kernel(const T *partial, int nblocks, int nbins, T *out) {
  __shared__ T red[6][32];
  __shared__ T sum[6];
  const int b = blockIdx.x, lane = threadIdx.x & 31, c = threadIdx.x >> 5;
  double acc = 0.0;
  for (int k = lane; k < nblocks; k += 32) acc += partial[((int64_t)k * nbins + b) * 6 + c];
  red[c][lane] = acc;
  __syncwarp();
  for (int w = 16; w > 0; w >>= 1) {
    if (lane < w) red[c][lane] += red[c][lane + w];
    __syncwarp();
  }
  if (lane == 0) sum[c] = red[c][0];
  __syncthreads();
  if (lane == 0) out[b * 6 + c] = c == 5 ? sum[5] : (sum[5] > 0 ? sum[c] / sum[5] : 0.0);
}

// The same means, the same order of additions, with a thread per bin and component (a block: 32 bins), for many bins
// of few blocks (at most 32), where a block per bin is mostly launch: 8^3 sites in 4096 bins 54.7 -> 29.0 us (39.1 with a thread per bin and a slower copy of the bins).
template <class T>
__global__ void __launch_bounds__(192) profile_finalize_few_kernel(const T *partial, int nblocks, int nbins, T *out) {
  __shared__ T sum[192];
  const int at = blockIdx.x * 192 + threadIdx.x, n = nbins * 6, c = threadIdx.x % 6;
  T v[32];
#pragma unroll
  for (int k = 0; k < 32; ++k) v[k] = k < nblocks && at < n ? T(0.0) + partial[(int64_t)k * n + at] : T(0.0);
#pragma unroll
  for (int w = 16; w > 0; w >>= 1)
#pragma unroll
    for (int k = 0; k < w; ++k)
      if (k + w < nblocks) v[k] += v[k + w];
  sum[threadIdx.x] = v[0];
  __syncthreads();
  const T count = sum[threadIdx.x - c + 5];
  if (at < n) out[at] = c == 5 ? count : (count > 0 ? v[0] / count : T(0.0));
}

// Blocks of a profile launch and the sites each one takes (a multiple of 32):
// as many blocks as `partial_doubles` holds rows for, at most max_blocks and at
// most one per 32 sites.
inline int64_t profile_blocks(int64_t N, int nbins, int64_t partial_doubles, int64_t max_blocks, int64_t *chunk) {
  int64_t blocks = partial_doubles / ((int64_t)nbins * 6);
  if (blocks > max_blocks) blocks = max_blocks;
  if (blocks > (N + 31) / 32) blocks = (N + 31) / 32;
  if (blocks < 1) blocks = 1;
  int64_t c = (N + blocks - 1) / blocks;
  c = (c + 31) / 32 * 32;
  *chunk = c;
  return (N + c - 1) / c;
}

// Shared memory of a block: the warps' bins and staged values, then the distance tables.  Up to eight warps, as
// many as fit in half an SM's shared memory next to a second block.
constexpr int kProfileWarps = 8;
constexpr size_t kProfileSmem = 110 << 10;
constexpr size_t kProfileMaxSmem = 227 << 10;

// Launch the partial and finalise kernels of one profile on stream st.
template <int LAT, int STEN, int KIND, class FA>
cudaError_t launch_profile_kind(const ForceParams &fp, ProfileArgs pa, const FA &fld, double *partial,
                                int64_t partial_doubles, int64_t max_blocks, double *out, cudaStream_t st) {
  const int64_t blocks = profile_blocks(fp.N, pa.nbins, partial_doubles, max_blocks, &pa.chunk);
  int e2 = 0;
  pa.inv_width = pa.bin_width > 0.0 && frexp(pa.bin_width, &e2) == 0.5 ? 1.0 / pa.bin_width : 0.0;
  const size_t warp_bytes = ((size_t)pa.nbins * 6 + 32 * 5) * sizeof(double);
  const size_t tab_bytes = KIND == SC_PROFILE_RADIAL ? ((size_t)fp.nx + fp.ny + fp.nz) * sizeof(double) : 0;
  const int tables = tab_bytes > 0 && tab_bytes <= (16 << 10) ? 1 : 0;
  const size_t tab = tables ? tab_bytes : 0;
  int warps = kProfileWarps;
  while (warps > 1 && (warps * warp_bytes + tab > kProfileSmem || (int64_t)32 * warps > pa.chunk)) --warps;
  const size_t smem = warps * warp_bytes + tab;
  auto *k = profile_partial_kernel<LAT, STEN, KIND, FA>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kProfileMaxSmem);
  if (e != cudaSuccess) return e;
  k<<<(int)blocks, 32 * warps, smem, st>>>(fp, pa, fld, tables, partial);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (blocks <= 32 && pa.nbins >= 1024)
    profile_finalize_few_kernel<double><<<(pa.nbins + 31) / 32, 192, 0, st>>>(partial, (int)blocks, pa.nbins, out);
  else
    profile_finalize_kernel<double><<<pa.nbins, 192, 0, st>>>(partial, (int)blocks, pa.nbins, out);
  return cudaGetLastError();
}

template <int LAT, int STEN, class FA>
cudaError_t launch_profile_lat(const ForceParams &fp, const ProfileArgs &pa, const FA &fld, double *partial,
                               int64_t partial_doubles, int64_t max_blocks, double *out, cudaStream_t st) {
  if (pa.kind == SC_PROFILE_RADIAL)
    return launch_profile_kind<LAT, STEN, SC_PROFILE_RADIAL>(fp, pa, fld, partial, partial_doubles, max_blocks, out, st);
  if (pa.kind == SC_PROFILE_PLANAR_Z)
    return launch_profile_kind<LAT, STEN, SC_PROFILE_PLANAR_Z>(fp, pa, fld, partial, partial_doubles, max_blocks, out, st);
  return launch_profile_kind<LAT, STEN, SC_PROFILE_AXIS_X>(fp, pa, fld, partial, partial_doubles, max_blocks, out, st);
}

// Dispatch on the lattice and stencil (D2Q9 takes E4 only).
template <class FA>
cudaError_t launch_profile(int lattice, int stencil, const ForceParams &fp, const ProfileArgs &pa, const FA &fld,
                           double *partial, int64_t partial_doubles, int64_t max_blocks, double *out,
                           cudaStream_t st) {
  if (lattice == SC_D2Q9) return launch_profile_lat<kD2Q9, kE4>(fp, pa, fld, partial, partial_doubles, max_blocks, out, st);
  if (stencil == SC_FORCE_E6)
    return launch_profile_lat<kD3Q19, kE6>(fp, pa, fld, partial, partial_doubles, max_blocks, out, st);
  return launch_profile_lat<kD3Q19, kE4>(fp, pa, fld, partial, partial_doubles, max_blocks, out, st);
}

}  // namespace scgb
