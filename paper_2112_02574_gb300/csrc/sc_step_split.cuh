// The time step in two passes (D3Q19, E4 or E6, tau_A = tau_B = 1, every side >= 4, any storage); split_default in
// sc_api.cu says which lattices take it.
//
//  * The moments pass pulls the populations of a site once and keeps what collisions need of them:
//    the density deviation pair, the three momentum-sum pairs (carry_size) and, with a self coupling,
//    the psi deviation pair.
//  * The collision pass reads those of the site, the density (and psi) of its stencil neighbours, and
//    writes the post-collision populations.
//
// The arithmetic is that of sc_step_kernel, operation by operation, so the stored bits are the same.
// Against the one-pass kernels no density is summed twice (they re-sum a halo of one or two sites around
// every tile and chunk, and evaluate psi there), a thread takes one site of the linear order whatever the
// sides are (no lane idles in a partial x tile), and no block waits at a barrier; in return 32 bytes a site
// (40 with a self coupling; twice that in FP64) are written and read again between the passes, through L2
// while that buffer fits there.
// Measured, one step, one-pass -> two passes (FP32 unless noted): E6 64 x 64 x 256 80.3 -> 58.0 us,
// E6 160^3 302 -> 259 us (FP16 363 -> 209 us), 65^3 29.5 -> 14.9 us (paper couplings), 201^3 567 -> 499 us,
// 64^3 21.4 -> 12.0 us, FP64 64^3 320 -> 212 us (one psi).  Bound: HBM at large sizes (256^3: 368 bytes a site at
// 6.9 TB/s; 512^3 FP16 with psi: 248 bytes a site, 80 of them moments, at 6.0 TB/s), FP64 arithmetic in FP64, latency
// below about 40^3.
#pragma once

#include "sc_step_kernel.cuh"

namespace scgb {

// One lattice as the two passes step it.
template <class CT>
struct SplitArgs {
  StepArgs<CT> a;
  int keep_moments, pad;  // L2 eviction priorities, see L2Policy
  // Pairs: density deviations [N], or with a self coupling density and psi deviations side by side [N][2] (a
  // stencil neighbour is then one 16-byte load, not two of 8 and two addresses), then momentum sums x, y, z [N].
  P2<CT> *mom;
  SiteDiv div;
};

// L2 eviction priorities.  The moments are written by one pass and read by the next; the populations of a large
// lattice stream through L2 in between and would push them out, though the next step cannot find them there
// either.  Up to a measured size (keep_moments, kKeptMoments in sc_api.cu) they are written with evict-last, the populations are read
// with evict-first, and so are the momentum sums, for the last time, so that no evict-last line of theirs is left
// behind.  Us a step, all normal -> so: E6 64 x 64 x 256 67.8 -> 59.4, 96^3 FP32 51.5 -> 42.1,
// 128^3 FP32 117.9 -> 108.2, FP16 94.1 -> 88.6, 160^3 FP32 (131 MB of moments) 227.5 -> 221.8; no effect at 64^3
// (all of it stays); 256^3 would lose 2 %.  Evict-first on the written populations loses 1-3 %.
struct L2Policy {
  unsigned long long first, last;
  __device__ __forceinline__ explicit L2Policy(int keep) {
    unsigned long long n, f, l;
    asm("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(n));
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(f));
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(l));
    first = keep ? f : n;
    last = keep ? l : n;
  }
};
__device__ __forceinline__ float2 load_hint(const float *p, unsigned long long pol) {
  float2 v;
  asm volatile("ld.global.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;" : "=f"(v.x), "=f"(v.y) : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ double2 load_hint(const double *p, unsigned long long pol) {
  double2 v;
  asm volatile("ld.global.L2::cache_hint.v2.f64 {%0, %1}, [%2], %3;" : "=d"(v.x), "=d"(v.y) : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ unsigned load_hint_u32(const void *p, unsigned long long pol) {
  unsigned u;
  asm volatile("ld.global.L2::cache_hint.b32 %0, [%1], %2;" : "=r"(u) : "l"(p), "l"(pol));
  return u;
}
__device__ __forceinline__ float2 load_hint(const __half *p, unsigned long long pol) {
  const unsigned u = load_hint_u32(p, pol);
  return __half22float2(*reinterpret_cast<const __half2 *>(&u));
}
__device__ __forceinline__ float2 load_hint(const __nv_bfloat16 *p, unsigned long long pol) {
  const unsigned u = load_hint_u32(p, pol);
  return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u));
}
__device__ __forceinline__ void store_hint(float2 *p, float2 v, unsigned long long pol) {
  asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(p), "f"(v.x), "f"(v.y), "l"(pol) : "memory");
}
__device__ __forceinline__ void store_hint(double2 *p, double2 v, unsigned long long pol) {
  asm volatile("st.global.L2::cache_hint.v2.f64 [%0], {%1, %2}, %3;" ::"l"(p), "d"(v.x), "d"(v.y), "l"(pol) : "memory");
}

// Element at a byte offset below 2^32 from a pointer that is the same for every thread: the address is the
// uniform base plus a 32-bit register, without 64-bit arithmetic per access.
template <class T>
__device__ __forceinline__ T *at(T *base, unsigned bytes) {
  return reinterpret_cast<T *>(reinterpret_cast<uintptr_t>(base) + bytes);
}

// Density and psi deviations of a site.
template <class CT>
struct DensityPsi {
  P2<CT> n, psi;
};
__device__ __forceinline__ DensityPsi<float> load_density_psi(const float2 *p) {
  const float4 v = *reinterpret_cast<const float4 *>(p);
  return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ DensityPsi<double> load_density_psi(const double2 *p) { return {p[0], p[1]}; }
__device__ __forceinline__ void store_density_psi(float2 *p, float2 n, float2 psi, unsigned long long pol) {
  asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p), "f"(n.x), "f"(n.y), "f"(psi.x),
               "f"(psi.y), "l"(pol)
               : "memory");
}
__device__ __forceinline__ void store_density_psi(double2 *p, double2 n, double2 psi, unsigned long long pol) {
  store_hint(p, n, pol);
  store_hint(p + 1, psi, pol);
}

// Moments pass at site s.
template <class ST, class CT>
__device__ __forceinline__ void split_moments(const SplitArgs<CT> &m, const ST *src, const float2 *nsrc, int s) {
  using L = Lattice<kD3Q19>;
  const StepArgs<CT> &a = m.a;
  const L2Policy pol(m.keep_moments);
  int x, y, z;
  m.div.coords(s, a.nx, a.ny, x, y, z);
  // byte offset of the source for a velocity component of -1, 0, +1
  constexpr int E = 2 * sizeof(ST);
  const int W = a.nx * a.ny;
  const unsigned X[3] = {unsigned(x == a.nx - 1 ? 1 - a.nx : 1) * E, 0u, unsigned(x == 0 ? a.nx - 1 : -1) * E};
  const unsigned Y[3] = {unsigned(y == a.ny - 1 ? a.nx * (1 - a.ny) : a.nx) * E, 0u,
                         unsigned(y == 0 ? a.nx * (a.ny - 1) : -a.nx) * E};
  const unsigned Z[3] = {unsigned(z == a.nz - 1 ? W * (1 - a.nz) : W) * E, 0u,
                         unsigned(z == 0 ? W * (a.nz - 1) : -W) * E};
  P2<CT> g[L::Q];
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    const unsigned o = unsigned(s) * E + X[L::c(i, 0) + 1] + Y[L::c(i, 1) + 1] + Z[L::c(i, 2) + 1];
    g[i] = load_hint(at(src + (int64_t)i * a.N * 2, o), pol.first);
    if constexpr (local_ref<ST>()) {
      const float2 ns = *at(nsrc, o * (8 / E));
      g[i] = pfma(wpair<kD3Q19, ST, CT>(i, a.scale), pset(CT(ns.x), CT(ns.y)), g[i]);
    }
  }
  P2<CT> sum = pbc(CT(0));
#pragma unroll
  for (int i = 0; i < L::Q; ++i) sum = padd(sum, g[i]);
  const P2<CT> dn = unscale<ST, CT>(sum, a.inv_scale);
  P2<CT> j[3];
  momentum_sums<kD3Q19, CT>(g, j);
  const unsigned p = unsigned(s) * unsigned(sizeof(P2<CT>));
  if (a.self_on)
    store_density_psi(at(m.mom, 2 * p), dn, psi_deviation<CT>(dn, a.nbar, a.psibar, a.psi_exp, a.gself), pol.last);
  else
    store_hint(at(m.mom, p), dn, pol.last);
  P2<CT> *jp = m.mom + (a.self_on ? 2 : 1) * a.N;
  store_hint(at(jp, p), j[0], pol.last);
  store_hint(at(jp + a.N, p), j[1], pol.last);
  store_hint(at(jp + 2 * a.N, p), j[2], pol.last);
}

// Collision pass at site s: Eq. sc_force from the stored densities in force_pair's order, then the shared collision.
template <int STEN, class ST, class CT>
__device__ __forceinline__ void split_collide(const SplitArgs<CT> &m, ST *dst, float2 *ndst, int s) {
  using L = Lattice<kD3Q19>;
  using SN = Stencil<kD3Q19, STEN>;
  constexpr int H = SN::HALO;
  const StepArgs<CT> &a = m.a;
  const L2Policy pol(m.keep_moments);
  int x, y, z;
  m.div.coords(s, a.nx, a.ny, x, y, z);
  constexpr unsigned E = sizeof(P2<CT>);
  const unsigned p = unsigned(s) * E, E1 = a.self_on ? 2 * E : E, o = unsigned(s) * E1;  // byte offsets
  const CT *jp = reinterpret_cast<const CT *>(m.mom + (a.self_on ? 2 : 1) * a.N);
  const P2<CT> j[3] = {load_hint(at(jp, p), pol.first), load_hint(at(jp + 2 * a.N, p), pol.first),
                       load_hint(at(jp + 4 * a.N, p), pol.first)};
  unsigned X[2 * H + 1], Y[2 * H + 1], Z[2 * H + 1];
  const int W = a.nx * a.ny;
#pragma unroll
  for (int d = -H; d <= H; ++d) {
    X[d + H] = unsigned(wrapi(x + d, a.nx) - x) * E1;
    Y[d + H] = unsigned((wrapi(y + d, a.ny) - y) * a.nx) * E1;
    Z[d + H] = unsigned((wrapi(z + d, a.nz) - z) * W) * E1;
  }
  const P2<CT> *mom = m.mom;
  P2<CT> S[3] = {pbc(CT(0)), pbc(CT(0)), pbc(CT(0))}, T[3] = {pbc(CT(0)), pbc(CT(0)), pbc(CT(0))};
  P2<CT> dn, psi = pbc(CT(0));
  if (a.self_on) {
    const DensityPsi<CT> own = load_density_psi(at(mom, o));
    dn = own.n;
    psi = padd(a.psibar, own.psi);
#pragma unroll
    for (int k = 0; k < SN::NH; ++k) {
      const int vx = SN::v(k, 0), vy = SN::v(k, 1), vz = SN::v(k, 2);
      const DensityPsi<CT> fp = load_density_psi(at(mom, o + X[H + vx] + Y[H + vy] + Z[H + vz])),
                           fm = load_density_psi(at(mom, o + X[H - vx] + Y[H - vy] + Z[H - vz]));
      const P2<CT> d = psub(fp.n, fm.n), e = psub(fp.psi, fm.psi);
      if (vx) S[0] = pfma(pbc(CT(SN::W(k) * vx)), d, S[0]);
      if (vy) S[1] = pfma(pbc(CT(SN::W(k) * vy)), d, S[1]);
      if (vz) S[2] = pfma(pbc(CT(SN::W(k) * vz)), d, S[2]);
      if (vx) T[0] = pfma(pbc(CT(SN::W(k) * vx)), e, T[0]);
      if (vy) T[1] = pfma(pbc(CT(SN::W(k) * vy)), e, T[1]);
      if (vz) T[2] = pfma(pbc(CT(SN::W(k) * vz)), e, T[2]);
    }
  } else {
    dn = *at(mom, o);
#pragma unroll
    for (int k = 0; k < SN::NH; ++k) {
      const int vx = SN::v(k, 0), vy = SN::v(k, 1), vz = SN::v(k, 2);
      const P2<CT> d = psub(*at(mom, o + X[H + vx] + Y[H + vy] + Z[H + vz]),
                            *at(mom, o + X[H - vx] + Y[H - vy] + Z[H - vz]));
      if (vx) S[0] = pfma(pbc(CT(SN::W(k) * vx)), d, S[0]);
      if (vy) S[1] = pfma(pbc(CT(SN::W(k) * vy)), d, S[1]);
      if (vz) S[2] = pfma(pbc(CT(SN::W(k) * vz)), d, S[2]);
    }
  }
  const P2<CT> n = padd(a.nbar, dn);
  const P2<CT> cn = pmul(pbc(a.gcross), n), cp = pmul(a.gself, psi);
  P2<CT> F[3], h[3], out[L::Q];
#pragma unroll
  for (int q = 0; q < 3; ++q) F[q] = pfma(cp, T[q], pmul(cn, pswap(S[q])));
  CT u[3];
  half_momentum<ST, CT>(j, F, a.inv_scale, h);
  common_velocity<CT>(h, n, u);
  collide_pair<kD3Q19, ST, CT, true>(a, nullptr, n, dn, u, F, out);
  check_density<CT, true>(a, n);
#pragma unroll
  for (int i = 0; i < L::Q; ++i)
    Codec2<ST, CT>::store(at(dst + (int64_t)i * a.N * 2, unsigned(s) * unsigned(2 * sizeof(ST))), out[i], a.scale);
  if constexpr (local_ref<ST>()) *at(ndst, unsigned(s) * 8u) = make_float2(float(dn.x), float(dn.y));
}

// Threads per block and the blocks per SM the register allocation must allow: eight (64 registers a thread), in FP64
// four (128).  128 threads against 256: 1-2 % faster from 64^3 up, equal below.  Six blocks (80 registers, more loads
// in flight per thread) for
//  * the FP16 moments, whose 19 pairs and 19 references a thread wait for each other otherwise: 128^3 84.5 -> 80.0 us
//    a step, with psi 95.2 -> 90.2, 256^3 with psi 724 -> 688 (BF16 and FP32: no change);
//  * the collisions of a small lattice with psi (16 bytes a neighbour), whose few waves are bound by latency: 51^3
//    10.1 -> 9.0, 65^3 15.0 -> 14.5; larger ones lose 2 % (128^3 115.1 -> 117.3);
//  * the 33 neighbours of E6 in a batch, which would spill.
constexpr int kSplitThreads = 128;
constexpr int kSmallCollide = 300000;  // sites
template <class CT>
constexpr int split_blocks(bool six = false) { return sizeof(CT) == 8 ? 4 : (six ? 6 : 8); }

template <class ST, class CT>
__global__ void __launch_bounds__(kSplitThreads, split_blocks<CT>(std::is_same<ST, __half>::value))
    sc_split_moments(const __grid_constant__ SplitArgs<CT> m) {
  const int s = blockIdx.x * kSplitThreads + threadIdx.x;
  pass_begin();
  if (s < m.a.N) split_moments<ST, CT>(m, static_cast<const ST *>(m.a.src), m.a.nsrc, s);
}

template <int STEN, class ST, class CT, bool SMALL>
__global__ void __launch_bounds__(kSplitThreads, split_blocks<CT>(SMALL))
    sc_split_collide(const __grid_constant__ SplitArgs<CT> m) {
  const int s = blockIdx.x * kSplitThreads + threadIdx.x;
  pass_begin();
  if (s < m.a.N) split_collide<STEN, ST, CT>(m, static_cast<ST *>(m.a.dst), m.a.ndst, s);
}

// Batched forms: block b takes kSplitBatchSites sites from site items[b].y of lattice items[b].x (the arguments
// args[lattice] in shared memory), source and destination swapped when swap != 0.  Two sites a thread: the
// fetch of the item and the arguments is paid once for both.
constexpr int kSplitBatchSites = 2 * kSplitThreads;

template <class CT>
__device__ __forceinline__ void split_fetch(SplitArgs<CT> &m, const SplitArgs<CT> *args, int lat) {
  static_assert(sizeof(SplitArgs<CT>) % 4 == 0 && sizeof(SplitArgs<CT>) <= 4 * 2 * kSplitThreads, "copied by words");
  const int *from = reinterpret_cast<const int *>(args + lat);
  int *to = reinterpret_cast<int *>(&m);
  for (int k = threadIdx.x; k < (int)(sizeof(SplitArgs<CT>) / 4); k += kSplitThreads) to[k] = from[k];
  __syncthreads();
}

template <class ST, class CT>
__global__ void __launch_bounds__(kSplitThreads, split_blocks<CT>(std::is_same<ST, __half>::value))
    sc_split_moments_batched(const SplitArgs<CT> *args, const int2 *items, int swap) {
  __shared__ SplitArgs<CT> m;
  const int2 it = items[blockIdx.x];
  split_fetch<CT>(m, args, it.x);
  pass_begin();
  const ST *src = static_cast<const ST *>(swap ? m.a.dst : m.a.src);
  const float2 *nsrc = swap ? m.a.ndst : m.a.nsrc;
  for (int k = 0; k < kSplitBatchSites; k += kSplitThreads) {
    const int64_t s = (int64_t)it.y + k + threadIdx.x;
    if (s < m.a.N) split_moments<ST, CT>(m, src, nsrc, (int)s);
  }
}

template <int STEN, class ST, class CT>
__global__ void __launch_bounds__(kSplitThreads, split_blocks<CT>(STEN == kE6))
    sc_split_collide_batched(const SplitArgs<CT> *args, const int2 *items, int swap) {
  __shared__ SplitArgs<CT> m;
  const int2 it = items[blockIdx.x];
  split_fetch<CT>(m, args, it.x);
  pass_begin();
  ST *dst = static_cast<ST *>(swap ? const_cast<void *>(m.a.src) : m.a.dst);
  float2 *ndst = swap ? const_cast<float2 *>(m.a.nsrc) : m.a.ndst;
  for (int k = 0; k < kSplitBatchSites; k += kSplitThreads) {
    const int64_t s = (int64_t)it.y + k + threadIdx.x;
    if (s < m.a.N) split_collide<STEN, ST, CT>(m, dst, ndst, (int)s);
  }
}

}  // namespace scgb
