// fields.cuh -- site-local kernels: layout conversion between the canonical
// FP64 host format and the even/odd chunked formats, link packing with the
// SU(3) check, noise generation, twist, precision casts and the BLAS-1 pieces
// of the reliable-update step.
#pragma once

#include "common.cuh"

namespace tsm {

constexpr int SITE_NT = 256;

// A component (complex) of a canonical spinor in storage S, as the canonical
// format's pack / unpack kernels stage it in shared memory.  PAD: words added
// to a site's row so that the column accesses of a warp spread over the banks.
template <class S> struct CanonComp;
template <> struct CanonComp<F64> {
  using type = double2;
  static constexpr int PAD = 1;
  static __device__ __forceinline__ type pack(double2 d) { return d; }
  static __device__ __forceinline__ double2 unpack(type v) { return v; }
};
template <> struct CanonComp<F32> {
  using type = float2;
  static constexpr int PAD = 1;
  static __device__ __forceinline__ type pack(double2 d) { return make_float2(narrow_f32(d.x), narrow_f32(d.y)); }
  static __device__ __forceinline__ double2 unpack(type v) { return make_double2(widen_f64(v.x), widen_f64(v.y)); }
};
template <class S> struct CanonComp16 {
  using type = uint32_t;
  static constexpr int PAD = 1;
  static __device__ __forceinline__ type pack(double2 d) {
    return Pack16<S>::pack(cx<float>{narrow_f32(d.x), narrow_f32(d.y)});
  }
  static __device__ __forceinline__ double2 unpack(type v) {
    const cx<float> c = Pack16<S>::unpack(v);
    return make_double2(widen_f64(c.re), widen_f64(c.im));
  }
};
template <> struct CanonComp<F16> : CanonComp16<F16> {};
template <> struct CanonComp<BF16> : CanonComp16<BF16> {};

constexpr int CANON_SITES = 128;   // lexicographic sites per block: 64 half-lattice indices of each parity

// Canonical spinors (24 doubles per lexicographic site) <-> even / odd fields
// in S, batched over blockIdx.y.  A block moves 128 consecutive sites through
// shared memory, so that both sides are read and written in whole lines (one
// thread per site touched 32 lines per warp and component): memory-bound.
// 24^3x48 in FP32, both parities: 191 MB in 37 us (pack), 35 us (unpack).
// A null field is not written (pack) or reads as zero (unpack).
template <class S>
__global__ void __launch_bounds__(SITE_NT) pack_spinor_kernel(Geom g, const double2* __restrict__ canon,
                                                              typename S::schunk* __restrict__ even,
                                                              typename S::schunk* __restrict__ odd, int sstride) {
  using C = CanonComp<S>;
  using T = typename C::type;
  constexpr int ROW = 12 + C::PAD, PER = 12 / S::SN;   // components per chunk
  __shared__ __align__(16) T sh[CANON_SITES * ROW];
  const int base = blockIdx.x * CANON_SITES, n = min(CANON_SITES, g.V - base);
  canon += (size_t)blockIdx.y * g.V * 12 + (size_t)base * 12;
  for (int e = threadIdx.x; e < n * 12; e += SITE_NT) {
    const int site = e / 12;
    sh[site * ROW + (e - site * 12)] = C::pack(canon[e]);
  }
  __syncthreads();
  const int half = n >> 1, h0 = base >> 1;
  for (int e = threadIdx.x; e < S::SN * n; e += SITE_NT) {
    const int k = e / n, rest = e - k * n, par = rest >= half, i = rest - par * half;
    typename S::schunk* out = par ? odd : even;
    if (out == nullptr) continue;
    int c[4];
    site_coords(g, par, h0 + i, c);
    const T* v = sh + (2 * i + (c[0] & 1)) * ROW + k * PER;
    typename S::schunk w;
    T* wt = reinterpret_cast<T*>(&w);
#pragma unroll
    for (int u = 0; u < PER; ++u) wt[u] = v[u];
    out[rhs_offset<S>(blockIdx.y, sstride) + (size_t)k * sstride + h0 + i] = w;
  }
}

template <class S>
__global__ void __launch_bounds__(SITE_NT) unpack_spinor_kernel(Geom g, const typename S::schunk* __restrict__ even,
                                                                const typename S::schunk* __restrict__ odd,
                                                                int sstride, double2* __restrict__ canon) {
  using C = CanonComp<S>;
  using T = typename C::type;
  constexpr int ROW = 12 + C::PAD, PER = 12 / S::SN;
  __shared__ __align__(16) T sh[CANON_SITES * ROW];
  const int base = blockIdx.x * CANON_SITES, n = min(CANON_SITES, g.V - base);
  const int half = n >> 1, h0 = base >> 1;
  for (int e = threadIdx.x; e < S::SN * n; e += SITE_NT) {
    const int k = e / n, rest = e - k * n, par = rest >= half, i = rest - par * half;
    const typename S::schunk* in = par ? odd : even;
    int c[4];
    site_coords(g, par, h0 + i, c);
    typename S::schunk w{};
    if (in != nullptr) w = in[rhs_offset<S>(blockIdx.y, sstride) + (size_t)k * sstride + h0 + i];
    T* v = sh + (2 * i + (c[0] & 1)) * ROW + k * PER;
    const T* wt = reinterpret_cast<const T*>(&w);
#pragma unroll
    for (int u = 0; u < PER; ++u) v[u] = wt[u];
  }
  __syncthreads();
  canon += (size_t)blockIdx.y * g.V * 12 + (size_t)base * 12;
  for (int e = threadIdx.x; e < n * 12; e += SITE_NT) {
    const int site = e / 12;
    canon[e] = C::unpack(sh[site * ROW + (e - site * 12)]);
  }
}

// canonical links [lex][mu][3][3] complex -> parity fields in every storage
// (FP64: 3 rows, FP32 and 16-bit: 2 rows, tensor-core stencil: see F16G);
// records the largest squared deviation from SU(3).  A block moves the links of
// 64 consecutive sites through shared memory, so that the reads and the stores
// of a direction run over consecutive sites.  Bound by the FP64 pipe: the check
// takes 64 FP64 instructions per link, products as chains of multiply-adds (2.7
// million links at 24^3x48: 290 us at two results per SM and clock; load_gauge
// 732 -> 648 us against sums of separate products); squares, compared as
// integers, need no square root or FP64 comparison, and the narrowing runs on
// the integer pipe.
constexpr int LINK_SITES = 64;

static __global__ void __launch_bounds__(SITE_NT) pack_links_kernel(Geom g, const double2* __restrict__ U,
                                                             double2* __restrict__ l64, float4* __restrict__ l32,
                                                             uint2* __restrict__ l16, uint2* __restrict__ lbf,
                                                             uint32_t* __restrict__ lmma, int lstride,
                                                             unsigned long long* __restrict__ maxdev2) {
  constexpr int ROW = 4 * 9 + 1;   // a site's links, padded by one entry
  __shared__ double2 sh[LINK_SITES * ROW];
  const int base = blockIdx.x * LINK_SITES, n = min(LINK_SITES, g.V - base);
  for (int e = threadIdx.x; e < n * 36; e += SITE_NT) {
    const int site = e / 36;
    sh[site * ROW + (e - site * 36)] = U[(size_t)base * 36 + e];
  }
  __syncthreads();
  const int mu = threadIdx.x >> 6, local = threadIdx.x & 63;
  unsigned long long dev2 = 0ull;
  if (local < n) {
    const int lex = base + local;
    const int ih = lex >> 1;
    int c[4];
    site_coords(g, 0, ih, c);
    const int parity = (lex & 1) != (c[0] & 1);   // c: the even site of the pair
    c[0] = (c[0] & ~1) | (lex & 1);
    const double2* m = sh + local * ROW + mu * 9;
    cx<double> r[9], w[3];
#pragma unroll
    for (int k = 0; k < 9; ++k) r[k] = {m[k].x, m[k].y};
    // the reconstructed row 2, conj(row0 x row1), as chains of multiply-adds
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const cx<double> x = r[(k + 1) % 3], y = r[3 + (k + 2) % 3], u = r[(k + 2) % 3], v = r[3 + (k + 1) % 3];
      w[k] = cconj(cmac(x * y, cx<double>{-u.re, -u.im}, v));
    }
    auto norm2_add = [](double acc, cx<double> a) { return fma(a.im, a.im, fma(a.re, a.re, acc)); };
    // SU(3) check: unit rows, orthogonal rows, stored row 2 equals the reconstruction
    auto worse = [&](double sq) {   // squares are non-negative: their bits order like the values, NaN on top
      const unsigned long long b = (unsigned long long)__double_as_longlong(sq) & 0x7fffffffffffffffull;
      dev2 = b > dev2 ? b : dev2;
    };
    const double n0 = norm2_add(norm2_add(norm2_add(-1.0, r[0]), r[1]), r[2]);
    const double n1 = norm2_add(norm2_add(norm2_add(-1.0, r[3]), r[4]), r[5]);
    worse(n0 * n0);
    worse(n1 * n1);
    worse(norm2(cjmac(cjmac(cjmul(r[0], r[3]), r[1], r[4]), r[2], r[5])));
#pragma unroll
    for (int k = 0; k < 3; ++k) worse(norm2(r[6 + k] - w[k]));
    const size_t off64 = (size_t)parity * 4 * F64::LN * lstride;
    const size_t off32 = (size_t)parity * 4 * F32::LN * lstride;
    store_link<F64>(l64 + off64, lstride, mu, ih, r);   // all three rows
    cx<float> rf[9];
#pragma unroll
    for (int k = 0; k < 6; ++k) rf[k] = {narrow_f32(r[k].re), narrow_f32(r[k].im)};
    store_link<F32>(l32 + off32, lstride, mu, ih, rf);
    store_link<F16>(l16 + off32, lstride, mu, ih, rf);
    store_link<BF16>(lbf + off32, lstride, mu, ih, rf);
    if (lmma != nullptr) {
      // tensor-core stencil: rows 0, 1 in FP16, row 2 = conj(row0 x row1) of those as FP16 hi + lo
      uint32_t w12[12], wlo[3];   // wlo: the scaled remainders of a forward link
      cx<float> q[6], lo[3];
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        w12[k] = Pack16<F16>::pack(rf[k]);
        q[k] = Pack16<F16>::unpack(w12[k]);
      }
      third_row_pair(q, w12 + 6, lo);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        w12[9 + k] = Pack16<F16>::pack(lo[k]);
        wlo[k] = Pack16<F16>::pack(F16G::LO_SCALE * lo[k]);
      }
      // [site][hop][12]: forward hop of this site, backward hop of x + mu, with the sign of an antiperiodic boundary
      bool wraps = false;
#pragma unroll
      for (int d = 0; d < 4; ++d)
        if (d == mu) {
          wraps = c[d] + 1 == g.L[d];
          c[d] = wraps ? 0 : c[d] + 1;
        }
      const uint32_t sign = wraps && mu == 3 && g.apbc ? 0x80008000u : 0u;
      const int fh = half_index(g, c[0], c[1], c[2], c[3]);
      uint4* own = reinterpret_cast<uint4*>(lmma) + (((size_t)parity * g.Vh + ih) * 8 + 2 * mu) * 3;
      uint4* fwd = reinterpret_cast<uint4*>(lmma) + (((size_t)(1 - parity) * g.Vh + fh) * 8 + 2 * mu + 1) * 3;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const uint4 v = make_uint4(w12[4 * k] ^ sign, w12[4 * k + 1] ^ sign, w12[4 * k + 2] ^ sign, w12[4 * k + 3] ^ sign);
        own[k] = k < 2 ? v : make_uint4(v.x, wlo[0] ^ sign, wlo[1] ^ sign, wlo[2] ^ sign);
        fwd[k] = v;
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, dev2, o);
    dev2 = v > dev2 ? v : dev2;
  }
  if ((threadIdx.x & 31) == 0 && dev2 > *reinterpret_cast<volatile unsigned long long*>(maxdev2))
    atomicMax(maxdev2, dev2);
}

// Thread -> (right-hand side, site) of the batched site-local kernels on
// grouped storage (F16G): 8 sources x 32 sites per block of 256 threads,
// sources fastest, so that a warp touches whole lines of the grouped side.
__device__ __forceinline__ bool grouped_site(int Vh, int nrhs, int* rhs, int* ih) {
  *rhs = blockIdx.y * 8 + (threadIdx.x & 7);
  *ih = blockIdx.x * (SITE_NT / 8) + (threadIdx.x >> 3);
  return *rhs < nrhs && *ih < Vh;
}

static __global__ void __launch_bounds__(SITE_NT) noise_grouped_kernel(Geom g, int parity, NoiseSpec n,
                                                                       uint32_t source0, uint4* __restrict__ out,
                                                                       int sstride, int nrhs) {
  int rhs, ih;
  if (!grouped_site(g.Vh, nrhs, &rhs, &ih)) return;
  int c[4];
  site_coords(g, parity, ih, c);
  const uint32_t lex = (uint32_t)(((c[3] * g.L[2] + c[2]) * g.L[1] + c[1]) * g.L[0] + c[0]);
  cx<float> v[12];
  noise_site<float>(n, lex, source0 + (uint32_t)rhs, v);
  store_spinor<F16G>(out + rhs_offset<F16G>(rhs, sstride), sstride, ih, v);
}

static __global__ void __launch_bounds__(SITE_NT) twist_grouped_kernel(int Vh, TwistF f, const uint4* __restrict__ in,
                                                                       uint4* __restrict__ out, int sstride,
                                                                       int nrhs) {
  int rhs, ih;
  if (!grouped_site(Vh, nrhs, &rhs, &ih)) return;
  const size_t off = rhs_offset<F16G>(rhs, sstride);
  cx<float> v[12];
  load_spinor<F16G>(in + off, sstride, ih, v);
  apply_twist(f, v);
  store_spinor<F16G>(out + off, sstride, ih, v);
}

template <class Si, class So>
__global__ void __launch_bounds__(SITE_NT) convert_grouped_kernel(int Vh, const typename Si::schunk* __restrict__ in,
                                                                  typename So::schunk* __restrict__ out, int sstride,
                                                                  int nrhs) {
  int rhs, ih;
  if (!grouped_site(Vh, nrhs, &rhs, &ih)) return;
  cx<typename Si::real> v[12];
  cx<typename So::real> w[12];
  load_spinor<Si>(in + rhs_offset<Si>(rhs, sstride), sstride, ih, v);
#pragma unroll
  for (int k = 0; k < 12; ++k) w[k] = {(typename So::real)v[k].re, (typename So::real)v[k].im};
  store_spinor<So>(out + rhs_offset<So>(rhs, sstride), sstride, ih, w);
}

// noise sources source0 + rhs -> batch of parity fields in S (eta is exactly
// representable in every tier except the 1/sqrt 2 amplitude, rounded once).
// Grid: x = right-hand side, y = blocks of SITE_NT sites.
template <class S>
__global__ void __launch_bounds__(SITE_NT) noise_kernel(Geom g, int parity, NoiseSpec n, uint32_t source0,
                                                        typename S::schunk* __restrict__ out, int sstride) {
  using R = typename S::real;
  const int rhs = blockIdx.x;
  const int ih = blockIdx.y * SITE_NT + threadIdx.x;
  if (ih >= g.Vh) return;
  int c[4];
  site_coords(g, parity, ih, c);
  const uint32_t lex = (uint32_t)(((c[3] * g.L[2] + c[2]) * g.L[1] + c[1]) * g.L[0] + c[0]);
  cx<R> v[12];
  noise_site<R>(n, lex, source0 + (uint32_t)rhs, v);
  store_spinor<S>(out + rhs_offset<S>(rhs, sstride), sstride, ih, v);
}

// noise source in the canonical layout (for exact comparisons)
static __global__ void __launch_bounds__(SITE_NT) noise_canon_kernel(int V, NoiseSpec n, uint32_t source,
                                                                     double2* __restrict__ out) {
  const int lex = blockIdx.x * SITE_NT + threadIdx.x;
  if (lex >= V) return;
  cx<double> v[12];
  noise_site<double>(n, (uint32_t)lex, source, v);
#pragma unroll
  for (int k = 0; k < 12; ++k) out[(size_t)lex * 12 + k] = make_double2(v[k].re, v[k].im);
}

// out = f * in (site-local chiral twist); a RHS with st[rhs].done is skipped
template <class S>
__global__ void __launch_bounds__(SITE_NT) twist_kernel(int Vh, Twist f, const typename S::schunk* __restrict__ in,
                                                        typename S::schunk* __restrict__ out, int sstride,
                                                        const int* active, const CGState* st) {
  const int rhs = rhs_slot(active);
  if (st != nullptr && st[rhs].done) return;
  const int ih = blockIdx.y * SITE_NT + threadIdx.x;
  if (ih >= Vh) return;
  const size_t off = rhs_offset<S>(rhs, sstride);
  cx<typename S::real> v[12];
  load_spinor<S>(in + off, sstride, ih, v);
  apply_twist(f, v);
  store_spinor<S>(out + off, sstride, ih, v);
}

// out (So) = in (Si), precision cast; in == nullptr writes zero
template <class Si, class So>
__global__ void __launch_bounds__(SITE_NT) convert_kernel(int Vh, const typename Si::schunk* __restrict__ in,
                                                          typename So::schunk* __restrict__ out, int sstride,
                                                          const int* active) {
  const int rhs = rhs_slot(active);
  const int ih = blockIdx.y * SITE_NT + threadIdx.x;
  if (ih >= Vh) return;
  cx<typename Si::real> v[12];
  cx<typename So::real> w[12];
  if (in != nullptr) {
    load_spinor<Si>(in + rhs_offset<Si>(rhs, sstride), sstride, ih, v);
#pragma unroll
    for (int k = 0; k < 12; ++k) w[k] = {(typename So::real)v[k].re, (typename So::real)v[k].im};
  } else {
#pragma unroll
    for (int k = 0; k < 12; ++k) w[k] = {0, 0};
  }
  store_spinor<So>(out + rhs_offset<So>(rhs, sstride), sstride, ih, w);
}

// reliable update, step 1: x64 += y (y in F32), y = 0 -- only for right-hand
// sides with a pending update (st[rhs].need_rel)
static __global__ void __launch_bounds__(SITE_NT) accumulate_solution_kernel(int Vh, float4* __restrict__ y,
                                                                             double2* __restrict__ x, int sstride,
                                                                             const int* active, const CGState* st) {
  const int rhs = rhs_slot(active);
  if (!st[rhs].need_rel) return;
  const int ih = blockIdx.y * SITE_NT + threadIdx.x;
  if (ih >= Vh) return;
  y += rhs_offset<F32>(rhs, sstride);
  x += rhs_offset<F64>(rhs, sstride);
  cx<float> yv[12];
  cx<double> xv[12];
  load_spinor<F32>(y, sstride, ih, yv);
  load_spinor<F64>(x, sstride, ih, xv);
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    xv[k] = xv[k] + cx<double>{(double)yv[k].re, (double)yv[k].im};
    yv[k] = {0.f, 0.f};
  }
  store_spinor<F64>(x, sstride, ih, xv);
  store_spinor<F32>(y, sstride, ih, yv);
}

// FP64 -> FP32 copy of a field for the right-hand sides with a reliable
// update pending (the others return at once)
static __global__ void __launch_bounds__(SITE_NT) rel_narrow_kernel(int Vh, const double2* __restrict__ in,
                                                                    float4* __restrict__ out, int sstride,
                                                                    const int* active, const CGState* st) {
  const int rhs = rhs_slot(active);
  if (!st[rhs].need_rel) return;
  const int ih = blockIdx.y * SITE_NT + threadIdx.x;
  if (ih >= Vh) return;
  cx<double> v[12];
  cx<float> w[12];
  load_spinor<F64>(in + rhs_offset<F64>(rhs, sstride), sstride, ih, v);
#pragma unroll
  for (int k = 0; k < 12; ++k) w[k] = {(float)v[k].re, (float)v[k].im};
  store_spinor<F32>(out + rhs_offset<F32>(rhs, sstride), sstride, ih, w);
}

// after a residual replacement the search direction restarts from the new
// residual, p = r: after many FP32 iterations the iterated residual can lie
// orders of magnitude below the true one, and the old direction would no
// longer be conjugate to the replaced residual
static __global__ void __launch_bounds__(SITE_NT) restart_direction_kernel(int Vh, const float4* __restrict__ r,
                                                                           float4* __restrict__ p, int sstride,
                                                                           const int* active, const CGState* st) {
  const int rhs = rhs_slot(active);
  if (!st[rhs].need_rel) return;
  const int ih = blockIdx.y * SITE_NT + threadIdx.x;
  if (ih >= Vh) return;
  cx<float> w[12];
  load_spinor<F32>(r + rhs_offset<F32>(rhs, sstride), sstride, ih, w);
  store_spinor<F32>(p + rhs_offset<F32>(rhs, sstride), sstride, ih, w);
}

// closes the reliable updates of one iteration: clears need_rel and, where the
// iterated residual had met the stopping rule, lets the true FP64 residual
// decide between stopping and iterating on
static __global__ void rel_finish_kernel(CGState* st, const int* active, int n) {
  const int k = threadIdx.x + blockIdx.x * blockDim.x;
  if (k >= n) return;
  CGState& s = st[active != nullptr ? active[k] : k];
  if (!s.need_rel) return;
  s.need_rel = 0;
  if (s.final_check) {
    s.final_check = 0;
    if (s.status != 0 || s.iter >= s.max_iter || rule_met(&s, s.rr)) s.done = 1;
  }
}

// a warm-started solve asks every iterating source for a residual replacement
// before its first iteration; final_check lets rel_finish_kernel stop a source
// whose starting guess already meets the rule
static __global__ void warm_start_kernel(CGState* st, int n) {
  const int k = threadIdx.x + blockIdx.x * blockDim.x;
  if (k >= n) return;
  CGState& s = st[k];
  if (s.done || s.status != 0) return;
  s.need_rel = 1;
  s.final_check = 1;
}

// states 0 .. n-1: fresh solve
static __global__ void state_init_kernel(CGState* st, int n, double tol, int max_iter, int rel, double delta2) {
  const int k = threadIdx.x + blockIdx.x * blockDim.x;
  if (k >= n) return;
  CGState& s = st[k];
  s.tol = tol;
  s.max_iter = max_iter;
  s.iter = 0;
  s.done = 0;
  s.status = 0;
  s.rel = rel;
  s.need_rel = 0;
  s.final_check = 0;
  s.delta2 = delta2;
  s.rr = s.rr0 = s.pAp = s.alpha = s.beta = s.aux = s.rr_ref = 0.0;
  s.alpha_f = s.beta_f = 0.0f;
}

}  // namespace tsm
