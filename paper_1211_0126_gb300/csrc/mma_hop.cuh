// mma_hop.cuh -- the FP16 tier's batched hopping stencil on the tensor cores.
//
// For one output site the SU(3) products of all right-hand sides are one
// contraction over (hop, colour): acc[source, spin][colour] = sum over the 8
// hops and 3 colours of h[source, spin][hop, colour] U[hop, colour][colour],
// with the projected half spinors h in FP16 (they are sums of two stored FP16
// values, rounded as in project_f16) and the links in FP16.  A warp takes one
// site and 8 sources and issues mma.sync m16n8k16 (FP16 operands, FP32
// accumulators): 8 of them replace the 576 FP32 multiply-adds per source.
//
//   rows (16)      8 sources x the two spins of the half spinor
//   columns (8)    3 colours x (re, im); columns 6, 7 see below
//   k (16)         two hops x 4 slots of (re, im): colours 0..2, slot 3 below
//
// The operand fragments make every step lane-local (lane = 4 * row + q):
// lane (row, q) loads the 16-byte chunk "colour q" of its source -- the four
// spins of that colour -- projects it, and that word is its A fragment; the D
// fragment of the lane is again (spin pair, colour q), so after the lower spin
// components are added up the lane holds the four spins of colour q and stores
// one 16-byte chunk.  Hence the storage F16G: per group of 8 sources, [site]
// [source][colour] chunks of four spins; a warp's load of one neighbour is 384
// contiguous bytes.
//
// Row 2 of a link, conj(row0 x row1), is kept as an FP16 pair hi + lo of its exact
// value: the lo part of a forward link, scaled by 2^11, sits in columns 6, 7 (added
// to colour 2 afterwards), that of a backward link in k slot 3, which carries
// colour 2 of the half spinor a second time.  Products are exact, sums FP32: the 16
// products of a direction on the tensor cores, which round towards zero, the four
// directions by additions.  Rounding error of H psi against 64 bits on the same FP16
// fields and links, relative rms: 6.97e-8 on random links (9.98e-8 with one
// accumulator over the directions and the pair of an FP32 row; FP32 sums of products
// with row 2 in FP32 7.03e-8), 0.978 of the FP32 products' near the identity.
//
// The lower spin components are the same products times a phase and in one
// of two orders: the MMA of a direction is issued a second time with the
// phase i^k and the sign folded into its B words; the directions x, y and z, t
// share an accumulator each.
//
// Neighbours reach the warps through shared memory: a block works on tiles of
// 2 x 2 rows (y, z) of up to W = 4 or 6 half-sites in x, one site per warp, and four
// more warps copy the tile's distinct neighbour sites (92 instead of 8 x 16 at W = 4) for
// one group of 8 sources per ring stage with TMA: the own rows as one box of
// (W + 2) x 2 x 2 sites, the y, z and t edges as two boxes each, and the sites
// that wrap around in x (at most 4, where a box has zeros) as plain bulk copies.
// The centre fields of the epilogues arrive in the same stage.
#pragma once

#include <cuda.h>

#include "dslash.cuh"
#include "mbar.cuh"

namespace tsm {

constexpr int MMA_COPIERS = 4;                       // copy warps (one thread each)
constexpr int MMA_GROUPS = 8;                        // groups of 8 sources of a batch at most
constexpr int MMA_FLUSH = 8;                         // tiles whose norms add up in FP32 before they join the FP64 sum
constexpr int MMA_CHUNKS = 24;                       // 16-byte chunks per site of a group
constexpr long long MMA_SPIN_LIMIT = 1ll << 22;      // polls of a ring wait
constexpr long long MMA_INJECT_LIMIT = 4096;         // the same where the copies are withheld (tests)

// A tile of 2 x 2 rows of W half-sites: a warp per site and the copy warps (one
// thread each).  Slots (sites) of a ring stage: the own rows [zz][yy][W + 2] from
// x0 - 1 on (the sites x +- 1 of the other parity; they are also the y and z
// neighbours inside the tile), the wrapped site of each row, the edges
// [e][row][W] in y, z and t, then the rows [zz][yy][W] of the centre fields.
template <int TW> struct MmaShape {
  static constexpr int W = TW, WARPS = 4 * W, NT = 32 * (WARPS + MMA_COPIERS);
  static constexpr int WRAP = 4 * (W + 2), Y = WRAP + 4, Z = Y + 4 * W, T = Z + 4 * W, F = T + 8 * W;
  static constexpr bool LINKS_SMEM = W > 4;   // the next tile's link words wait in shared memory instead of registers
  static constexpr int LINK_BYTES = LINKS_SMEM ? WARPS * 96 * 4 : 0;
};

// box shapes (x, y, z sites) of the tensor maps of a shape
enum MmaBox { MMA_BOX_OWN = 0, MMA_BOX_Y = 1, MMA_BOX_Z = 2, MMA_BOX_TILE = 3, MMA_BOXES = 4 };
inline void mma_box(int k, int w, int box[3]) {
  box[0] = k == MMA_BOX_OWN ? w + 2 : w;
  box[1] = k == MMA_BOX_Y ? 1 : 2;
  box[2] = k == MMA_BOX_Z ? 1 : 2;
}

enum { MMA_HOP = 0, MMA_HOP_CENTER = 1, MMA_HOP_CENTER_NORM = 3, MMA_UPDATE = 8 };

template <int MODE, class SH> struct MmaStage {
  static constexpr int FIELDS = MODE == MMA_HOP ? 0 : MODE == MMA_UPDATE ? 4 : 1;
  static constexpr int SLOTS = SH::F + 4 * SH::W * FIELDS;
  static constexpr int BYTES = SLOTS * MMA_CHUNKS * 16;
  static constexpr int COUNT = (MODE == MMA_HOP ? 5 : MODE == MMA_UPDATE ? 3 : 4) - (SH::W > 4);
  static constexpr int SMEM = BYTES * COUNT + SH::LINK_BYTES;
};

// tiles of a lattice: ntx x nyp x nzp x T, x fastest; gx .. gt: the grid's
// stride in the same mixed radix
struct MmaTiles {
  int Lxh, Ly, Lz, T, W, ntx, nyp, nzp, ntiles;
  int gx, gy, gz, gt;
};

struct MmaTile {
  int tx, yp, zp, t;
  __device__ __forceinline__ MmaTile(const MmaTiles& g, int i) {
    tx = i % g.ntx;
    i /= g.ntx;
    yp = i % g.nyp;
    i /= g.nyp;
    zp = i % g.nzp;
    t = i / g.nzp;
  }
  __device__ __forceinline__ void next(const MmaTiles& g) {
    tx += g.gx;
    int c = tx >= g.ntx;
    tx -= c ? g.ntx : 0;
    yp += g.gy + c;
    c = yp >= g.nyp;
    yp -= c ? g.nyp : 0;
    zp += g.gz + c;
    c = zp >= g.nzp;
    zp -= c ? g.nzp : 0;
    t += g.gt + c;
  }
};

struct MmaMaps {
  CUtensorMap in[MMA_BOXES];   // the input field (other parity)
  CUtensorMap f[4];            // centre fields: K2 centre; K4 w, p, r, x
};

struct MmaHopArgs {
  MmaTiles tl;
  int Vh, parity;
  const uint32_t* links;       // words [site][hop][12] of the output parity, boundary sign included
  const uint4* in;             // the other parity
  uint4* out;                  // hops
  TwistF fto_ah, fto_tc_ac, fts;
  uint4* r;                    // K4
  uint4* x;
  float kappa2;
  const int* active;
  int nrhs;
  const CGState* skip;         // sources with skip[src].done are left out
  CGState* st;
  int post;
  RedSlot red;
  int* err;                    // host-mapped: set when a ring wait ran out
  int withhold;                // fault injection: no copies, ring waits of MMA_INJECT_LIMIT polls
};

// ring wait: one try, then the bounded loop; true on timeout
__device__ __forceinline__ bool mma_wait_failed(uint64_t* bar, uint32_t parity, int withhold) {
  return !mbar_try(bar, parity) && !mbar_wait(bar, parity, withhold ? MMA_INJECT_LIMIT : MMA_SPIN_LIMIT);
}

// d = a b (no accumulator: the tensor cores round a sum towards zero, so that only
// the 16 products of one direction are added there)
__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ uint32_t h2_fma(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
__device__ __forceinline__ uint32_t h2_swap(uint32_t a) { return __byte_perm(a, 0u, 0x1032); }
// p + i v and p - i v of words (re, im): the swapped word times (-1, +1) or
// (+1, -1), one rounding of the exact sum (the values of h2_add / h2_sub)
__device__ __forceinline__ uint32_t h2_add_i(uint32_t p, uint32_t v) { return h2_fma(h2_swap(v), 0x3C00BC00u, p); }
__device__ __forceinline__ uint32_t h2_sub_i(uint32_t p, uint32_t v) { return h2_fma(h2_swap(v), 0xBC003C00u, p); }

// the two projected spins (1 + SG gamma_MU) of one colour
template <int MU, int SG>
__device__ __forceinline__ void project_word(const uint4 u, uint32_t& h0, uint32_t& h1) {
  if constexpr (MU == 0) {
    h0 = SG > 0 ? h2_sub_i(u.x, u.w) : h2_add_i(u.x, u.w);
    h1 = SG > 0 ? h2_sub_i(u.y, u.z) : h2_add_i(u.y, u.z);
  } else if constexpr (MU == 1) {
    h0 = SG > 0 ? h2_sub(u.x, u.w) : h2_add(u.x, u.w);
    h1 = SG > 0 ? h2_add(u.y, u.z) : h2_sub(u.y, u.z);
  } else if constexpr (MU == 2) {
    h0 = SG > 0 ? h2_sub_i(u.x, u.z) : h2_add_i(u.x, u.z);
    h1 = SG > 0 ? h2_add_i(u.y, u.w) : h2_sub_i(u.y, u.w);
  } else {
    h0 = SG > 0 ? h2_add(u.x, u.z) : h2_sub(u.x, u.z);
    h1 = SG > 0 ? h2_add(u.y, u.w) : h2_sub(u.y, u.w);
  }
}

// Lane constants of the B words.  Column n = lane / 4 is colour c = n / 2
// (3: the lo columns) and part n % 2; k slot q = lane % 4 is colour q (3: the
// lo slot).  With V the (phase times) link entry, the word is (Vr, -Vi) in the
// real column and (Vi, Vr) in the imaginary one.
struct MmaLane {
  int wf, wb;                    // word of a forward / backward link
  uint32_t mf, mb;               // 0 where the entry is zero
  uint32_t sel, seli;            // byte orders for V = W and V = i W
  uint32_t xf, xb, xif, xib;     // signs for W, W^dag, i W, i W^dag
  __device__ __forceinline__ explicit MmaLane(int lane) {
    const int n = lane >> 2, q = lane & 3, c = n >> 1, part = n & 1;
    wf = q < 3 ? c * 3 + q : 0;
    wb = c < 3 ? q * 3 + c : 0;
    mf = q < 3 ? 0xffffffffu : 0u;
    mb = c < 3 ? 0xffffffffu : 0u;
    sel = part ? 0x1032u : 0x3210u;
    seli = part ? 0x3210u : 0x1032u;
    xf = part ? 0u : 0x80000000u;
    xb = part ? 0x00008000u : 0u;
    xif = part ? 0x80000000u : 0x80008000u;
    xib = part ? 0u : 0x80000000u;
  }
};

// B words of direction MU: b = W (forward), W^dag (backward); bl = the same
// times the phase and sign of the lower components
template <int DAG, int MU>
__device__ __forceinline__ void make_b(const MmaLane& L, uint32_t rf, uint32_t rb, uint32_t (&b)[2],
                                       uint32_t (&bl)[2]) {
  constexpr uint32_t NEG = 0x80008000u;
  constexpr uint32_t sf = DAG ? 0u : NEG, sb = DAG ? NEG : 0u;   // s of the forward / backward projector
  b[0] = (__byte_perm(rf, 0u, L.sel) ^ L.xf) & L.mf;
  b[1] = (__byte_perm(rb, 0u, L.sel) ^ L.xb) & L.mb;
  if constexpr (MU == 0 || MU == 2) {
    bl[0] = (__byte_perm(rf, 0u, L.seli) ^ (L.xif ^ sf)) & L.mf;
    bl[1] = (__byte_perm(rb, 0u, L.seli) ^ (L.xib ^ sb)) & L.mb;
  } else {
    bl[0] = sf ? b[0] ^ NEG : b[0];
    bl[1] = sb ? b[1] ^ NEG : b[1];
  }
}

// chunk offsets of a site's neighbours in a stage: t + 1 two rows of edges after t - 1
struct MmaSlots {
  int xf, xb, yf, yb, zf, zb, t;
};

// H psi (or H^dag psi) of one site for 8 sources: nb points at the lane's chunk
// of the stage.
// acc: four spins of colour q (lanes q = 3: the lo part of colour 2)
template <int DAG, int W>
__device__ __forceinline__ void mma_site(const uint4* nb, const MmaSlots& sl, const uint32_t (&B)[4][2],
                                         const uint32_t (&BL)[4][2], float (&acc)[8]) {
  constexpr int SF = DAG ? +1 : -1;
  uint32_t a[4];
  float d[4], e[4];   // a direction's upper and lower components
  project_word<0, SF>(nb[sl.xf], a[0], a[1]);
  project_word<0, -SF>(nb[sl.xb], a[2], a[3]);
  mma_f16(d, a, B[0][0], B[0][1]);
  mma_f16(e, a, BL[0][0], BL[0][1]);       // rows: spin 3 | spin 2
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    acc[k] = d[k];
    acc[4 + k] = e[k ^ 2];
  }
  project_word<1, SF>(nb[sl.yf], a[0], a[1]);
  project_word<1, -SF>(nb[sl.yb], a[2], a[3]);
  mma_f16(d, a, B[1][0], B[1][1]);
  mma_f16(e, a, BL[1][0], BL[1][1]);       // rows: -spin 3 | spin 2
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    acc[k] += d[k];
    acc[4 + k] += k < 2 ? e[k ^ 2] : -e[k ^ 2];
  }
  project_word<2, SF>(nb[sl.zf], a[0], a[1]);
  project_word<2, -SF>(nb[sl.zb], a[2], a[3]);
  mma_f16(d, a, B[2][0], B[2][1]);
  mma_f16(e, a, BL[2][0], BL[2][1]);       // rows: spin 2 | -spin 3
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    acc[k] += d[k];
    acc[4 + k] += k < 2 ? e[k] : -e[k];
  }
  project_word<3, SF>((nb + sl.t)[4 * W * MMA_CHUNKS], a[0], a[1]);
  project_word<3, -SF>(nb[sl.t], a[2], a[3]);
  mma_f16(d, a, B[3][0], B[3][1]);
  mma_f16(e, a, BL[3][0], BL[3][1]);       // rows: spin 2 | spin 3
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    acc[k] += d[k];
    acc[4 + k] += e[k];
  }
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float lo = __shfl_sync(0xffffffffu, acc[k], lane | 3);
    if ((lane & 3) == 2) acc[k] = fmaf(lo, 1.f / F16G::LO_SCALE, acc[k]);
  }
}

__device__ __forceinline__ void unpack4(const uint4 u, float (&v)[8]) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const cx<float> c = Pack16<F16>::unpack(w[s]);
    v[2 * s] = c.re;
    v[2 * s + 1] = c.im;
  }
}
__device__ __forceinline__ uint4 pack4(const float (&v)[8]) {
  return make_uint4(Pack16<F16>::pack({v[0], v[1]}), Pack16<F16>::pack({v[2], v[3]}), Pack16<F16>::pack({v[4], v[5]}),
                    Pack16<F16>::pack({v[6], v[7]}));
}
__device__ __forceinline__ void twist4(const TwistF& f, float (&v)[8]) {
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const cx<float> a = {f.re[s >> 1], f.im[s >> 1]};
    const cx<float> q = a * cx<float>{v[2 * s], v[2 * s + 1]};
    v[2 * s] = q.re;
    v[2 * s + 1] = q.im;
  }
}

__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, int t,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], "
      "[%7];" ::"r"(dst),
      "l"(map), "r"(0), "r"(x), "r"(y), "r"(z), "r"(t), "r"(smem_u32(bar))
      : "memory");
}

// K4 is bound by HBM.  K1-K3 are bound within the SM, by no single unit: copies
// and stores alone take 192 us where K1 takes 290, arithmetic on resident data
// alone 291 (24^3x48, 24 sources, W = 4); issue slots 67 % busy, shared-memory
// wavefronts 55 % and the copies' writes beside them, HMMA 19 %, in chains of 1350
// cycles a site and group that four warps per scheduler overlap.  W = 6 has six
// (24 + 4 warps at 72 registers: the next link words wait in shared memory, the lane
// constants are formed per tile) and fewer neighbour sites per output site (5.5
// against 5.75).  24^3x48, 32 sources: K1 370 -> 349 us, K2 473 -> 463; 12^3x24 (3
// half-sites of a W = 4 tile used): K1 42.8 -> 35.0, K2 56.6 -> 48.6.  With the
// directions added outside the tensor cores (24 additions a lane for 8): K1 357, K2
// 484, K3 353, K4 621 at 24^3x48 x 32, 34.7 / 50.1 / 33.9 / 66.6 at 12^3x24 x 32.  Against
// the FP32 FMA stencil that these kernels replaced (1727 thread instructions per
// source-site), 24^3x48, 32 sources: K1 575, K2 690, K3 574, K4 849 -> 614 (5.9
// TB/s); with one group of 8: K1 152 -> 139, K2 199 -> 171, K4 233 -> 194.  A group
// costs the same however few of its 8 rows are used (4 sources: K1 83 -> 139 us),
// but a source's bits must not depend on its batch: the lattice alone decides which
// solves run here (f16_grouped_solve, f16_grouped_loops), and the loop estimators
// fill whole groups.  Tried on the way: neighbours loaded
// from L2 by each warp one item ahead (K1 560 us, latency-bound at 39 % issue),
// bulk copies of rows issued by one warp (676 us, the copy warp set the pace) and
// by four (375 us), all boxes issued by one thread (485 us), W = 6 with two copy
// warps (356).
//
// K1-K4 of the FP16 tier: persistent blocks, block b takes the tiles b, b +
// gridDim.y, ... and walks the live groups of 8 sources of each with the site's
// B words in registers.  Sites, order and reductions do not depend on the
// sources that share a launch, so a source's iterates are the same bits in any
// batch.
//   MODE MMA_HOP*:   out = ts q, q = to_ah H in + to_tc_ac center; <q, q> with NORM
//   MODE MMA_UPDATE: v = A(-mu) w - kappa^2 H in, r -= alpha v, x += alpha p; <r, r>
template <int DAG, int MODE, int W>
__global__ void __launch_bounds__(MmaShape<W>::NT, 1) mma_hop_kernel(const MmaHopArgs a, const __grid_constant__ MmaMaps maps) {
  constexpr bool NORM = MODE == MMA_HOP_CENTER_NORM || MODE == MMA_UPDATE;
  constexpr bool CENTER = MODE != MMA_HOP;
  constexpr bool UPD = MODE == MMA_UPDATE;
  using SH = MmaShape<W>;
  using ST = MmaStage<MODE, SH>;
  extern __shared__ __align__(128) uint4 mma_ring[];
  __shared__ __align__(8) uint64_t s_full[ST::COUNT], s_empty[ST::COUNT];
  __shared__ unsigned long long s_mask;
  __shared__ int s_grp[MMA_GROUPS], s_timeout, s_issued;
  __shared__ size_t s_goff[MMA_GROUPS];   // chunk offset of each live group
  __shared__ float s_alpha[UPD ? MMA_GROUPS * 8 : 1];
  __shared__ float s_part[NORM ? SH::WARPS : 1][MMA_GROUPS][32];
  __shared__ double s_sum[NORM ? SH::WARPS : 1][MMA_GROUPS][8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = lane & 3, row = lane >> 2;
  const int qc = q < 3 ? q : 2;
  if (threadIdx.x == 0) {
    s_mask = 0ull;
    s_timeout = 0;
    s_issued = 0;
#pragma unroll
    for (int i = 0; i < ST::COUNT; ++i) {
      mbar_init(&s_full[i], 1);
      mbar_init(&s_empty[i], SH::WARPS);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if constexpr (NORM) {
    if (warp < SH::WARPS)
      for (int j = 0; j < MMA_GROUPS; ++j) {
        s_part[warp][j][lane] = 0.f;
        if (lane < 8) s_sum[warp][j][lane] = 0.0;
      }
  }
  pdl_wait();
  __syncthreads();
  // the launch's live sources as a bit mask over the batch
  if (threadIdx.x < a.nrhs) {
    const int src = a.active != nullptr ? a.active[threadIdx.x] : (int)threadIdx.x;
    if (a.skip == nullptr || !a.skip[src].done) atomicOr(&s_mask, 1ull << src);
    if constexpr (UPD) s_alpha[src] = a.st[src].alpha_f;
  }
  __syncthreads();
  const unsigned long long mask = s_mask;
  if (mask == 0ull) return;   // every source is idle (the same in all blocks)
  int ng = 0;
#pragma unroll
  for (int g = 0; g < MMA_GROUPS; ++g)
    if ((mask >> (8 * g)) & 0xffull) {
      if (threadIdx.x == 0) {
        s_grp[ng] = g;
        s_goff[ng] = (size_t)g * (size_t)a.Vh * MMA_CHUNKS;
      }
      ++ng;
    }
  __syncthreads();
  const int ntile = a.tl.ntiles;
  if (warp >= SH::WARPS) {
    // ---- copy warps: one thread of each issues every fourth box of a stage (a
    // box costs its thread about 150 cycles; one thread alone set the pace)
    const int copier = warp - SH::WARPS;
    if (lane == 0) {
      const MmaTiles& g = a.tl;
      MmaTile tl(g, blockIdx.y);
      int stage = 0, round = 0, issued = 0;
      bool go = !a.withhold;
      for (int tile = blockIdx.y; tile < ntile && go; tile += gridDim.y, tl.next(g)) {
        const int x0 = tl.tx * g.W, w = min(g.W, g.Lxh - x0), y0 = 2 * tl.yp, z0 = 2 * tl.zp, t = tl.t;
        const int ym = y0 == 0 ? g.Ly - 1 : y0 - 1, yp = y0 + 2 == g.Ly ? 0 : y0 + 2;
        const int zm = z0 == 0 ? g.Lz - 1 : z0 - 1, zp = z0 + 2 == g.Lz ? 0 : z0 + 2;
        const int tm = t == 0 ? g.T - 1 : t - 1, tp = t + 1 == g.T ? 0 : t + 1;
        const bool left = x0 == 0, right = x0 + w == g.Lxh;
        for (int j = 0; j < ng && go; ++j) {
          if (round > 0 && mma_wait_failed(&s_empty[stage], (uint32_t)((round - 1) & 1), 0))
            *reinterpret_cast<volatile int*>(&s_timeout) = 1;
          go = *reinterpret_cast<volatile int*>(&s_timeout) == 0;
          if (!go) break;
          uint64_t* bar = &s_full[stage];
          const uint32_t dst = smem_u32(mma_ring) + (uint32_t)(stage * ST::BYTES);
          const int tg = g.T * s_grp[j];
          // rows whose output sites start even (s = 0) wrap on the left, the others on the right
          const int wraps = (left ? 2 : 0) + (right ? 2 : 0);
          if (copier == 0)
            mbar_expect_tx(bar, (uint32_t)((SH::F - 4 + wraps + 4 * W * ST::FIELDS) * MMA_CHUNKS * 16));
          auto at = [&](int slot) { return dst + (uint32_t)(slot * MMA_CHUNKS * 16); };
          if (copier == 0) {
            tma_load_5d(at(0), &maps.in[MMA_BOX_OWN], x0 - 1, y0, z0, tg + t, bar);
            tma_load_5d(at(SH::Y), &maps.in[MMA_BOX_Y], x0, ym, z0, tg + t, bar);
          } else if (copier == 1) {
            tma_load_5d(at(SH::Y + 2 * W), &maps.in[MMA_BOX_Y], x0, yp, z0, tg + t, bar);
            tma_load_5d(at(SH::Z), &maps.in[MMA_BOX_Z], x0, y0, zm, tg + t, bar);
          } else if (copier == 2) {
            tma_load_5d(at(SH::Z + 2 * W), &maps.in[MMA_BOX_Z], x0, y0, zp, tg + t, bar);
            tma_load_5d(at(SH::T), &maps.in[MMA_BOX_TILE], x0, y0, z0, tg + tm, bar);
          } else {
            tma_load_5d(at(SH::T + 4 * W), &maps.in[MMA_BOX_TILE], x0, y0, z0, tg + tp, bar);
            if (ST::FIELDS == 1) tma_load_5d(at(SH::F), &maps.f[0], x0, y0, z0, tg + t, bar);
          }
          if (ST::FIELDS == 4) tma_load_5d(at(SH::F + 4 * W * copier), &maps.f[copier], x0, y0, z0, tg + t, bar);
          if (wraps) {
            const int r = copier, s = (a.parity + r + (r >> 1) + t) & 1;
            if (s ? right : left) {
              const int rb = ((t * g.Lz + z0 + (r >> 1)) * g.Ly + y0 + (r & 1)) * g.Lxh;
              bulk_load(at(SH::WRAP + r), a.in + s_goff[j] + (size_t)(rb + (s ? 0 : g.Lxh - 1)) * MMA_CHUNKS,
                        MMA_CHUNKS * 16, bar);
            }
          }
          ++issued;
          if (++stage == ST::COUNT) {
            stage = 0;
            ++round;
          }
        }
      }
      atomicMax(&s_issued, issued);
    }
  } else {
    // ---- one site of the tile per warp
    const int r = warp / W, dx = warp % W, yy = r & 1, zz = r >> 1;
    // the site's link words, fetched one tile ahead
    uint32_t wr[8];
    uint32_t* link_words = reinterpret_cast<uint32_t*>(reinterpret_cast<unsigned char*>(mma_ring) + ST::BYTES * ST::COUNT) + warp * 96;
    const MmaLane L0(lane);
    auto site_of = [&](const MmaTile& tl) {
      return ((tl.t * a.tl.Lz + 2 * tl.zp + zz) * a.tl.Ly + 2 * tl.yp + yy) * a.tl.Lxh + tl.tx * a.tl.W + dx;
    };
    auto width = [&](const MmaTile& tl) { return min(a.tl.W, a.tl.Lxh - tl.tx * a.tl.W); };
    auto fetch_links = [&](int site) {
      const uint32_t* u = a.links + (size_t)site * 96;
      if constexpr (SH::LINKS_SMEM) {
        if (lane < 24)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(link_words + 4 * lane)),
                       "l"(u + 4 * lane)
                       : "memory");
      } else {
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
          wr[2 * mu] = __ldg(u + L0.wf + 24 * mu);
          wr[2 * mu + 1] = __ldg(u + L0.wb + 24 * mu + 12);
        }
      }
    };
    MmaTile tl(a.tl, blockIdx.y);
    int site = site_of(tl);
    bool valid = dx < width(tl);
    if (valid) fetch_links(site);
    int stage = 0, phase = 0, flush = 0;
    bool dead = false;        // a wait of this warp ran out: wait no more
    uint32_t live = 0;        // bit j: this lane stores its source of group j
    for (int j = 0; j < ng; ++j)
      if (q < 3 && ((mask >> (8 * s_grp[j] + row)) & 1ull)) live |= 1u << j;
    const uint4* lane_chunk = mma_ring + (row * 3 + qc);
    // chunk offsets in a stage that do not depend on the tile
    MmaSlots sl;
    {
      const int iy = ((r ^ 1) * (W + 2) + dx + 1) * MMA_CHUNKS, iz = ((r ^ 2) * (W + 2) + dx + 1) * MMA_CHUNKS;   // inside the tile
      const int ey = (SH::Y + (2 * yy + zz) * W + dx) * MMA_CHUNKS, ez = (SH::Z + (2 * zz + yy) * W + dx) * MMA_CHUNKS;
      sl.yf = yy ? ey : iy;
      sl.yb = yy ? iy : ey;
      sl.zf = zz ? ez : iz;
      sl.zb = zz ? iz : ez;
      sl.t = (SH::T + r * W + dx) * MMA_CHUNKS;
    }
    const int own = (r * (W + 2) + dx) * MMA_CHUNKS, wrap = (SH::WRAP + r) * MMA_CHUNKS;
    for (int tile = blockIdx.y; tile < ntile; tile += gridDim.y) {
      const bool more = tile + (int)gridDim.y < ntile;
      const int s = (a.parity + yy + zz + tl.t) & 1;
      uint32_t B[4][2], BL[4][2];
      auto make = [&](const MmaLane& L) {
        make_b<DAG, 0>(L, wr[0], wr[1], B[0], BL[0]);
        make_b<DAG, 1>(L, wr[2], wr[3], B[1], BL[1]);
        make_b<DAG, 2>(L, wr[4], wr[5], B[2], BL[2]);
        make_b<DAG, 3>(L, wr[6], wr[7], B[3], BL[3]);
      };
      if constexpr (SH::LINKS_SMEM) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        int ln = lane;
        asm volatile("" : "+r"(ln));   // the lane constants are formed again: registers are short
        const MmaLane L(ln);
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
          wr[2 * mu] = link_words[L.wf + 24 * mu];
          wr[2 * mu + 1] = link_words[L.wb + 24 * mu + 12];
        }
        make(L);
        __syncwarp();   // the words are read
      } else {
        make(L0);
      }
      const int xh = tl.tx * a.tl.W + dx;
      sl.xf = s && xh + 1 == a.tl.Lxh ? wrap : own + (1 + s) * MMA_CHUNKS;
      sl.xb = !s && xh == 0 ? wrap : own + s * MMA_CHUNKS;
      const size_t lane_site = (size_t)site * MMA_CHUNKS + row * 3 + qc;
      const bool active = valid;
      tl.next(a.tl);
      site = site_of(tl);
      valid = dx < width(tl);
      if (more && valid) fetch_links(site);
      for (int j = 0; j < ng; ++j) {
        if (!dead && mma_wait_failed(&s_full[stage], (uint32_t)phase, a.withhold)) {
          dead = true;
          *reinterpret_cast<volatile int*>(&s_timeout) = 1;
        }
        const uint4* nb = lane_chunk + stage * (ST::SLOTS * MMA_CHUNKS);
        uint64_t* empty = &s_empty[stage];
        if (++stage == ST::COUNT) {
          stage = 0;
          phase ^= 1;
        }
        float acc[8];
        uint4 cw, pw, rw, xw;
        if (active) {
          mma_site<DAG, W>(nb, sl, B, BL, acc);
          const uint4* f = nb + (SH::F + r * W + dx) * MMA_CHUNKS;
          if constexpr (CENTER) cw = f[0];
          if constexpr (UPD) {
            pw = f[4 * W * MMA_CHUNKS];
            rw = f[8 * W * MMA_CHUNKS];
            xw = f[12 * W * MMA_CHUNKS];
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty);   // the stage is read
        if (!active) continue;
        const bool store = (live >> j) & 1u;
        const size_t at = s_goff[j] + lane_site;
        float part = 0.f;
        if constexpr (UPD) {
          float v[8], y[8];
          unpack4(cw, v);
          twist4(a.fto_tc_ac, v);
#pragma unroll
          for (int e = 0; e < 8; ++e) acc[e] = v[e] - a.kappa2 * acc[e];
          const float alpha = s_alpha[8 * s_grp[j] + row];
          unpack4(rw, v);
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            v[e] = v[e] - alpha * acc[e];
            part += v[e] * v[e];
          }
          unpack4(xw, y);
          unpack4(pw, acc);
#pragma unroll
          for (int e = 0; e < 8; ++e) y[e] = y[e] + alpha * acc[e];
          if (store) {
            a.r[at] = pack4(v);
            a.x[at] = pack4(y);
          }
        } else {
          twist4(a.fto_ah, acc);
          if constexpr (CENTER) {
            float v[8];
            unpack4(cw, v);
            twist4(a.fto_tc_ac, v);
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e] = acc[e] + v[e];
          }
          if constexpr (NORM) {
#pragma unroll
            for (int e = 0; e < 8; ++e) part += acc[e] * acc[e];
            twist4(a.fts, acc);
          }
          if (store) a.out[at] = pack4(acc);
        }
        if constexpr (NORM) s_part[warp][j][lane] += store ? part : 0.f;
      }
      if constexpr (NORM) {
        if (++flush == MMA_FLUSH || !more) {
          flush = 0;
          for (int j = 0; j < ng; ++j) {
            float v = s_part[warp][j][lane];
            s_part[warp][j][lane] = 0.f;
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            v += __shfl_xor_sync(0xffffffffu, v, 2);
            if (q == 0) s_sum[warp][s_grp[j]][row] += (double)v;
          }
        }
      }
    }
  }
  __syncthreads();
  if (s_timeout) {   // let the copies in flight land, then report
    if (threadIdx.x == 0) {
      const int n = s_issued;
      for (int it = max(0, n - ST::COUNT); it < n; ++it)
        mbar_wait(&s_full[it % ST::COUNT], (uint32_t)((it / ST::COUNT) & 1), MMA_SPIN_LIMIT);
      *reinterpret_cast<volatile int*>(a.err) = 1;
    }
    __syncthreads();
  }
  pdl_trigger();
  if constexpr (NORM) {
    __shared__ bool s_last;
    if (threadIdx.x < 64 && ((mask >> threadIdx.x) & 1ull)) {
      double s = 0.0;
#pragma unroll
      for (int w = 0; w < SH::WARPS; ++w) s += s_sum[w][threadIdx.x >> 3][threadIdx.x & 7];
      a.red.partials[(size_t)threadIdx.x * a.red.stride + blockIdx.y] = s;
      __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(a.red.counter, 1u) == gridDim.y - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // eight threads per source add its blocks' partials in a fixed order
    const int src = threadIdx.x >> 3, l8 = threadIdx.x & 7;
    const bool on = src < 64 && ((mask >> (src & 63)) & 1ull);
    double s = on ? strided_sum_ordered(a.red.partials + (size_t)src * a.red.stride, l8, (int)gridDim.y, 8) : 0.0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o, 8);
    if (on && l8 == 0 && a.st != nullptr) post_action(a.st + src, a.post, s);
    if (threadIdx.x == 0) a.red.counter[0] = 0u;
  }
}

// K5 of the FP16 tier, p = r + beta p: one warp pass = one site of 8 sources
// (24 chunks); memory-bound
static __global__ void __launch_bounds__(256) mma_p_kernel(const uint4* __restrict__ r, uint4* __restrict__ p, int Vh,
                                                           const int* active, int nrhs, const CGState* st) {
  pdl_wait();
  const int lane = threadIdx.x & 31, q = lane % 3, row = lane / 3;
  const int k = blockIdx.x * 8 + row;
  if (lane >= 24 || k >= nrhs) return;
  const int src = active != nullptr ? active[k] : k;
  if (st[src].done) return;
  const float beta = st[src].beta_f;
  const size_t off = (size_t)(src >> 3) * ((size_t)Vh * 24) + (src & 7) * 3 + q;
  const int w = blockIdx.y * 8 + (threadIdx.x >> 5), nw = gridDim.y * 8;
  for (int site = w; site < Vh; site += nw) {
    const size_t at = off + (size_t)site * 24;
    float rv[8], pv[8];
    unpack4(__ldg(r + at), rv);
    unpack4(p[at], pv);
#pragma unroll
    for (int e = 0; e < 8; ++e) pv[e] = rv[e] + beta * pv[e];
    p[at] = pack4(pv);
  }
}

}  // namespace tsm
