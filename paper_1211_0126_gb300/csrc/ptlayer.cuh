// ptlayer.cuh -- a whole parallel-transport layer in one kernel: the transports
// are computed straight into the tensor-core operand, so that the gathered
// matrix Z (5 KB per site at 12 channels) never goes through memory.
#pragma once

#include "ptnet.cuh"
#include "umma.cuh"

namespace tsm {

constexpr int PT_MIN_BLOCKS = 120;           // fewest blocks of a lattice that the fused layer is taken for
constexpr int PT_SITES = 42;                 // sites of a CTA: 126 of the MMA's 128 rows (3 colours each)
constexpr int PT_CORE = 144;                 // bytes from a core matrix to the next in K: 128 + 16, so that the
                                             // stores of neighbouring channels fall into different banks
constexpr int PT_MAX_GROUPS = 12;            // column groups of 8 (path, channel pairs) of a stage at most

// (path, channel) groups per stage: an even number, so that a stage is whole
// K = 16 MMAs; the last stage is padded with zeros
inline int pt_groups(int cin) {
  const int j = PT_PATHS * cin;
  return j < PT_MAX_GROUPS ? (j + 1) & ~1 : PT_MAX_GROUPS;
}
template <int BN> inline int pt_layer_smem(int groups) { return 2 * (16 + BN / 8) * groups * PT_CORE + 1024; }
inline int pt_steps(int cin) { return (PT_PATHS * cin + pt_groups(cin) - 1) / pt_groups(cin); }
// column width of the tile that holds 8 cout columns (0: too wide for one)
inline int pt_tile(int cout) {
  const int n = 8 * cout;
  return n <= 16 ? 16 : n <= 64 ? 64 : n <= 96 ? 96 : n <= 128 ? 128 : n <= 192 ? 192 : n <= 256 ? 256 : 0;
}

// block weights B [N][8 J] -> stage after stage in the operand layout of
// pt_layer_kernel (zeros past N and J), so that a stage is one bulk copy
__global__ void __launch_bounds__(256) pt_pack_stages_kernel(const __nv_bfloat16* __restrict__ B, int N, int J, int BN,
                                                             int GJ, int steps, uint4* __restrict__ out) {
  const int rows9 = PT_CORE / 16;   // 8 rows and the pad of a core matrix
  const int idx = blockIdx.x * 256 + threadIdx.x;
  if (idx >= steps * (BN / 8) * GJ * rows9) return;
  const int r = idx % rows9, core = idx / rows9, gj = core % GJ, nk = core / GJ, n = (nk % (BN / 8)) * 8 + r;
  const int j = (nk / (BN / 8)) * GJ + gj;
  uint4 v = make_uint4(0u, 0u, 0u, 0u);
  if (r < 8 && n < N && j < J) v = *reinterpret_cast<const uint4*>(B + (size_t)n * 8 * J + 8 * j);
  out[idx] = v;
}

// Y = Z B^T of one layer, Z (BF16) formed on the fly.  CTA = 42 sites of sample
// blockIdx.y, 256 threads, two stages of shared memory (two CTAs per SM up to
// BN = 128).  Stage k holds column groups k GJ .. k GJ + GJ - 1 of Z and of B in
// the no-swizzle core-matrix layout.  A thread owns one site and two
// groups of every stage, half a stage apart: it loads the neighbour's channels
// (a site's threads read consecutive 16-byte pieces; the neighbours of the block's sites are found
// once), rebuilds the link once for both, transports in FP32 and stores three
// 16-byte core-matrix rows per group; a stage of B is one bulk copy of weights
// packed in its layout.  One thread issues the stage's MMAs, which run while the
// next stage is computed.  Every wait is bounded; a thread whose wait ran out
// says so at the stage's barrier, where all leave the loop together, the MMAs and
// copies in flight are waited for (bounded), TMEM is freed and the error is
// recorded.  withhold: fault injection as in umma.cuh (no weight copies).
// 12 -> 12 channels at 16^3x32: 340 us against 310 (gather, 680 MB of Z written)
// + 170 (GEMM); 12 -> 1: 267 against 310 + 108.  Bound by the latency of the
// neighbour loads (16 warps of 128 registers per SM, 40 % issue; the ring leaves
// 30 KB of L1).
template <int BN>
__global__ void __launch_bounds__(256, BN <= 128 ? 2 : 1)
    pt_layer_kernel(NetGeom ng, const float* __restrict__ X, int C, const uint8_t* __restrict__ B, int N,
                    float* __restrict__ Y, int GJ, int steps, int* __restrict__ error, int withhold) {
  constexpr int TMEM_COLS = BN <= 32 ? 32 : (BN <= 64 ? 64 : (BN <= 128 ? 128 : 256));
  extern __shared__ uint8_t pt_dyn[];
  __shared__ __align__(8) uint64_t bar[2], wbar[2];   // a stage's MMAs, its weights
  __shared__ uint32_t tmem_slot;
  __shared__ int s_nbr[PT_SITES][8];   // neighbour of path p = 1 .. 8, its complement if the hop changes sign
  const uint32_t ring = (smem_u32(pt_dyn) + 127u) & ~127u;
  const uint32_t a_bytes = 16u * GJ * PT_CORE, stage_bytes = a_bytes + (uint32_t)(BN / 8) * GJ * PT_CORE;
  const uint32_t group_rows = (uint32_t)GJ * PT_CORE;   // bytes from 8 rows to the next 8
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const Geom& g = ng.g;
  if (tid == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_init(&wbar[0], 1);
    mbar_init(&wbar[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  // rows of Z that no site fills stay zero (each thread's proxy fence in the loop
  // orders these stores before the MMAs).  The weight parts are left to the bulk
  // copies, which write every byte of them: nothing orders a generic store here
  // before a copy of the async proxy to the same bytes
  for (uint32_t o = tid * 16; o < 2 * a_bytes; o += 256 * 16)
    asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(ring + o + (o < a_bytes ? 0u : stage_bytes - a_bytes)),
                 "r"(0u)
                 : "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  constexpr uint32_t idesc = umma_idesc_bf16(UMMA_BM, BN);
  const int J = PT_PATHS * C;
  const uint32_t b_bytes = (uint32_t)(BN / 8) * GJ * PT_CORE;
  const uint32_t inv_c = 0xffffu / (uint32_t)C + 1u;   // j / C = j inv_c >> 16 for j < 1024, C <= 64
  X += (size_t)blockIdx.y * 3 * g.V * 8 * C;
  Y += (size_t)blockIdx.y * 3 * g.V * N;
  const int pairs = GJ >> 1;
  const int site = tid / pairs, cg = tid - site * pairs;
  const int x = blockIdx.x * PT_SITES + site;
  const bool mine = site < PT_SITES && x < g.V;
  int parity = 0;
  if (mine) {
    int c[4];
    lex_coords(g, x, c);
    parity = (c[0] + c[1] + c[2] + c[3]) & 1;
    for (int p = 1 + cg; p <= 8; p += pairs) {
      const PathHop h = path_hop(g, c[0], c[1], c[2], c[3], p);
      s_nbr[site][p - 1] = h.sign < 0.f ? ~h.src : h.src;
    }
  }
  __syncthreads();
  const long long limit = withhold ? UMMA_INJECT_LIMIT : MBAR_SPIN_LIMIT;
  bool failed = false;   // a wait of this thread ran out; all threads learn of it at the stage's barrier
  int wcopies = 0;       // thread 0: weight copies issued
  int k = 0;             // stages whose MMAs were issued
  for (; k < steps; ++k) {
    const int s = k & 1;
    const uint32_t sa = ring + s * stage_bytes, sb = sa + a_bytes;
    // the stage's previous MMAs are done
    if (k >= 2) failed = !mbar_wait(&bar[s], (uint32_t)((k / 2 - 1) & 1), limit);
    if (tid == 0 && !failed && !withhold) {
      mbar_expect_tx(&wbar[s], b_bytes);
      bulk_load(sb, B + (size_t)k * b_bytes, b_bytes, &wbar[s]);
      wcopies = k + 1;
    }
    if (mine) {
      int path = -1, src = x;
      bool fwd = true;
      cx<float> u[9];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int gj = cg + i * pairs, j = k * GJ + gj;
        cx<float> out[4][3];
        if (j < J) {
          const int p = (int)(((uint32_t)j * inv_c) >> 16), ch = j - p * C;
          if (p == 0) {
            load_channel(X, C, x, ch, out);
          } else {
            if (p != path) {
              path = p;
              const int n = s_nbr[site][p - 1];
              src = n < 0 ? ~n : n;
              const int mu = (p - 1) >> 1;
              fwd = (p & 1) != 0;
              net_link_at(ng, fwd ? x : src, fwd ? parity : 1 - parity, mu, u);
              if (n < 0) {
#pragma unroll
                for (int e = 0; e < 9; ++e) u[e] = {-u[e].re, -u[e].im};
              }
            }
            cx<float> v[4][3];
            load_channel(X, C, src, ch, v);
            if (fwd) {
#pragma unroll
              for (int s2 = 0; s2 < 4; ++s2)
#pragma unroll
                for (int a = 0; a < 3; ++a)
                  out[s2][a] = cdot3(u[3 * a], v[s2][0], u[3 * a + 1], v[s2][1], u[3 * a + 2], v[s2][2]);
            } else {
#pragma unroll
              for (int s2 = 0; s2 < 4; ++s2)
#pragma unroll
                for (int a = 0; a < 3; ++a)
                  out[s2][a] = cjdot3(u[a], v[s2][0], u[3 + a], v[s2][1], u[6 + a], v[s2][2]);
            }
          }
        } else {
#pragma unroll
          for (int s2 = 0; s2 < 4; ++s2)
#pragma unroll
            for (int a = 0; a < 3; ++a) out[s2][a] = {0.f, 0.f};
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const int row = 3 * site + a;
          __nv_bfloat162 q[4] = {__floats2bfloat162_rn(out[0][a].re, out[1][a].re),
                                 __floats2bfloat162_rn(out[2][a].re, out[3][a].re),
                                 __floats2bfloat162_rn(out[0][a].im, out[1][a].im),
                                 __floats2bfloat162_rn(out[2][a].im, out[3][a].im)};
          const uint32_t* q32 = reinterpret_cast<const uint32_t*>(q);
          asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(sa + (row >> 3) * group_rows + gj * PT_CORE +
                                                                        (row & 7) * 16),
                       "r"(q32[0]), "r"(q32[1]), "r"(q32[2]), "r"(q32[3])
                       : "memory");
        }
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic stores -> tensor core
    if (tid == 0 && !failed) failed = !mbar_wait(&wbar[s], (uint32_t)((k / 2) & 1), limit);
    if (__syncthreads_or(failed)) break;   // the same iteration for every thread
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      for (int kk = 0; kk < pairs; ++kk) {
        const uint64_t da = umma_desc(sa + kk * 2 * PT_CORE, PT_CORE, group_rows);
        const uint64_t db = umma_desc(sb + kk * 2 * PT_CORE, PT_CORE, group_rows);
        const uint32_t acc = (k > 0 || kk > 0) ? 1u : 0u;
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
            "l"(da), "l"(db), "r"(idesc), "r"(acc));
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                       smem_u32(&bar[s]))
                   : "memory");
    }
  }
  // the last commit covers every earlier MMA (after a timeout: of the stages issued)
  failed = k < steps;
  if (k > 0 && !mbar_wait(&bar[(k - 1) & 1], (uint32_t)(((k - 1) / 2) & 1))) failed = true;
  const bool timed_out = __syncthreads_or(failed);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (!timed_out) {
    // warp w: accumulator lanes (rows) 32 (w % 4) .., columns of half w / 4
    const int row = (warp & 3) * 32 + lane;
    const long long grow = (long long)blockIdx.x * 3 * PT_SITES + row;
    const bool store = row < 3 * PT_SITES && grow < 3ll * g.V;
    for (int c0 = (warp >> 2) * (BN / 2); c0 < ((warp >> 2) + 1) * (BN / 2) && c0 < N; c0 += 8) {
      uint32_t v[8];
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
          : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
          : "r"(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      if (store) {
        float4* dst = reinterpret_cast<float4*>(Y + (size_t)grow * N + c0);
        dst[0] = make_float4(__uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2]), __uint_as_float(v[3]));
        dst[1] = make_float4(__uint_as_float(v[4]), __uint_as_float(v[5]), __uint_as_float(v[6]), __uint_as_float(v[7]));
      }
    }
  } else {
    // the MMAs in flight were waited for above, now the copies, before the memory is released
    if (tid == 0) {
      for (int c = max(0, wcopies - 2); c < wcopies; ++c) mbar_wait(&wbar[c & 1], (uint32_t)((c / 2) & 1));
      if (error != nullptr) atomicExch(error, 1);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
  }
}

}  // namespace tsm
