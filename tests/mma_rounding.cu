// One site's hop sum for 8 sources, as the tensor-core stencil forms it and, per
// source, as sums of separately formed products (FP32, row 2 of a link in FP32)
// and in FP64, on the same FP16 fields and link rows.  Built and called by
// test_gpu_mma_rounding.py.  Every kernel: one warp (tensor cores) or one thread
// (products) per site and source inside arrays of `ns` sites.
#include "mma_hop.cuh"

using namespace tsm;

constexpr int SLOTS = 24;                       // sites of a stage: neighbours 0 .. 7, t + 1 at 7 + 16
__device__ __forceinline__ int slot_of(int hop) { return hop == 6 ? 23 : hop == 7 ? 7 : hop; }

// rows 0, 1 of the links of every hop -> the stencil's words
__global__ void pack_rows(const uint32_t* rows, uint32_t* words, int n) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= n) return;
  cx<float> q[6], lo[3];
  uint32_t hi[3];
  for (int k = 0; k < 6; ++k) q[k] = Pack16<F16>::unpack(words[12 * l + k] = rows[6 * l + k]);
  third_row_pair(q, hi, lo);
  for (int k = 0; k < 3; ++k) {
    words[12 * l + 6 + k] = hi[k];
    words[12 * l + 9 + k] = Pack16<F16>::pack((l & 1 ? 1.f : F16G::LO_SCALE) * lo[k]);
  }
}

__global__ void tensor_cores(const uint4* nb, const uint32_t* words, float* out, int ns) {
  const int lane = threadIdx.x & 31, site = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (site >= ns) return;
  const int q = lane & 3, row = lane >> 2;
  const MmaLane L(lane);
  const uint32_t* u = words + (size_t)site * 96;
  uint32_t B[4][2], BL[4][2];
  make_b<0, 0>(L, u[L.wf], u[L.wb + 12], B[0], BL[0]);
  make_b<0, 1>(L, u[L.wf + 24], u[L.wb + 36], B[1], BL[1]);
  make_b<0, 2>(L, u[L.wf + 48], u[L.wb + 60], B[2], BL[2]);
  make_b<0, 3>(L, u[L.wf + 72], u[L.wb + 84], B[3], BL[3]);
  const MmaSlots sl{0, 1 * MMA_CHUNKS, 2 * MMA_CHUNKS, 3 * MMA_CHUNKS, 4 * MMA_CHUNKS, 5 * MMA_CHUNKS, 7 * MMA_CHUNKS};
  float acc[8];
  mma_site<0, 4>(nb + (size_t)site * SLOTS * MMA_CHUNKS + row * 3 + (q < 3 ? q : 2), sl, B, BL, acc);
  for (int e = 0; q < 3 && e < 8; ++e)
    out[((size_t)site * 8 + row) * 24 + (3 * (e >> 1) + q) * 2 + (e & 1)] = acc[e];
}

template <class R, int MU, bool FWD>
__device__ void one_hop(const uint4* n, const uint32_t* rows, int src, cx<R> acc[12]) {
  uint32_t v[12];
  cx<float> hf[6], rf[9];
  for (int c = 0; c < 3; ++c) {
    const uint4 u = n[slot_of(2 * MU + !FWD) * MMA_CHUNKS + src * 3 + c];
    v[c] = u.x;
    v[3 + c] = u.y;
    v[6 + c] = u.z;
    v[9 + c] = u.w;
  }
  project_f16<MU, FWD ? -1 : 1>(v, hf);
  for (int k = 0; k < 6; ++k) rf[k] = Pack16<F16>::unpack(rows[6 * (2 * MU + !FWD) + k]);
  cx<R> r[9], h[6], u[6];
  for (int k = 0; k < 6; ++k) {
    r[k] = {(R)rf[k].re, (R)rf[k].im};
    h[k] = {(R)hf[k].re, (R)hf[k].im};
  }
  third_row(r, r + 6);
  for (int s = 0; s < 2; ++s)
    for (int i = 0; i < 3; ++i) {
      const cx<R>*a = h + 3 * s, w[3] = {FWD ? r[3 * i] : cconj(r[i]), FWD ? r[3 * i + 1] : cconj(r[3 + i]),
                                        FWD ? r[3 * i + 2] : cconj(r[6 + i])};
      u[3 * s + i] = w[0] * a[0] + w[1] * a[1] + w[2] * a[2];
    }
  accumulate<MU, FWD ? -1 : 1, MU == 0 && FWD>(acc, u);
}

template <class R>
__global__ void products(const uint4* nb, const uint32_t* rows, R* out, int ns) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x, site = t >> 3, src = t & 7;
  if (site >= ns) return;
  const uint4* n = nb + (size_t)site * SLOTS * MMA_CHUNKS;
  const uint32_t* u = rows + (size_t)site * 48;
  cx<R> acc[12];
  one_hop<R, 0, true>(n, u, src, acc);
  one_hop<R, 0, false>(n, u, src, acc);
  one_hop<R, 1, true>(n, u, src, acc);
  one_hop<R, 1, false>(n, u, src, acc);
  one_hop<R, 2, true>(n, u, src, acc);
  one_hop<R, 2, false>(n, u, src, acc);
  one_hop<R, 3, true>(n, u, src, acc);
  one_hop<R, 3, false>(n, u, src, acc);
  for (int k = 0; k < 12; ++k) {
    out[((size_t)site * 8 + src) * 24 + 2 * k] = acc[k].re;
    out[((size_t)site * 8 + src) * 24 + 2 * k + 1] = acc[k].im;
  }
}

// device pointers: fields [ns][24][24] chunks, rows [ns][8][6] words, scratch [ns][8][12] words, outputs [ns][8][24]
extern "C" int mma_rounding(const void* fields, const void* rows, void* scratch, float* tc, float* f32, double* f64, int ns) {
  const uint4* nb = static_cast<const uint4*>(fields);
  const uint32_t* r = static_cast<const uint32_t*>(rows);
  uint32_t* w = static_cast<uint32_t*>(scratch);
  pack_rows<<<(ns * 8 + 127) / 128, 128>>>(r, w, ns * 8);
  tensor_cores<<<(ns + 3) / 4, 128>>>(nb, w, tc, ns);
  products<float><<<(ns * 8 + 127) / 128, 128>>>(nb, r, f32, ns);
  products<double><<<(ns * 8 + 127) / 128, 128>>>(nb, r, f64, ns);
  return (int)cudaDeviceSynchronize();
}
