// ops_f16g.cu -- launch helpers of the grouped FP16 storage (F16G): the
// tensor-core stencil and CG update, and the site-local kernels around them.
#include <algorithm>

#include "context.h"
#include "fields.cuh"
#include "mma_hop.cuh"
#include "tma_map.h"

namespace tsm {

namespace {

inline int blocks_for(int n, int nt) { return (n + nt - 1) / nt; }
inline int groups_of(int nrhs) { return (nrhs + 7) / 8; }

// tiles of the lattice and the persistent grid: one block per SM, never more
// than there are tiles or partial slots (the grid fixes the reduction order, so
// it depends on the lattice and the device alone)
MmaHopArgs mma_args(const Ctx& c, int p_out, int w, dim3* grid) {
  MmaHopArgs m{};
  MmaTiles& t = m.tl;
  t.Lxh = c.g.Lxh;
  t.Ly = c.g.L[1];
  t.Lz = c.g.L[2];
  t.T = c.g.L[3];
  t.ntx = blocks_for(t.Lxh, w);
  t.W = blocks_for(t.Lxh, t.ntx);
  t.nyp = t.Ly / 2;
  t.nzp = t.Lz / 2;
  t.ntiles = t.ntx * t.nyp * t.nzp * t.T;
  const int gy = std::min(std::min(t.ntiles, c.sm_count), (int)c.red_cap);
  int n = gy;
  t.gx = n % t.ntx;
  n /= t.ntx;
  t.gy = n % t.nyp;
  n /= t.nyp;
  t.gz = n % t.nzp;
  t.gt = n / t.nzp;
  *grid = dim3(1, gy);
  m.Vh = c.g.Vh;
  m.parity = p_out;
  m.links = c.links_of<F16G>(p_out);
  m.err = c.h_err;
  m.withhold = copies_withheld();
  return m;
}

// tensor map of a grouped field: [T * groups][Lz][Ly][Lxh] sites of 384 bytes
// (48 elements of 8), read in boxes of whole sites, zeros outside
int make_map(const Ctx& c, CUtensorMap* m, const void* base, int kind, int w) {
  int box[3];
  mma_box(kind, w, box);
  PFN_cuTensorMapEncodeTiled_v12000 fn = tensor_map_encoder();
  const cuuint64_t dims[5] = {48, (cuuint64_t)c.g.Lxh, (cuuint64_t)c.g.L[1], (cuuint64_t)c.g.L[2],
                              (cuuint64_t)c.g.L[3] * MMA_GROUPS};
  cuuint64_t strides[4];
  strides[0] = MMA_CHUNKS * 16;
  for (int k = 1; k < 4; ++k) strides[k] = strides[k - 1] * dims[k];
  const cuuint32_t b[5] = {48, (cuuint32_t)box[0], (cuuint32_t)box[1], (cuuint32_t)box[2], 1};
  const cuuint32_t es[5] = {1, 1, 1, 1, 1};
  if (fn == nullptr ||
      fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 5, const_cast<void*>(base), dims, strides, b, es,
         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
    set_error("tensor map of a grouped FP16 field could not be encoded");
    return TSM_ERR_CUDA;
  }
  return TSM_OK;
}

int in_maps(const Ctx& c, MmaMaps* m, const void* in, int w) {
  for (int k = 0; k < MMA_BOXES; ++k) TSM_TRY(make_map(c, &m->in[k], in, k, w));
  return TSM_OK;
}

template <int DAG, int MODE, int W>
int mma_launch(Ctx& c, const MmaHopArgs& m, const MmaMaps& maps, dim3 grid) {
  using SH = MmaShape<W>;
  constexpr int smem = MmaStage<MODE, SH>::SMEM;
  TSM_CUDA(cudaFuncSetAttribute(mma_hop_kernel<DAG, MODE, W>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  (void)launch_pdl(c, mma_hop_kernel<DAG, MODE, W>, grid, dim3(SH::NT), smem, m, maps);
  c.launches++;
  return check_launch(c, "mma_hop_kernel");
}

// width of the hops' tiles in half-sites: 6, with 24 warps, where its tiles cover a
// row with no more idle warps than those of 4 (Lx / 2 = 5, 6, 9 .. 12, ...), else 4,
// with 16 (24^3x48 K1 349 against 370 us, 12^3x24 35.0 against 42.8; Lx / 2 = 8 would
// leave a third of the warps idle).  The update (K4), bound by HBM, keeps 4: four
// fields of a stage of 6 leave two stages, and its epilogue needs the registers.
int mma_width(const Ctx& c) {
  return 6 * blocks_for(c.g.Lxh, 6) <= 4 * blocks_for(c.g.Lxh, 4) ? 6 : 4;
}

template <int DAG, int MODE>
int mma_hop(Ctx& c, const MmaHopArgs& m, const MmaMaps& maps, dim3 grid, int w) {
  return w == 6 ? mma_launch<DAG, MODE, 6>(c, m, maps, grid) : mma_launch<DAG, MODE, 4>(c, m, maps, grid);
}

}  // namespace

template <>
int launch_hop<F16G>(Ctx& c, const HopArgs<F16G>& a0, int dag, int mode, int prof_kind, int nrhs) {
  if (a0.g.Vh == 0 || nrhs == 0) return TSM_OK;
  HopArgs<F16G> a = a0;
  hop_factors(&a);
  if ((!(mode & HOP_NORM) && !a.one_ts) || a.skip_rel || a.base != nullptr) {
    set_error("grouped FP16 hop: epilogue not built (dag %d, mode %d)", dag, mode);
    return TSM_ERR_ARG;
  }
  dim3 grid;
  const int w = mma_width(c);
  MmaHopArgs m = mma_args(c, a.p_out, w, &grid);
  m.in = a.in;
  m.out = a.out;
  MmaMaps maps;
  TSM_TRY(in_maps(c, &maps, a.in, w));
  if (mode & HOP_CENTER) TSM_TRY(make_map(c, &maps.f[0], a.center, MMA_BOX_TILE, w));
  m.fto_ah = a.fto_ah;
  m.fto_tc_ac = a.fto_tc_ac;
  m.fts = a.fts;
  m.active = a.active;
  m.nrhs = nrhs;
  m.skip = a.skip;
  m.st = a.st;
  m.post = a.post;
  m.red = a.red;
  const int kind = prof_kind >= 0 ? prof_kind : (dag ? PK_HOP_DAG : (mode & HOP_CENTER) ? PK_HOP_XPAY : PK_HOP);
  const double sb = spinor_site_bytes(F16::id), lb = link_site_bytes(F16::id);
  TimedLaunch tl(c, 4 * F16::id + kind, (double)a.g.Vh * (lb + nrhs * sb * (2 + ((mode & HOP_CENTER) ? 1 : 0))));
  int rc;
  if (dag == 0 && mode == 0) rc = mma_hop<0, MMA_HOP>(c, m, maps, grid, w);
  else if (dag == 0 && mode == HOP_CENTER) rc = mma_hop<0, MMA_HOP_CENTER>(c, m, maps, grid, w);
  else if (dag == 0 && mode == (HOP_CENTER | HOP_NORM)) rc = mma_hop<0, MMA_HOP_CENTER_NORM>(c, m, maps, grid, w);
  else if (dag == 1 && mode == 0) rc = mma_hop<1, MMA_HOP>(c, m, maps, grid, w);
  else if (dag == 1 && mode == (HOP_CENTER | HOP_NORM)) rc = mma_hop<1, MMA_HOP_CENTER_NORM>(c, m, maps, grid, w);
  else {
    set_error("grouped FP16 hop variant dag=%d mode=%d not built", dag, mode);
    return TSM_ERR_ARG;
  }
  tl.done();
  return rc;
}

template <>
int launch_cg_update<F16G, F16G>(Ctx& c, const CGUpdArgs<F16G, F16G>& a, int nrhs) {
  if (a.g.Vh == 0 || nrhs == 0) return TSM_OK;
  dim3 grid;
  constexpr int w = 4;
  MmaHopArgs m = mma_args(c, 0, w, &grid);
  m.in = a.t;
  MmaMaps maps;
  TSM_TRY(in_maps(c, &maps, a.t, w));
  const void* fields[4] = {a.w, a.p, a.r, a.x};
  for (int k = 0; k < 4; ++k) TSM_TRY(make_map(c, &maps.f[k], fields[k], MMA_BOX_TILE, w));
  m.r = a.r;
  m.x = a.x;
  m.fto_tc_ac = to_float(a.tw);
  m.kappa2 = (float)a.kappa2;
  m.active = a.active;
  m.nrhs = nrhs;
  m.skip = a.st;
  m.st = a.st;
  m.post = POST_RR;
  m.red = a.red;
  const double sb = spinor_site_bytes(F16::id), lb = link_site_bytes(F16::id);
  TimedLaunch tl(c, 4 * F16::id + PK_HOP_UPDATE, (double)a.g.Vh * (lb + nrhs * 7 * sb));
  const int rc = mma_launch<1, MMA_UPDATE, w>(c, m, maps, grid);
  tl.done();
  return rc;
}

template <>
int launch_cg_p<F16G, F16G>(Ctx& c, const PField& r, const PField& p, CGState* st, const int* active, int nrhs) {
  if (c.g.Vh == 0 || nrhs == 0) return TSM_OK;
  const dim3 grid(groups_of(nrhs), std::min(blocks_for(c.g.Vh, 32), 8 * c.sm_count));
  (void)launch_pdl(c, mma_p_kernel, grid, dim3(256), 0, r.as<F16G>(), p.as<F16G>(), c.g.Vh, active, nrhs, st);
  c.launches++;
  return check_launch(c, "mma_p_kernel");
}

template <>
int launch_noise<F16G>(Ctx& c, int parity, const NoiseSpec& n, uint32_t source0, const PField& out, int nrhs) {
  if (nrhs == 0) return TSM_OK;
  noise_grouped_kernel<<<dim3(blocks_for(c.g.Vh, SITE_NT / 8), groups_of(nrhs)), SITE_NT, 0, c.stream>>>(
      c.g, parity, n, source0, out.as<F16G>(), c.sstride, nrhs);
  c.launches++;
  return check_launch(c, "noise_grouped_kernel");
}

template <>
int launch_twist<F16G>(Ctx& c, const Twist& f, const PField& in, const PField& out, const CGState*, const int*,
                       int nrhs) {
  if (nrhs == 0) return TSM_OK;
  twist_grouped_kernel<<<dim3(blocks_for(c.g.Vh, SITE_NT / 8), groups_of(nrhs)), SITE_NT, 0, c.stream>>>(
      c.g.Vh, to_float(f), in.as<F16G>(), out.as<F16G>(), c.sstride, nrhs);
  c.launches++;
  return check_launch(c, "twist_grouped_kernel");
}

// whole groups: a copy, or zeros when in has no memory
template <>
int launch_convert<F16G, F16G>(Ctx& c, const PField& in, const PField& out, const int*, int nrhs) {
  if (nrhs == 0) return TSM_OK;
  const size_t bytes = field_bytes(F16G::id, c.sstride) * (size_t)(8 * groups_of(nrhs));
  if (in.p == nullptr) TSM_CUDA(cudaMemsetAsync(out.p, 0, bytes, c.stream));
  else TSM_CUDA(cudaMemcpyAsync(out.p, in.p, bytes, cudaMemcpyDeviceToDevice, c.stream));
  return TSM_OK;
}

template <class Si, class So>
static int convert_grouped(Ctx& c, const PField& in, const PField& out, int nrhs) {
  if (nrhs == 0) return TSM_OK;
  convert_grouped_kernel<Si, So><<<dim3(blocks_for(c.g.Vh, SITE_NT / 8), groups_of(nrhs)), SITE_NT, 0, c.stream>>>(
      c.g.Vh, in.as<Si>(), out.as<So>(), c.sstride, nrhs);
  c.launches++;
  return check_launch(c, "convert_grouped_kernel");
}
template <>
int launch_convert<F32, F16G>(Ctx& c, const PField& in, const PField& out, const int*, int nrhs) {
  return convert_grouped<F32, F16G>(c, in, out, nrhs);
}
template <>
int launch_convert<F16G, F32>(Ctx& c, const PField& in, const PField& out, const int*, int nrhs) {
  return convert_grouped<F16G, F32>(c, in, out, nrhs);
}
template <>
int launch_convert<F16G, F64>(Ctx& c, const PField& in, const PField& out, const int*, int nrhs) {
  return convert_grouped<F16G, F64>(c, in, out, nrhs);
}
template <>
int launch_convert<F16G, F16>(Ctx& c, const PField& in, const PField& out, const int*, int nrhs) {
  return convert_grouped<F16G, F16>(c, in, out, nrhs);
}

}  // namespace tsm
