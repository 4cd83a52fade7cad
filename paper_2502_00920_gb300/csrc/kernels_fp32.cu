// FP32 storage and arithmetic, u as a float pair: kernel instantiations and launchers of liblbs.
#include <string.h>

#include "lbs_device.cuh"
#include "lbs_batch.cuh"
#include "lbs_column.cuh"
#include "lbs_resident.cuh"

namespace lbs {
namespace {
using P = F32;
// tile variants (nodes along x, nodes along y, thread rows)
using V0 = Cfg<P, 32, 16, 8>;
using V1 = Cfg<P, 32, 8, 8>;
using V2 = Cfg<P, 64, 8, 4>;
using V3 = Cfg<P, 32, 24, 8>;
using V4 = Cfg<P, 32, 16, 8>;
using M6 = MarchCfg<V4, 8, 128, 2>;
using V8 = Cfg<P, 32, 32, 8>;
using V9 = Cfg<P, 32, 16, 16>;  // one node per thread, 512 threads
// 0-3: V0-V3 tiles read from global memory; 4: V4 tiles staged by TMA;
// 5: V4 tiles, persistent blocks with a two-stage TMA ring; 6: row-marching
// strips over the V4 tile columns; 7: V3 tiles staged by TMA; 8: V8 tiles
// (four nodes per thread) read from global memory; 9: two fused iterations per
// launch on V9 tiles (periodic lattices; one V0 iteration per call otherwise);
// 10: two iterations per launch in warp columns (periodic lattices of even
// width; variant 4 otherwise).
constexpr int kVariants = 11;
// periodic lattices from this many nodes on take variant 10: below, too few
// strips march to fill the GPU (us per iteration, variant 4 / 10: 512^2 12.9 /
// 23.1, 1024^2 26.4 / 31.2, 1024 x 2048 45.3 / 44.0, 1536^2 48.9 / 48.4, 2048^2
// 77.2 / 72.5, 400 x 6000 57.5 / 47.5, 4096^2 275 / 233, 16384^2 4204 / 3269)
constexpr int64_t kColumnNodes = 1 << 21;
// lattices below this many nodes default to variant 0 (see default_variant)
constexpr int64_t kSmallNodes = 400000;

TileShape shape(int v) {
  switch (v) {
    case 1: return {V1::TX, V1::TY};
    case 2: return {V2::TX, V2::TY};
    case 3:
    case 7: return {V3::TX, V3::TY};
    case 4:
    case 5:
    case 6: return {V4::TX, V4::TY};
    case 8: return {V8::TX, V8::TY};
    case 9: return {V9::TX, V9::TY};
    case 10: return {64, 64};
    default: return {V0::TX, V0::TY};
  }
}

const char *name(int v) {
  switch (v) {
    case 4: return "step_tma_kernel";
    case 5: return "step_tma2_kernel";
    case 6: return "step_march_kernel";
    case 7: return "step_tma_kernel";
    case 9: return "step_fused2_tma_kernel";
    case 10: return "step_column_kernel";
    default: return "step_interior_kernel";
  }
}

// one iteration on V4 tiles (variant 10 outside its lattices)
cudaError_t step_single(const Params &p, const StepPtrs &s, cudaStream_t st) {
  return s.tm_g ? launch_step_tma<V4>(p, s, st) : launch_step<V0>(p, s, st);
}

cudaError_t step(const Params &p, const StepPtrs &s, int v, cudaStream_t st) {
  switch (v) {
    case 1: return launch_step<V1>(p, s, st);
    case 2: return launch_step<V2>(p, s, st);
    case 3: return launch_step<V3>(p, s, st);
    case 4: return launch_step_tma<V4>(p, s, st);
    case 5: return launch_step_tma2<V4>(p, s, st);
    case 6: return launch_step_march<V4, M6>(p, s, st);
    case 7: return launch_step_tma<V3>(p, s, st);
    case 8: return launch_step<V8>(p, s, st);
    case 9: return fused2_applies(p) ? launch_step_fused2<V9>(p, s, st) : launch_step<V0>(p, s, st);
    case 10: return column_wraps(p) ? launch_column_periodic<P, 2>(p, s, st) : step_single(p, s, st);
    default: return launch_step<V0>(p, s, st);
  }
}

int kernels_per_step(const Params &p, int v) {
  switch (v) {
    case 1: return step_kernel_count<V1>(p);
    case 2: return step_kernel_count<V2>(p);
    case 3:
    case 7: return step_kernel_count<V3>(p);
    case 4:
    case 5:
    case 6: return step_kernel_count<V4>(p);
    case 8: return step_kernel_count<V8>(p);
    case 10: return column_wraps(p) ? 1 : step_kernel_count<V4>(p);
    case 9: {
      if (!fused2_applies(p)) return step_kernel_count<V0>(p);
      const int ntx = (p.nx + V9::TX - 1) / V9::TX, nty = (p.ny + V9::TY - 1) / V9::TY;
      int a_lo, a_hi, b_lo, b_hi;
      interior_range_m(p.nx, p.ny, V9::TX, V9::TY, 6, a_lo, a_hi, b_lo, b_hi);
      const int ni = (a_hi - a_lo) * (b_hi - b_lo);
      return (ni > 0 ? 1 : 0) + (ntx * nty > ni ? 1 : 0);
    }
    default: return step_kernel_count<V0>(p);
  }
}

int iterations_per_call(const Params &p, int v) {
  return (v == 9 && fused2_applies(p)) || (v == 10 && column_wraps(p)) ? 2 : 1;
}

cudaError_t step1(const Params &p, const StepPtrs &s, int v, cudaStream_t st) {
  return v == 10 ? step_single(p, s, st) : launch_step<V0>(p, s, st);
}
int kernels_per_step1(const Params &p, int v) { return v == 10 ? step_kernel_count<V4>(p) : step_kernel_count<V0>(p); }

// Small lattices (a wave of tiles or less: every launch is one tile's latency)
// pull from global memory, where a tile starts without waiting for its boxes;
// us per iteration, one lattice alone / three side by side, variant 0 against 4:
// 300^2 walled 6.7 / 2.9 against 7.5 / 3.0, 512^2 7.7 / 5.7 against 13.2 / 5.6, 1021
// x 509 13.2 / 12.7 against 15.5 / 11.5, 1024^2 26.5 / 25.0 against 26.5 / 20.7.
int default_variant(const Params &p) {
  const int64_t nodes = (int64_t)p.nx * p.ny;
  return column_wraps(p) && nodes >= kColumnNodes ? 10 : (nodes < kSmallNodes ? 0 : 4);
}

bool tma_maps(const Params &p, int v, const void *g, const void *u, void *og, void *ou) {
  if (v == 9) return make_fused2_maps<V9>(p, g, u, og, ou);
  if (v == 6) return make_march_maps<V4, M6>(p, g, u, og, ou);
  if (v == 7) return make_tma_maps<V3>(p, g, u, og, ou);
  if (v != 4 && v != 5 && v != 10) return false;
  return make_tma_maps<V4>(p, g, u, og, ou);
}

void coef(const Params &p, void *out) {
  const auto k = make_coef<P::gs, P::real>(p);
  memcpy(out, &k, sizeof(k));
}

// resident launches (us per iteration on walled neo-Hooke lattices, one lattice
// alone / three advancing side by side; launching every iteration from a graph
// before them): 32 x 32 10.7 / 3.7 -> 2.2 / 0.75 and 128 x 128 10.4 / 3.6 ->
// 2.6 / 1.9 on 16 x 8 tiles, 160 x 160 10.5 / 3.8 -> 3.6 / 2.4 and 256 x 256
// 10.5 / 4.5 -> 3.6 / 3.6 on 32 x 14 tiles (21 warps at 80 registers, one block
// per SM; 32 x 16 tiles, 23 warps, 3.7 / 3.65: they would reach 78 000 nodes
// instead of 68 000, and no size in between was measured; two nodes a thread, to
// fit two blocks, spilled: 6.4 / 4.0).
// Two-point wall extrapolation: 160 x 40 11.8 / 4.1 -> 4.5 / 1.6; its large
// tiles lose beside others once they fill the GPU (391 x 173 12.3 / 5.4 -> 7.2
// / 7.1), so they stop at half.
using RS = ResCfg<P, 16, 8>;
using RL = ResCfg<P, 32, 14>;
int resident_large(const Params &p) { return p.extrap ? resident_sms() / 2 : resident_sms(); }
int resident_plan(const Params &p) { return choose_resident<RS, RL>(p, resident_large(p)); }
cudaError_t resident(const Params &p, const ResidentPtrs &s, int plan, int parity, int64_t k0, int n,
                     cudaStream_t st) {
  return launch_resident<RS, RL>(p, s, plan, parity, k0, n, st);
}

// the server's batch tile shapes: the global-memory tiles V0-V3
constexpr int kBatchShapes = 4;
TileShape batch_shape(int b) { return shape(b); }
cudaError_t batch_step(int b, BatchLattice *lats, int nlats, const BatchTile *interior, int ni, const BatchTile *edge,
                       int ne, const BatchTile *edge_lin, int nl, int it, int *err, cudaStream_t st,
                       const StreamFork *fork) {
  switch (b) {
    case 1: return launch_batch_step<V1>(lats, nlats, interior, ni, edge, ne, edge_lin, nl, it, err, st, fork);
    case 2: return launch_batch_step<V2>(lats, nlats, interior, ni, edge, ne, edge_lin, nl, it, err, st, fork);
    case 3: return launch_batch_step<V3>(lats, nlats, interior, ni, edge, ne, edge_lin, nl, it, err, st, fork);
    default: return launch_batch_step<V0>(lats, nlats, interior, ni, edge, ne, edge_lin, nl, it, err, st, fork);
  }
}

const Launchers kL = {kVariants,
                      (1 << 4) | (1 << 5) | (1 << 6) | (1 << 7) | (1 << 9),
                      default_variant,
                      shape,
                      name,
                      step,
                      kernels_per_step,
                      iterations_per_call,
                      step1,
                      kernels_per_step1,
                      launch_edge_table<P::real>,
                      launch_batch_edges<P::real>,
                      coef,
                      resident_plan,
                      resident,
                      tma_maps,
                      launch_init<V0>,
                      launch_fields<V0>,
                      launch_monitor<V0>,
                      launch_probe<V0>,
                      launch_grid_error<V0>,
                      batch_step,
                      kBatchShapes,
                      batch_shape,
                      sizeof(typename P::gs),
                      sizeof(typename P::us),
                      sizeof(typename P::real)};
}  // namespace

const Launchers &launchers_fp32() { return kL; }

}  // namespace lbs
