// FP16 storage (scaled), FP32 arithmetic, u as a float pair: kernel instantiations and launchers of liblbs.
#include <string.h>

#include "lbs_device.cuh"
#include "lbs_batch.cuh"
#include "lbs_column.cuh"
#include "lbs_resident.cuh"

namespace lbs {
namespace {
using P = F16;
// tile variants (nodes along x, nodes along y, thread rows)
using V0 = Cfg<P, 32, 16, 8>;
using V1 = Cfg<P, 32, 8, 8>;
using V2 = Cfg<P, 64, 8, 4>;
using V3 = Cfg<P, 32, 32, 8>;
using V4 = Cfg<P, 32, 16, 8>;
using M6 = MarchCfg<V4, 8, 128, 2>;
// 0-3: V0-V3 tiles read from global memory; 4: V4 tiles staged by TMA;
// 5: V4 tiles, persistent blocks with a two-stage TMA ring; 6: row-marching
// strips over the V4 tile columns; 7: V3 tiles staged by TMA; 8: warp columns
// (two iterations per launch on periodic lattices of even width, else one, with
// V0 frame tiles)
constexpr int kVariants = 9;
// lattices from this many nodes on take variant 8 (us per iteration, variant 7
// / 8; periodic, two iterations per launch: 1024^2 22.4 / 32.5, 1536^2 56.0 /
// 48.5, 6000 x 400 55.9 / 50.2, 4096^2 236 / 210, 16384^2 3381 / 3001; walled:
// 1021 x 509 18.9 / 33.2, 1500 x 1000 39.1 / 39.7, 400 x 5000 62.7 / 57.6, 2048^2
// 83.3 / 72.7, 3000 x 1501 85.5 / 74.7, 4096^2 246 / 241, 6000 x 5000 419 / 417)
constexpr int64_t kColumnNodes = 1 << 21;
// lines of default_variant
constexpr int64_t kSmallNodes = 400000, kWaveNodes = 800000;

TileShape shape(int v) {
  switch (v) {
    case 1: return {V1::TX, V1::TY};
    case 2: return {V2::TX, V2::TY};
    case 3:
    case 7: return {V3::TX, V3::TY};
    case 4:
    case 5:
    case 6: return {V4::TX, V4::TY};
    case 8: return {64, 64};
    default: return {V0::TX, V0::TY};
  }
}

const char *name(int v) {
  switch (v) {
    case 4: return "step_tma_kernel";
    case 5: return "step_tma2_kernel";
    case 6: return "step_march_kernel";
    case 7: return "step_tma_kernel";
    case 8: return "step_column_kernel";
    default: return "step_interior_kernel";
  }
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
    case 8: return column_wraps(p) ? launch_column_periodic<P, 2>(p, s, st) : launch_step_column<V0>(p, s, st);
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
    case 8: return column_wraps(p) ? 1 : step_kernel_count<V0>(p);
    default: return step_kernel_count<V0>(p);
  }
}

int iterations_per_call(const Params &p, int v) { return v == 8 && column_wraps(p) ? 2 : 1; }

cudaError_t step1(const Params &p, const StepPtrs &s, int, cudaStream_t st) {
  return launch_column_periodic<P, 1>(p, s, st);
}
int kernels_per_step1(const Params &, int) { return 1; }

// Below the columns, by size and edges; us per iteration, one lattice alone /
// three side by side.  Small lattices pull from global memory (walled 300^2
// variant 0 6.8 / 3.0, 7 11.6 / 3.6; 512^2 7.9 / 5.3, 15.4 / 5.4). Walled ones of
// several waves take the smaller TMA tiles, which leave fewer nodes to the frame
// tiles (4096 x 256 variant 4 21.1 / 18.4, 7 24.1 / 21.3; 2650 x 463 24.4 / 20.9, 25.1
// / 21.6; 1500 x 1300 36.6 / 31.9, 36.5 / 30.6); the rest the larger (1021 x 509
// variant 4 15.3 / 9.9, 7 16.7 / 9.6; 1024^2 periodic 23.0 / 18.5, 21.6 / 17.8).
int default_variant(const Params &p) {
  const int64_t nodes = (int64_t)p.nx * p.ny;
  if (nodes >= kColumnNodes) return 8;
  if (nodes < kSmallNodes) return 0;
  return nodes >= kWaveNodes && !(p.per_x && p.per_y) ? 4 : 7;
}

bool tma_maps(const Params &p, int v, const void *g, const void *u, void *og, void *ou) {
  if (v == 6) return make_march_maps<V4, M6>(p, g, u, og, ou);
  if (v == 7) return make_tma_maps<V3>(p, g, u, og, ou);
  if (v != 4 && v != 5) return false;
  return make_tma_maps<V4>(p, g, u, og, ou);
}

void coef(const Params &p, void *out) {
  const auto k = make_coef<P::gs, P::real>(p);
  memcpy(out, &k, sizeof(k));
}

// resident launches: the tiles and lines of single precision (us per iteration
// on walled neo-Hooke lattices, one lattice alone / three side by side, against
// launching every iteration from a graph: 40 x 40 11.4 / 3.9 -> 2.7 / 0.90,
// 128 x 128 11.4 / 4.0 -> 3.0 / 2.1, 256 x 256 11.8 / 5.1 -> 3.7 / 3.8)
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
                      (1 << 4) | (1 << 5) | (1 << 6) | (1 << 7),
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

const Launchers &launchers_fp16() { return kL; }

}  // namespace lbs
