// FP64 storage and arithmetic: kernel instantiations and launchers of liblbs.
#include <string.h>

#include "lbs_device.cuh"
#include "lbs_batch.cuh"
#include "lbs_resident.cuh"

namespace lbs {
namespace {
using P = F64;
// tile variants (nodes along x, nodes along y, thread rows)
using V0 = Cfg<P, 32, 16, 8>;
using V1 = Cfg<P, 32, 8, 8>;
using V2 = Cfg<P, 64, 8, 4>;
using V3 = Cfg<P, 32, 24, 8>;  // 32x32 would need 57 KB of static shared memory in FP64
using V4 = Cfg<P, 32, 8, 8>;  // interior tiles staged by TMA
constexpr int kVariants = 5;

TileShape shape(int v) {
  switch (v) {
    case 1: return {V1::TX, V1::TY};
    case 2: return {V2::TX, V2::TY};
    case 3: return {V3::TX, V3::TY};
    case 4: return {V4::TX, V4::TY};
    default: return {V0::TX, V0::TY};
  }
}

const char *name(int v) {
  switch (v) {
    case 4: return "step_tma_kernel";
    default: return "step_interior_kernel";
  }
}

cudaError_t step(const Params &p, const StepPtrs &s, int v, cudaStream_t st) {
  switch (v) {
    case 1: return launch_step<V1>(p, s, st);
    case 2: return launch_step<V2>(p, s, st);
    case 3: return launch_step<V3>(p, s, st);
    case 4: return launch_step_tma<V4>(p, s, st);
    default: return launch_step<V0>(p, s, st);
  }
}

int kernels_per_step(const Params &p, int v) {
  switch (v) {
    case 1: return step_kernel_count<V1>(p);
    case 2: return step_kernel_count<V2>(p);
    case 3: return step_kernel_count<V3>(p);
    case 4: return step_kernel_count<V4>(p);
    default: return step_kernel_count<V0>(p);
  }
}

int iterations_per_call(const Params &, int) { return 1; }
cudaError_t step1(const Params &p, const StepPtrs &s, int v, cudaStream_t st) { return step(p, s, v, st); }
int kernels_per_step1(const Params &p, int v) { return kernels_per_step(p, v); }

// the fastest on the 4096^2 and 16384^2 periodic lattices
int default_variant(const Params &) { return 3; }

bool tma_maps(const Params &p, int v, const void *g, const void *u, void *og, void *ou) {
  if (v != 4) return false;
  return make_tma_maps<V4>(p, g, u, og, ou);
}

void coef(const Params &p, void *out) {
  const auto k = make_coef<P::gs, P::real>(p);
  memcpy(out, &k, sizeof(k));
}

// resident launches (us per iteration on walled neo-Hooke lattices, one lattice
// alone / three side by side, against launching every iteration from a graph):
// 40 x 40 27.5 / 9.2 -> 7.5 / 2.5, 160 x 40 26.2 / 8.8 -> 7.5 / 3.5 and 96 x 96
// 30.1 / 10.2 -> 7.5 / 6.7 on 8 x 8 tiles, 128 x 128 30.3 / 10.3 -> 15.4 / 10.2 on
// 16 x 16 tiles.  FP64 operations bound both (a warp's operation holds its
// scheduler's FP64 unit for tens of cycles), so a tile's halo is dear: past
// half the SMs the 16 x 16 tiles lose beside others (160 x 160 31.6 / 15.1 ->
// 19.7 / 19.6), and with the two-point wall extrapolation they do not pay.
using RS = ResCfg<P, 8, 8>;
using RL = ResCfg<P, 16, 16>;
int resident_large(const Params &p) { return p.extrap ? 0 : resident_sms() / 2; }
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
                      1 << 4,
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

const Launchers &launchers_fp64() { return kL; }

}  // namespace lbs
