// Small lattices whose kernel may not (or may no longer) run as a thread-block
// cluster of more than eight blocks.  The permission for those belongs to a
// kernel on one device; a device on which it was never given is stood in for
// by withdrawing it.  Linked with the library's objects, with calls of
// cudaFuncSetAttribute passing through here.  Prints "ok" and exits 0, else
// names the check.
#include <cuda_runtime.h>
#include <stdio.h>
#include <string.h>

#include <set>
#include <vector>

#include "lbs.h"

static std::set<const void *> g_given;  // kernels given the permission
static int g_refuse = 0;                // the runtime refuses to give it

extern "C" cudaError_t __real_cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v);
extern "C" cudaError_t __wrap_cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v) {
  if (a != cudaFuncAttributeNonPortableClusterSizeAllowed) return __real_cudaFuncSetAttribute(f, a, v);
  g_given.insert(f);
  return g_refuse ? cudaErrorNotSupported : __real_cudaFuncSetAttribute(f, a, v);
}
static bool withdraw() {
  for (const void *f : g_given)
    if (__real_cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 0) != cudaSuccess) return false;
  return true;
}

#define CHECK(cond)                                                                              \
  do {                                                                                           \
    if (!(cond)) {                                                                               \
      printf("failed: %s (%dx%d, precision %d, extrapolation %d, %s: %s)\n", #cond, nx, ny,       \
             precision, extrap, what, lbs_last_error());                                         \
      return false;                                                                              \
    }                                                                                            \
  } while (0)

// ten iterations in one launch and four more; `between`: withdraw the
// permission when the handle has been created
static bool run(int nx, int ny, int precision, int extrap, const char *what, bool between, std::vector<double> &u) {
  lbs_lattice lat;
  memset(&lat, 0, sizeof(lat));
  lat.nx = nx;
  lat.ny = ny;
  lat.dx = 0.01;
  lat.tau = 0.55;
  lat.precision = precision;
  lat.wall_extrap = extrap;
  lbs_material mat = {LBS_NH, 1.0, 0.2, 1.0, {0.01, 0.0}};
  lbs_handle *h = nullptr;
  CHECK(lbs_create(&lat, &mat, nullptr, &h) == LBS_OK);
  if (between) CHECK(withdraw());
  const int64_t before = lbs_launch_count(h);
  CHECK(lbs_step(h, 10) == LBS_OK);
  CHECK(lbs_step(h, 4) == LBS_OK);
  CHECK(lbs_launch_count(h) - before == 2);
  CHECK(lbs_sync(h) == LBS_OK);
  u.assign((size_t)2 * nx * ny, 0.0);
  CHECK(lbs_fields(h, u.data(), nullptr, nullptr) == LBS_OK);
  CHECK(lbs_destroy(h) == LBS_OK);
  return true;
}

int main() {
  // 15, 16 and 9 blocks (beyond the portable cluster), 8 (within it), a grid
  // without cluster, one block
  const int cases[][4] = {{40, 40, LBS_FP32, LBS_EXTRAP_OWN},  {32, 32, LBS_FP64, LBS_EXTRAP_OWN},
                          {33, 20, LBS_FP16S, LBS_EXTRAP_OWN}, {40, 40, LBS_FP32, LBS_EXTRAP_LINEAR},
                          {32, 32, LBS_FP16S, LBS_EXTRAP_OWN}, {100, 90, LBS_FP32, LBS_EXTRAP_OWN},
                          {16, 8, LBS_FP32, LBS_EXTRAP_OWN}};
  for (auto &c : cases) {
    std::vector<double> ref, u;
    auto same = [&](const char *what) {
      if (u.size() == ref.size() && memcmp(u.data(), ref.data(), u.size() * sizeof(double)) == 0) return true;
      printf("failed: %dx%d, precision %d differs %s\n", c[0], c[1], c[2], what);
      return false;
    };
    if (!run(c[0], c[1], c[2], c[3], "first", false, ref)) return 1;
    // a device on which no handle has asked for it yet
    if (!withdraw() || !run(c[0], c[1], c[2], c[3], "not given yet", false, u) || !same("where it was not given")) return 1;
    // refused at the launch
    if (!run(c[0], c[1], c[2], c[3], "refused at the launch", true, u) || !same("refused at the launch")) return 1;
    // refused when the handle asks
    g_refuse = 1;
    if (!withdraw() || !run(c[0], c[1], c[2], c[3], "refused", false, u) || !same("refused")) return 1;
    g_refuse = 0;
  }
  printf("ok\n");
  return 0;
}
