// Resident iterations of liblbs: many iterations of a small lattice in one
// cooperative launch.  Included by kernels_fp64.cu / kernels_fp32.cu /
// kernels_fp16.cu after lbs_device.cuh.
#pragma once
#include <atomic>

#include "lbs_device.cuh"

namespace lbs {

template <class Pr, int TX_, int TY_>
struct ResCfg : ResGeom<TX_, TY_> {
  using PrT = Pr;
  using real = typename Pr::real;
  using us = typename Pr::us;
  using gs = typename Pr::gs;
};

// Barrier over the blocks of one cooperative launch: every block adds one to
// *count, thread 0 polls until `target` arrivals (a bounded number of times:
// false, with *err set, if they do not come).  The release of the arrival
// covers the block's stores (ordered before it by the block barrier), the
// acquire of the poll the reads that follow.  (Anything more in the loop shows:
// a limit handed in took 256 x 256 FP32 from 1.75 to 1.84 ms for 500 iterations,
// a mark in the count that ends the wait early to 1.79.)
constexpr uint32_t kMaxBarrierPolls = 1u << 22;
__device__ __forceinline__ bool grid_barrier(unsigned *count, unsigned target, int *err) {
  __syncthreads();
  int ok = 1;
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
    ok = 0;
    for (uint32_t i = 0; i < kMaxBarrierPolls; ++i) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
      if (v >= target) {
        ok = 1;
        break;
      }
    }
    if (!ok) atomicExch(err, 1);
  }
  return __syncthreads_and(ok) != 0;
}

// iterations whose edge values are evaluated at once
constexpr int kSevBatch = 32;

// n iterations from iteration k0 (buffers of `parity`) of the whole lattice,
// one block per tile, a grid barrier between iterations.  The phases are those
// of step_tile with every node's operations unchanged (the results are the
// same bits), but what does not depend on the iteration is computed once: each
// thread keeps its node's streaming sources, its finite-difference taps and
// u(t) in registers (u on the halo is recomputed by every block that needs
// it, so it never travels), and own nodes keep their g.  g and the walls' N go
// through L2, both buffers in turn; u is stored by the last iteration.  The
// barrier's counters are zero between launches: the last block to leave clears
// them.  Where a block gives up waiting, the counters stay as they are and the
// error flag is set; a launch that finds it set does nothing, until setting the
// state anew clears both.
// What bounds an iteration: latency. Of the 2.6 us of 128 x 128 FP32 (128 blocks)
// the grid barrier alone takes 1.1, and the schedulers issue 12 % of the cycles;
// in FP64 a dependent operation takes 303 cycles, some 40 of them in a row in
// the 7.5 us of 40 x 40.
// CLUSTER: the grid is one thread-block cluster, whose hardware barrier takes
// 0.5 us where the grid barrier takes 0.9 at 16 blocks (it orders global memory
// within the cluster, and cannot run out: a cluster's blocks run together).
// 32 x 32 FP32: 0.34 -> 0.30 ms for 400 iterations among three lattices.
template <class C, bool LIN, bool CLUSTER>
__global__ void __launch_bounds__(C::NT) resident_kernel(const Params P, const Coef<typename C::real> c,
                                                         const ResidentPtrs S, int parity, int64_t k0, int n,
                                                         int ntx) {
  using gs = typename C::gs;
  using us = typename C::us;
  using R = typename C::real;
  using T = EdgeType<R, LIN>;
  __shared__ us su[C::R2H * C::R2W];
  __shared__ R sn[4][C::R1H * C::R1W];
  __shared__ T sev[kSevBatch][kEdgeEntries][2];
  int bad = 0;
  if (threadIdx.x == 0) bad = *(volatile int *)S.err;
  if (__syncthreads_or(bad)) return;

  const int x0 = (int)(blockIdx.x % ntx) * C::TX, y0 = (int)(blockIdx.x / ntx) * C::TY;
  const int plane = P.ny * P.pitch;
  const bool walls = !(P.per_x && P.per_y);
  const R scl = c.scl, kap = c.kap, sbx = c.sbxs, sby = c.sbys, ics2 = c.ics2, cj = c.cj;

  // phase 1: this thread's node of R2
  const int e = threadIdx.x;
  int rx = 0, ry = 0, x = 0, y = 0, idx = 0, src[9], xw = -1, yw = -1;
  bool in = false, own = false;
  us uu;
  if (e < C::OWN + C::NRING) {
    resident_pos<C>(e, rx, ry);
    x = x0 - 2 + rx;
    y = y0 - 2 + ry;
    own = e < C::OWN && x < P.nx && y < P.ny;
    in = locate(P, x, y);
  }
  const int us_at = ry * C::R2W + rx;
  if (in) {
    idx = y * P.pitch + x;
    walls_of(P, x, y, xw, yw);
    int xb, xf, yb, yf;
    stream_sides(x, P.nx, P.per_x, xb, xf);
    stream_sides(y, P.ny, P.per_y, yb, yf);
#pragma unroll
    for (int q = 0; q < 9; ++q)
      src[q] = q * plane + (ey(q) > 0 ? yb : (ey(q) < 0 ? yf : y)) * P.pitch +
               (ex(q) > 0 ? xb : (ex(q) < 0 ? xf : x));
    uu = ld_coh((const us *)S.u[parity] + idx);
  }
  const bool nx_ = xw >= 0 && P.etype[xw] == LBS_NEUMANN, ny_ = yw >= 0 && P.etype[yw] == LBS_NEUMANN;
  const int wx_at = nx_ ? (int)side_entry(P, 0, xw, y) : 0, wy_at = ny_ ? (int)side_entry(P, 0, yw, x) : 0;

  // phase 2: this thread's node of R1 and its taps of u
  const int r1x = e % C::R1W, r1y = e / C::R1W;
  int ux1 = 0, ux0 = 0, uy1 = 0, uy0 = 0, gx1 = x0 - 1 + r1x, gy1 = y0 - 1 + r1y;
  bool in1 = e < C::R1W * C::R1H && locate(P, gx1, gy1), keep1 = false;
  bool onex1 = false, oney1 = false;
  if (in1) {
    int xa, xb, ya, yb;
    fd_taps<true>(P, r1x + 1, r1y + 1, gx1, gy1, xa, xb, ya, yb, onex1, oney1);
    ux1 = (r1y + 1) * C::R2W + xa;
    ux0 = (r1y + 1) * C::R2W + xb;
    uy1 = ya * C::R2W + r1x + 1;
    uy0 = yb * C::R2W + r1x + 1;
    keep1 = r1_own_node<C>(P, x0, y0, r1x, r1y) && (on_wall(P, gx1, gy1) || (LIN && P.extrap));
  }
  // phase 3: the own node's taps of N
  int nx1 = 0, nx0 = 0, ny1 = 0, ny0 = 0;
  R sx2 = 0, sy2 = 0;
  if (own) {
    int xa, xb, ya, yb;
    bool onex, oney;
    fd_taps<true>(P, rx - 1, ry - 1, x, y, xa, xb, ya, yb, onex, oney);
    nx1 = (ry - 1) * C::R1W + xa;
    nx0 = (ry - 1) * C::R1W + xb;
    ny1 = ya * C::R1W + rx - 1;
    ny0 = yb * C::R1W + rx - 1;
    sx2 = onex ? c.idxs : c.hdxs;
    sy2 = oney ? c.idxs : c.hdxs;
  }

  R g0[9];
  for (int it = 0; it < n; ++it) {
    const int p = (parity + it) & 1;
    const gs *g = (const gs *)S.g[p];
    const R *bnd = (const R *)S.b[p];
    R f[9], wn[4] = {R(0), R(0), R(0), R(0)};
    if (in) {
      if (nx_) {
        wn[0] = ld_coh(bnd + wx_at);
        wn[1] = ld_coh(bnd + wx_at + 2);
      }
      if (ny_) {
        wn[2] = ld_coh(bnd + wy_at + 3);
        wn[3] = ld_coh(bnd + wy_at + 1);
      }
#pragma unroll
      for (int q = 0; q < 9; ++q) f[q] = half_wide(ld_coh(g + src[q]));
      if (it == 0 || !own) {
#pragma unroll
        for (int q = 0; q < 9; ++q) g0[q] = half_wide(ld_coh(g + (q * plane + idx)));
      }
    }
    if (walls && it % kSevBatch == 0) {
      // (while the populations are in flight)
      constexpr int E = LIN ? 4 : kEdgeEntries;
      for (int j = threadIdx.x; j < kSevBatch * E; j += C::NT)
        if (it + j / E < n) edge_entry<T>(P, j % E, k0 + it + j / E, sev[j / E][j % E]);
      __syncthreads();
    }
    if (in) {
      if (xw >= 0 || yw >= 0) {
        if constexpr (LIN) {
          R wnl[4];
          wall_n<true>(P, bnd, xw, yw, x, y, wnl);
          wall_rules<R, gs, true>(P, bnd, g, sev[it % kSevBatch], x, y, xw, yw, wnl, g0, crosses_x(xw) | crosses_y(yw),
                                  f, ics2, cj);
        } else {
          wall_rules_own<R>(P, xw, yw, sev[it % kSevBatch], ics2, cj, wn, g0, f);
        }
      }
      R gmx, gmy, fmx, fmy;
      first_moment(g0, gmx, gmy);
      first_moment(f, fmx, fmy);
      uu = uadd_k(uu, kap, gmx + fmx, gmy + fmy);
      su[us_at] = uu;
    }
    __syncthreads();
    if (in1) {
      R N[4], dxx, dxy, dyx, dyy;
      udiff(su[ux1], su[ux0], dxx, dxy);
      udiff(su[uy1], su[uy0], dyx, dyy);
      stress_n<R>(P, c, dxx, dxy, dyx, dyy, onex1, oney1, N);
#pragma unroll
      for (int m = 0; m < 4; ++m) sn[m][e] = N[m];
      if (keep1) {
        R *bo = (R *)S.b[p ^ 1];
        if (on_wall(P, gx1, gy1)) store_wall_n<R>(P, bo, gx1, gy1, N);
        if (LIN && P.extrap) store_inner_n<R>(P, bo, gx1, gy1, N);
      }
    }
    __syncthreads();
    if (own) {
      const R Sx = fmr(sn[0][nx1] - sn[0][nx0], sx2, fmr(sn[1][ny1] - sn[1][ny0], sy2, sbx));
      const R Sy = fmr(sn[2][nx1] - sn[2][nx0], sx2, fmr(sn[3][ny1] - sn[3][ny0], sy2, sby));
      collide<R>(f, Sx, Sy, c.K);
      gs *go = (gs *)S.g[p ^ 1];
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        gstore(go, (size_t)(q * plane + idx), f[q], scl);
        if constexpr (sizeof(gs) == 2) g0[q] = __half2float(__float2half_rn(f[q]));
        else g0[q] = f[q];
      }
    }
    if (CLUSTER) {
      asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    } else if (it + 1 < n && gridDim.x > 1) {
      if (!grid_barrier(S.bar, (unsigned)(it + 1) * gridDim.x, S.err)) return;
    } else {
      __syncthreads();
    }
  }
  if (own) ((us *)S.u[(parity + n) & 1])[idx] = uu;
  if (!CLUSTER && gridDim.x > 1 && threadIdx.x == 0 && atomicAdd(&S.bar[1], 1u) == gridDim.x - 1) {
    S.bar[0] = 0;
    S.bar[1] = 0;
  }
}

// A figure of the current device, evaluated once per device.
class PerDevice {
 public:
  template <class F>
  int get(F f) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return f(dev);
    int x = v_[dev].load(std::memory_order_relaxed);
    if (x == 0) {
      x = f(dev) + 1;
      v_[dev].store(x, std::memory_order_relaxed);
    }
    return x - 1;
  }

 private:
  static constexpr int kDevices = 64;
  std::atomic<int> v_[kDevices] = {};  // the figure plus one, 0: not evaluated yet
};

inline int resident_sms() {
  static PerDevice sms;
  return sms.get([](int dev) {
    int n = 0;
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n;
  });
}

// blocks of a resident kernel that are on the GPU at once
template <class C, bool LIN>
int resident_capacity() {
  static PerDevice per;
  return resident_sms() * per.get([](int) {
    int n = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, resident_kernel<C, LIN, false>, C::NT, 0);
    return n;
  });
}

template <class C>
int resident_tiles(const Params &P) {
  const int64_t n = (int64_t)((P.nx + C::TX - 1) / C::TX) * ((P.ny + C::TY - 1) / C::TY);
  return n < (1 << 20) ? (int)n : 1 << 20;
}

// Largest cluster of resident blocks: 16 (non-portable) where the GPU places
// one, else 0.  The permission belongs to the kernel on one device (and ends
// with its context), so it is given for every handle; a launch without it is
// refused.
constexpr int kClusterMost = 16;
template <class C, bool LIN>
int resident_cluster() {
  if (cudaFuncSetAttribute(resident_kernel<C, LIN, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
      cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  static PerDevice most;
  return most.get([](int) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    cfg.gridDim = dim3(kClusterMost);
    cfg.blockDim = dim3(C::NT);
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim = {kClusterMost, 1, 1};
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, resident_kernel<C, LIN, true>, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
    return n > 0 ? kClusterMost : 0;
  });
}

// How a lattice's resident launches run, chosen once per handle on its device:
// on the small tile while every tile has an SM of its own (as one cluster where
// that holds them), on the large one while its tiles number at most
// `large_most`, not at all (kResidentNone) for larger lattices, which advance
// one iteration per launch.  Small tiles have the shorter iteration, large ones
// reach further and leave room for other lattices' launches (each shape's lines
// are measured at the precisions' instantiations).
template <class Small, class Large, bool LIN>
int choose_resident_of(const Params &P, int large_most) {
  const int ns = resident_tiles<Small>(P), nl = resident_tiles<Large>(P);
  if (ns <= resident_sms() && ns <= resident_capacity<Small, LIN>()) {
    if (ns == 1) return kResidentOne;
    return ns <= kClusterMost && ns <= resident_cluster<Small, LIN>() ? kResidentCluster : kResidentSmall;
  }
  if (nl <= large_most && nl <= resident_capacity<Large, LIN>()) return kResidentLarge;
  return kResidentNone;
}
template <class Small, class Large>
int choose_resident(const Params &P, int large_most) {
  return P.extrap ? choose_resident_of<Small, Large, true>(P, large_most)
                  : choose_resident_of<Small, Large, false>(P, large_most);
}

template <class C, bool LIN>
cudaError_t launch_resident_cluster(const Params &P, const ResidentPtrs &S, int parity, int64_t k0, int n, int ntx,
                                    int ntiles, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  cfg.gridDim = dim3(ntiles);
  cfg.blockDim = dim3(C::NT);
  cfg.stream = st;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim = {(unsigned)ntiles, 1, 1};
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, resident_kernel<C, LIN, true>, P, make_coef<typename C::gs, typename C::real>(P), S,
                            parity, k0, n, ntx);
}

// (only the small tile has lattices of so few)
template <class C, bool SMALL>
cudaError_t launch_resident_c(const Params &P, const ResidentPtrs &S, bool cluster, int parity, int64_t k0, int n,
                              cudaStream_t st) {
  int ntx = (P.nx + C::TX - 1) / C::TX, nty = (P.ny + C::TY - 1) / C::TY;
  const int ntiles = ntx * nty;
  if constexpr (SMALL) {
    if (cluster)
      return P.extrap ? launch_resident_cluster<C, true>(P, S, parity, k0, n, ntx, ntiles, st)
                      : launch_resident_cluster<C, false>(P, S, parity, k0, n, ntx, ntiles, st);
  }
  auto c = make_coef<typename C::gs, typename C::real>(P);
  void *args[] = {(void *)&P, &c, (void *)&S, &parity, &k0, &n, &ntx};
  const void *kernel = P.extrap ? (const void *)resident_kernel<C, true, false>
                                : (const void *)resident_kernel<C, false, false>;
  return cudaLaunchCooperativeKernel(kernel, dim3(ntiles), dim3(C::NT), args, 0, st);
}

template <class Small, class Large>
cudaError_t launch_resident(const Params &P, const ResidentPtrs &S, int plan, int parity, int64_t k0, int n,
                            cudaStream_t st) {
  switch (plan) {
    case kResidentOne:
    case kResidentSmall:
    case kResidentCluster: return launch_resident_c<Small, true>(P, S, plan == kResidentCluster, parity, k0, n, st);
    case kResidentLarge: return launch_resident_c<Large, false>(P, S, false, parity, k0, n, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lbs
