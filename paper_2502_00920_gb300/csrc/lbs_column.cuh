// Warp columns of liblbs: one warp advances a strip of 64 lattice columns, two
// per lane, marching up the rows with everything in registers; its x
// neighbours come by shuffles.  Single-precision arithmetic (FP32 and FP16
// storage).  Included by kernels_fp32.cu / kernels_fp16.cu after
// lbs_device.cuh.
//
// Why: the TMA-staged tiles read and write the state once per iteration (FP32:
// 104 B a node, which at 16384^2 takes the copy bandwidth's time, 4.20 ms) and
// pass every value through shared memory several times (FP16 storage: the
// shared-memory pipe was 80 % busy, 3.38 ms). Two iterations per pass over the
// state halve the bytes; values kept in registers halve the shared-memory
// work. 16384^2 periodic, ms per iteration: FP32 4.20 -> 3.27 (two iterations
// per launch), FP16 storage 3.38 -> 3.00. What bounds it now: instruction
// issue and latency with the 12 warps an SM holds at 168 registers (4096^2
// FP32: issue 59 %, shared-memory pipe 63 %, DRAM 4.1 TB/s). Packed FP32
// instructions (add.f32x2 and so on) measured the same (two issue cycles each)
// and ptxas fuses their products into sums, which changes the rounding.
#pragma once
#include "lbs_device.cuh"

namespace lbs {

// ------------------------------------------------------------------ pairs
// The values of a lane's two neighbouring nodes.
struct alignas(8) Two {
  float x, y;
};
__device__ __forceinline__ Two two(float a, float b) { return {a, b}; }
__device__ __forceinline__ Two two(float a) { return {a, a}; }
__device__ __forceinline__ float lo(Two a) { return a.x; }
__device__ __forceinline__ float hi(Two a) { return a.y; }
__device__ __forceinline__ Two operator+(Two a, Two b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ Two operator-(Two a, Two b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ Two operator*(Two a, Two b) { return {a.x * b.x, a.y * b.y}; }
__device__ __forceinline__ Two fmr(Two a, Two b, Two c) { return {fmr(a.x, b.x, c.x), fmr(a.y, b.y, c.y)}; }

constexpr unsigned kAll = 0xffffffffu;

// (value at c - 1, value at c) and (value at c + 1, value at c + 2) of this
// lane's columns c, c + 1; the strip's outermost columns get their own value
__device__ __forceinline__ Two from_left(Two a) { return two(__shfl_up_sync(kAll, hi(a), 1), lo(a)); }
__device__ __forceinline__ Two from_right(Two a) { return two(hi(a), __shfl_down_sync(kAll, lo(a), 1)); }
__device__ __forceinline__ uint32_t from_left(uint32_t a) {
  return __byte_perm(__shfl_up_sync(kAll, a, 1), a, 0x5432);
}
__device__ __forceinline__ uint32_t from_right(uint32_t a) {
  return __byte_perm(a, __shfl_down_sync(kAll, a, 1), 0x5432);
}

// a stored pair of populations: two floats, or two halves in one word
template <class Pr>
struct RawOf {
  using type = Two;
};
template <>
struct RawOf<F16> {
  using type = uint32_t;
};
__device__ __forceinline__ Two wide(Two a) { return a; }
__device__ __forceinline__ Two wide(uint32_t a) {
  const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&a));
  return two(f.x, f.y);
}
__device__ __forceinline__ void narrow(Two a, Two &out) { out = a; }
__device__ __forceinline__ void narrow(Two a, uint32_t &out) {
  const __half2 h = __floats2half2_rn(lo(a), hi(a));
  out = *reinterpret_cast<const uint32_t *>(&h);
}

// both halves the first
__device__ __forceinline__ Two first_of(Two a) { return two(lo(a)); }
__device__ __forceinline__ uint32_t first_of(uint32_t a) { return __byte_perm(a, a, 0x1010); }

// neo-Hooke where J < 1/2: double precision, out of line (as material())
static __device__ __noinline__ float4 nh_wide(double lam, double mu, float h11, float h12, float h21, float h22) {
  const double H[4] = {h11, h12, h21, h22};
  double N[4];
  constitutive_n<double>(LBS_NH, lam, mu, H, N);
  return make_float4((float)N[0], (float)N[1], (float)N[2], (float)N[3]);
}

// constitutive_n<float> on two nodes: the same operations, with negations
// folded into factors (exact).  This and collide_v2 follow the functions they
// restate operation by operation (tests/test_column_gpu.py compares the bits):
// a change of either belongs in both.
__device__ __forceinline__ void stress_v2(const Params &P, const Coef<float> &c, Two dxx, Two dxy, Two dyx, Two dyy,
                                          Two N[4]) {
  const Two h = two(c.hdx);
  const Two h11 = dxx * h, h12 = dyx * h, h21 = dxy * h, h22 = dyy * h;
  const Two trH = h11 + h22;
  if (P.model == LBS_NH) {
    const Two nh12 = dyx * two(-c.hdx);
    const Two detH = fmr(h11, h22, nh12 * h21);
    const Two a = trH + detH;
    const Two one = two(1.0f);
    const Two J = one + a;
    const Two iJ = two(1.0f / lo(J), 1.0f / hi(J));
    const Two m = two(c.mu) * iJ, nma = (two(-c.mu) * iJ) * a;
    const Two nt2 = two(-2.0f) - a;
    const Two l = two(-0.5f * c.lam) * a * nt2 * iJ;
    const Two diag = m * fmr(nt2, trH, a);
    const Two w = nma - l;
    N[0] = fmr(nma, h11, fmr(l, one + h22, diag));
    N[1] = w * h21;
    N[2] = w * h12;
    N[3] = fmr(nma, h22, fmr(l, one + h11, diag));
    if (lo(J) < 0.5f || hi(J) < 0.5f) {
      float4 n0 = make_float4(lo(N[0]), lo(N[1]), lo(N[2]), lo(N[3]));
      float4 n1 = make_float4(hi(N[0]), hi(N[1]), hi(N[2]), hi(N[3]));
      if (lo(J) < 0.5f) n0 = nh_wide(P.lam, P.mu, lo(h11), lo(h12), lo(h21), lo(h22));
      if (hi(J) < 0.5f) n1 = nh_wide(P.lam, P.mu, hi(h11), hi(h12), hi(h21), hi(h22));
      N[0] = two(n0.x, n1.x);
      N[1] = two(n0.y, n1.y);
      N[2] = two(n0.z, n1.z);
      N[3] = two(n0.w, n1.w);
    }
  } else if (P.model == LBS_SVK) {
    const Two lam = two(c.lam), mu = two(c.mu), k2 = two(2.0f);
    const Two c11 = fmr(h11, h11, h21 * h21), c12 = fmr(h11, h12, h21 * h22), c22 = fmr(h12, h12, h22 * h22);
    const Two trE = fmr(two(0.5f), c11 + c22, trH);
    const Two s11 = fmr(lam, trE, mu * (k2 * h11 + c11));
    const Two s12 = mu * ((h12 + h21) + c12);
    const Two s22 = fmr(lam, trE, mu * (k2 * h22 + c22));
    const Two d = fmr(lam, trE, two(-c.mu) * trH);
    const Two mc12 = mu * c12;
    N[0] = fmr(h12, s12, fmr(h11, s11, fmr(mu, c11, d)));
    N[1] = fmr(h12, s22, fmr(h11, s12, mc12));
    N[2] = fmr(h22, s12, fmr(h21, s11, mc12));
    N[3] = fmr(h22, s22, fmr(h21, s12, fmr(mu, c22, d)));
  } else {
    const Two d = two(c.lam - c.mu) * trH;
    N[0] = d;
    N[1] = two(0.0f);
    N[2] = two(0.0f);
    N[3] = d;
  }
}

// collide<float> on two nodes
__device__ __forceinline__ void collide_v2(Two f[9], Two Sx, Two Sy, const CollideK<float> &K) {
  const Two s13 = f[1] + f[3], s24 = f[2] + f[4], s57 = f[5] + f[7], s68 = f[6] + f[8];
  const Two d13 = f[1] - f[3], d24 = f[2] - f[4], d57 = f[5] - f[7], d68 = f[6] - f[8];
  const Two Q = fmr(two(4.0f), s57 + s68, fmr(two(-2.0f), s13 + s24, f[0]));
  const Two s9 = two(K.s9), s36 = two(K.s36), mo = two(K.mo);
  const Two fx = Sx * s9, fy = Sy * s9;
  const Two f57 = (Sx + Sy) * s36, f68 = (Sy - Sx) * s36;
  const Two A1 = Q * two(K.a1), A5 = Q * two(K.a5);
  const Two nc3 = two(-(1.0f / 3.0f)), c3 = two(1.0f / 3.0f), c6 = two(1.0f / 6.0f), nc12 = two(-(1.0f / 12.0f));
  const Two ox = fmr(d13, c6, (d57 - d68) * nc3);
  const Two oy = fmr(d24, c6, (d57 + d68) * nc3);
  const Two o57 = fmr(d57, c3, (d13 + d24) * nc12);
  const Two o68 = fmr(d68, c3, (d24 - d13) * nc12);
  const Two bx = fmr(mo, ox, fx), by = fmr(mo, oy, fy), b57 = fmr(mo, o57, f57), b68 = fmr(mo, o68, f68);
  f[0] = fmr(mo, Q * two(1.0f / 9.0f), f[0]);
  f[1] = (f[1] + A1) + bx;
  f[3] = (f[3] + A1) - bx;
  f[2] = (f[2] + A1) + by;
  f[4] = (f[4] + A1) - by;
  f[5] = (f[5] + A5) + b57;
  f[7] = (f[7] + A5) - b57;
  f[6] = (f[6] + A5) + b68;
  f[8] = (f[8] + A5) - b68;
}

// ------------------------------------------------------------------ one row
// The state a warp carries up its strip.  Advancing by row r (step): row r's g
// arrives and with it f of row r - 1 is complete; u(t+dt) of row r - 1, N of
// row r - 2 and the new g of row r - 3 follow.  x differences are taken where a
// row is made and used one row later, off the step's critical path.  Rows
// rotate through four slots (I = r mod 4, a compile-time constant), so
// nothing is moved.
template <class Pr>
struct Column {
  using Raw = typename RawOf<Pr>::type;
  // populations 9 - kParked .. 8 are parked: 32-bit populations of two complete
  // rows would take the warp past 168 registers (three warps a scheduler), and
  // spilled registers come back from L2 here
  static constexpr int kParked = sizeof(typename Pr::gs) == 4 ? 7 : 0;
  Raw f[4][9];          // streamed populations
  Two u[4][4];           // (hi_x, hi_y, lo_x, lo_y) at t + dt
  Two n1[4], n3[4];      // N12, N22
  Two gmx, gmy;          // own first moment of the newest row
  Two udx, udy;          // x differences of u of the newest row (u_x, u_y)
  Two nd0, nd2;          // x differences of N11, N21 of the newest row

  __device__ __forceinline__ void clear() {
    const Two z = two(0.0f);
#pragma unroll
    for (int s = 0; s < 4; ++s) {
#pragma unroll
      for (int q = 0; q < 9; ++q) narrow(z, f[s][q]);
#pragma unroll
      for (int m = 0; m < 4; ++m) u[s][m] = z;
      n1[s] = n3[s] = z;
    }
    gmx = gmy = udx = udy = nd0 = nd2 = z;
  }

  // g: row r as stored; uk: u(t) of row r - 1; out: the new g of row r - 3
  // (whose u is u[(I + 1) & 3] until the next call).  `park`: this lane's words
  // in shared memory where kParked complete populations wait the two steps to
  // their collision (two rows in turn).
  template <int I>
  __device__ __forceinline__ void step(const Params &P, const Coef<float> &c, const Raw g[9], const Two uk[4],
                                       Raw out[9], Raw (*park)[kParked > 0 ? kParked : 1][32]) {
    constexpr int S0 = I, S1 = (I + 3) & 3, S2 = (I + 2) & 3, S3 = (I + 1) & 3;  // rows r, r-1, r-2, r-3 (= r+1)
    // row r - 1 is complete
    f[S1][4] = g[4];
    f[S1][7] = from_right(g[7]);
    f[S1][8] = from_left(g[8]);
    Two w[9], mx, my;
#pragma unroll
    for (int q = 1; q < 9; ++q) w[q] = wide(f[S1][q]);
    moment(w, mx, my);
    const Two kap = two(c.kap);
    pair_add2(uk[0], uk[2], kap * (gmx + mx), u[S1][0], u[S1][2]);
    pair_add2(uk[1], uk[3], kap * (gmy + my), u[S1][1], u[S1][3]);
#pragma unroll
    for (int q = 1; q < 9; ++q) w[q] = wide(g[q]);
    moment(w, gmx, gmy);
    // N of row r - 2
    Two N[4];
    stress_v2(P, c, udx, udy, (u[S1][0] - u[S3][0]) + (u[S1][2] - u[S3][2]),
              (u[S1][1] - u[S3][1]) + (u[S1][3] - u[S3][3]), N);
    udx = (from_right(u[S1][0]) - from_left(u[S1][0])) + (from_right(u[S1][2]) - from_left(u[S1][2]));
    udy = (from_right(u[S1][1]) - from_left(u[S1][1])) + (from_right(u[S1][3]) - from_left(u[S1][3]));
    n1[S2] = N[1];
    n3[S2] = N[3];
    // source and collision of row r - 3
    const Two h = two(c.hdxs);
    const Two Sx = fmr(nd0, h, fmr(n1[S2] - n1[S0], h, two(c.sbxs)));
    const Two Sy = fmr(nd2, h, fmr(n3[S2] - n3[S0], h, two(c.sbys)));
    nd0 = from_right(N[0]) - from_left(N[0]);
    nd2 = from_right(N[2]) - from_left(N[2]);
#pragma unroll
    for (int q = 0; q < 9 - kParked; ++q) w[q] = wide(f[S3][q]);
#pragma unroll
    for (int q = 9 - kParked; q < 9; ++q) {
      w[q] = wide(park[I & 1][q - (9 - kParked)][0]);
      park[I & 1][q - (9 - kParked)][0] = f[S1][q];
    }
    collide_v2(w, Sx, Sy, c.K);
#pragma unroll
    for (int q = 0; q < 9; ++q) narrow(w[q], out[q]);
    // what row r sends to rows r and r + 1
    f[S0][0] = g[0];
    f[S0][1] = from_left(g[1]);
    f[S0][3] = from_right(g[3]);
    f[S3][2] = g[2];
    f[S3][5] = from_left(g[5]);
    f[S3][6] = from_right(g[6]);
  }

  static __device__ __forceinline__ void moment(const Two v[9], Two &mx, Two &my) {
    const Two d57 = v[5] - v[7], d68 = v[6] - v[8];
    mx = (v[1] - v[3]) + (d57 - d68);
    my = (v[2] - v[4]) + (d57 + d68);
  }
  // pair_add() on two nodes
  static __device__ __forceinline__ void pair_add2(Two h, Two l, Two d, Two &oh, Two &ol) {
    const Two s = h + d;
    const Two bp = s - h;
    const Two e = (h - (s - bp)) + (d - bp);
    ol = l + e;
    oh = s;
  }
};

// ------------------------------------------------------------------ kernels
// T iterations per launch.  Block: T warps on one strip; warp t advances
// iteration t, taking its rows from warp t - 1 through shared memory (warp 0
// from global memory), the last one storing.  A strip of 64 columns loses three
// on each side per iteration: kOut<T> columns are stored.
template <int I>
struct Slot {
  static constexpr int value = I;
};
__device__ __forceinline__ void store_raw(float *p, Two a) { *reinterpret_cast<float2 *>(p) = make_float2(a.x, a.y); }
__device__ __forceinline__ void store_raw(__half *p, uint32_t a) { *reinterpret_cast<uint32_t *>(p) = a; }

template <int BYTES>
__device__ __forceinline__ void copy_async(void *dst, const void *src) {
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src));
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(BYTES));
}

// A row on its way to a warp: the strip's populations by lane, u of the row by
// node (node i at u_slot(i): a lane reads two neighbouring nodes, and the swap
// in every other eight keeps its reads of either clear of bank conflicts).
template <class Pr>
struct ColumnRow {
  typename RawOf<Pr>::type g[9][32];
  float4 u[64];
};
__device__ __forceinline__ int u_slot(int i) { return i ^ ((i >> 3) & 1); }
// rows of each warp's ring: the first warp's fill ahead from global memory, the
// others' from the warp before, two rows (one block barrier) at a time
constexpr int kColumnRing = 4;

template <class Pr, int T>
__global__ void __launch_bounds__(32 * T, 12 / T) step_column_kernel(const Params P, const Coef<float> c,
                                                                     const StepPtrs S, const ColumnRegion R) {
  using Raw = typename RawOf<Pr>::type;
  using gs = typename Pr::gs;
  __shared__ ColumnRow<Pr> rows[T][kColumnRing];
  constexpr int kP = Column<Pr>::kParked > 0 ? Column<Pr>::kParked : 1;
  __shared__ Raw parked[T][2][kP][32];
  const int lane = threadIdx.x % 32, t = threadIdx.x / 32;
  int xo, ya, yb;
  column_block<T>(R, (int)blockIdx.x, xo, ya, yb);
  const int xc = xo - kColumnHalo<T> + 2 * lane;  // this lane's columns xc, xc + 1
  const bool mine = column_mine<T>(R, lane, xc);
  const size_t plane = plane_of(P);
  // (without wrap, lanes past the last node repeat the last pair; where that
  // pair is the last node and a word of the row's padding, which holds
  // anything, the node stands for both)
  const int xl = column_pair(P, R, xc);
  const bool pad = xl == P.nx - 1;
  const bool pads = __any_sync(kAll, pad);
  const gs *gin = (const gs *)S.g_in + xl;
  // u is copied by whole lines: this lane brings nodes lane and lane + 32
  const float4 *uin = (const float4 *)S.u_in + column_node(P, R, xo - kColumnHalo<T> + lane);
  const int u32 = column_node(P, R, xo - kColumnHalo<T> + lane + 32) - column_node(P, R, xo - kColumnHalo<T> + lane);

  Column<Pr> col;
  col.clear();
#pragma unroll
  for (int k = 0; k < 2 * kP; ++k) narrow(two(0.0f), parked[t][k / kP][k % kP][lane]);
  const int r0 = ya - 3 * T, n = column_steps<T>(ya, yb);
  // warp t is 5 rows behind warp t - 1 (3 that its new rows lag, 2 of the ring)
  auto fetch = [&](int j) {
    if (j < n) {
      ColumnRow<Pr> &w = rows[0][j & (kColumnRing - 1)];
      const gs *p = gin + (size_t)column_row(P, R, r0 + j) * P.pitch;
#pragma unroll
      for (int q = 0; q < 9; ++q) copy_async<sizeof(Raw)>(&w.g[q][lane], p + q * plane);
      const float4 *pu = uin + (size_t)column_row(P, R, r0 + j) * P.pitch;
      copy_async<16>(&w.u[u_slot(lane)], pu);
      copy_async<16>(&w.u[u_slot(lane + 32)], pu + u32);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  Two uk[4] = {two(0.0f), two(0.0f), two(0.0f), two(0.0f)};
  // step j: warp t's row r0 + j - 5 t
  auto step = [&](auto slot, int j) {
    constexpr int I = decltype(slot)::value;
    if (t == 0) {
      __syncwarp();  // every lane has read the row whose slot is filled next
      fetch(j + kColumnRing - 1);
      asm volatile("cp.async.wait_group %0;" ::"n"(kColumnRing - 1) : "memory");
      __syncwarp();
    }
    const ColumnRow<Pr> &w = rows[t][(j + 2 * (t & 1)) & (kColumnRing - 1)];
    Raw g[9], out[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) g[q] = w.g[q][lane];
    if (pads) {
#pragma unroll
      for (int q = 0; q < 9; ++q)
        if (pad) g[q] = first_of(g[q]);
    }
    col.template step<I>(P, c, g, uk, out, (Raw(*)[kP][32]) & parked[t][0][0][lane]);
    // u(t) of this row, for the next step
    const float4 p0 = w.u[u_slot(2 * lane)], p1 = w.u[u_slot(2 * lane + 1)];
    uk[0] = two(p0.x, p1.x);
    uk[1] = two(p0.y, p1.y);
    uk[2] = two(p0.z, p1.z);
    uk[3] = two(p0.w, p1.w);
    const Two *u = col.u[(I + 1) & 3];
    if (T > 1 && t < T - 1) {
      ColumnRow<Pr> &o = rows[t + 1][(j + 2 * (t & 1)) & (kColumnRing - 1)];
#pragma unroll
      for (int q = 0; q < 9; ++q) o.g[q][lane] = out[q];
      o.u[u_slot(2 * lane)] = make_float4(lo(u[0]), lo(u[1]), lo(u[2]), lo(u[3]));
      o.u[u_slot(2 * lane + 1)] = make_float4(hi(u[0]), hi(u[1]), hi(u[2]), hi(u[3]));
    } else {
      const int row = column_stored<T>(r0, j);
      if (mine && row >= ya && row < yb) {
        const size_t o = (size_t)row * P.pitch + xc;
        gs *go = (gs *)S.g_out + o;
#pragma unroll
        for (int q = 0; q < 9; ++q) store_raw(go + q * plane, out[q]);
        asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"((float4 *)S.u_out + o),
                     "f"(lo(u[0])), "f"(lo(u[1])), "f"(lo(u[2])), "f"(lo(u[3])), "f"(hi(u[0])), "f"(hi(u[1])),
                     "f"(hi(u[2])), "f"(hi(u[3]))
                     : "memory");
      }
    }
    if constexpr (T > 1 && I % 2 == 1) __syncthreads();
  };
  if (t == 0) {
    for (int j = 0; j < kColumnRing - 1; ++j) fetch(j);
  } else {
    // (the rows before the first ones handed over)
    for (int k = 0; k < kColumnRing; ++k) {
#pragma unroll
      for (int q = 0; q < 9; ++q) narrow(two(0.0f), rows[t][k].g[q][lane]);
      rows[t][k].u[lane] = rows[t][k].u[lane + 32] = make_float4(0, 0, 0, 0);
    }
  }
  if constexpr (T > 1) __syncthreads();
  for (int j = 0; j < n; j += 4) {
    step(Slot<0>{}, j);
    step(Slot<1>{}, j + 1);
    if (j + 2 >= n) break;
    step(Slot<2>{}, j + 2);
    step(Slot<3>{}, j + 3);
  }
}

// strips and segments of a region on this device
template <class Pr, int T>
ColumnRegion column_region(int x0, int x1, int y0, int y1, int wrap) {
  static const int resident = [] {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, step_column_kernel<Pr, T>, 32 * T, 0);
    return (sms > 0 ? sms : 1) * (per > 0 ? per : 1);
  }();
  return column_split<T>(x0, x1, y0, y1, wrap, resident);
}

template <class Pr, int T>
cudaError_t launch_column(const Params &P, const StepPtrs &S, const ColumnRegion &R, cudaStream_t st) {
  const int nseg = (R.y1 - R.y0 + R.seg - 1) / R.seg;
  step_column_kernel<Pr, T><<<R.nstrip * nseg, 32 * T, 0, st>>>(
      P, make_coef<typename Pr::gs, typename Pr::real>(P), S, R);
  return cudaGetLastError();
}

// a periodic lattice whole, T iterations a launch
template <class Pr, int T>
cudaError_t launch_column_periodic(const Params &P, const StepPtrs &S, cudaStream_t st) {
  return launch_column<Pr, T>(P, S, column_region<Pr, T>(0, P.nx, 0, P.ny, 1), st);
}

// One iteration of any lattice: the nodes of the interior tiles of C through
// the columns, the frame tiles as in launch_step.
template <class C>
cudaError_t launch_step_column(const Params &P, const StepPtrs &S, cudaStream_t st) {
  using Pr = typename C::PrT;
  const int ntx = (P.nx + C::TX - 1) / C::TX, nty = (P.ny + C::TY - 1) / C::TY;
  int a_lo, a_hi, b_lo, b_hi;
  interior_range(P.nx, P.ny, C::TX, C::TY, a_lo, a_hi, b_lo, b_hi);
  const int ni = a_hi - a_lo, nj = b_hi - b_lo;
  const int nedge = ntx * nty - ni * nj;
  const bool beside = fork_begin(S, st, ni > 0 && nj > 0 && nedge > 0);
  if (beside) launch_edge<C>(P, S, nedge, ntx, a_lo, a_hi, b_lo, b_hi, S.fork->side);
  if (ni > 0 && nj > 0)
    launch_column<Pr, 1>(P, S, column_region<Pr, 1>(a_lo * C::TX, a_hi * C::TX, b_lo * C::TY, b_hi * C::TY, 0), st);
  if (!beside) launch_edge<C>(P, S, nedge, ntx, a_lo, a_hi, b_lo, b_hi, st);
  fork_end(S, st, beside);
  return cudaGetLastError();
}

}  // namespace lbs
