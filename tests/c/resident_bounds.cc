// Host-side bounds audit of what the frame, batch and resident kernels take
// from paper_2502_00920_gb300/csrc/lbs_tiles.h beside tile_bounds.cc's part.
//
// Streaming sides and wall masks (stream_sides, crosses_x, crosses_y: the
// gather of a frame or resident tile and the wall rules): on every node of
// small lattices with every combination of periodic and walled axes, a
// direction's bit is set exactly where its source x - e_q lies beyond that
// axis' wall, the source read is that node (wrapped) where it is not, and a
// lattice node in any case.
//
// Resident launches (resident_kernel) on every tile shape the library
// compiles, over ragged and degenerate lattices, both wall readings, three
// iterations of one launch:
//   - every thread's entry, ring and tap index lies in its array, and every
//     shared entry read was written in the same iteration;
//   - every global read hits a lattice node stored by the iteration before,
//     every node is stored once per iteration (and u by the last);
//   - side-array entries are written once per iteration, exactly those of the
//     wall (and inner) nodes, and read only where the iteration before wrote;
//   - offsets fit the kernel's 32-bit arithmetic on the largest lattices.
// Prints "ok <cases>" and exits 0, or lists the first failures and exits 1.
#include <stdio.h>

#include <string>
#include <vector>

#include "lbs_tiles.h"

using namespace lbs;

namespace {

struct Lat {
  int nx, ny, pitch, per_x, per_y, blen, extrap;
};

long g_fail = 0, g_cases = 0;
std::string g_ctx;
void fail(const char *what, int a, int b, int c) {
  if (g_fail++ < 25) fprintf(stderr, "FAIL [%s] %s (%d, %d, %d)\n", g_ctx.c_str(), what, a, b, c);
}
#define CHECK(cond, a, b, c)             \
  do {                                   \
    if (!(cond)) fail(#cond, a, b, c);   \
  } while (0)

bool inside(const Lat &P, int x, int y) { return x >= 0 && x < P.nx && y >= 0 && y < P.ny; }

// D2Q9 as the paper's Tab. 1 lists it
const int EX[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, EY[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};

// the nine sources of a node as the kernels form them
void sources(const Lat &P, int x, int y, int sx[9], int sy[9]) {
  int xb, xf, yb, yf;
  stream_sides(x, P.nx, P.per_x, xb, xf);
  stream_sides(y, P.ny, P.per_y, yb, yf);
  for (int q = 0; q < 9; ++q) {
    sx[q] = ex(q) > 0 ? xb : (ex(q) < 0 ? xf : x);
    sy[q] = ey(q) > 0 ? yb : (ey(q) < 0 ? yf : y);
  }
}

void sides_and_masks(const Lat &P) {
  for (int y = 0; y < P.ny; ++y)
    for (int x = 0; x < P.nx; ++x) {
      int xw, yw, sx[9], sy[9];
      walls_of(P, x, y, xw, yw);
      sources(P, x, y, sx, sy);
      for (int q = 0; q < 9; ++q) {
        CHECK(ex(q) == EX[q] && ey(q) == EY[q], q, 0, 0);
        const int tx = x - EX[q], ty = y - EY[q];
        const bool ox = !P.per_x && (tx < 0 || tx >= P.nx), oy = !P.per_y && (ty < 0 || ty >= P.ny);
        CHECK(((crosses_x(xw) >> q) & 1) == (unsigned)ox, x, y, q);
        CHECK(((crosses_y(yw) >> q) & 1) == (unsigned)oy, x, y, q);
        CHECK(inside(P, sx[q], sy[q]), x, y, q);
        if (!ox && !oy) CHECK(sx[q] == (tx + P.nx) % P.nx && sy[q] == (ty + P.ny) % P.ny, x, y, q);
      }
    }
  ++g_cases;
}

size_t side_values(const Lat &P) { return (size_t)(P.extrap ? 2 : 1) * 4 * P.blen * 4; }

// the side entries that the nodes of a lattice fill
std::vector<int> side_wanted(const Lat &P) {
  std::vector<int> w(side_values(P) / 4, 0);
  for (int y = 0; y < P.ny; ++y)
    for (int x = 0; x < P.nx; ++x) {
      const bool l = !P.per_x && x == 0, r = !P.per_x && x == P.nx - 1, b = !P.per_y && y == 0, t = !P.per_y && y == P.ny - 1;
      if (l) w[side_entry(P, 0, kLeft, y) / 4] += 1;
      if (r) w[side_entry(P, 0, kRight, y) / 4] += 1;
      if (b) w[side_entry(P, 0, kBottom, x) / 4] += 1;
      if (t) w[side_entry(P, 0, kTop, x) / 4] += 1;
      if (!P.extrap) continue;
      if (!P.per_x && x == 1) w[side_entry(P, 1, kLeft, y) / 4] += 1;
      if (!P.per_x && x == P.nx - 2) w[side_entry(P, 1, kRight, y) / 4] += 1;
      if (!P.per_y && y == 1) w[side_entry(P, 1, kBottom, x) / 4] += 1;
      if (!P.per_y && y == P.ny - 2) w[side_entry(P, 1, kTop, x) / 4] += 1;
    }
  return w;
}

// one launch of resident_kernel over the whole lattice
template <class C>
void resident(const Lat &P, int iterations) {
  const int ntx = (P.nx + C::TX - 1) / C::TX, nty = (P.ny + C::TY - 1) / C::TY;
  const int64_t plane = (int64_t)P.ny * P.pitch;
  CHECK(9 * plane <= INT32_MAX, P.nx, P.ny, 0);
  CHECK(C::OWN + C::NRING == C::R2W * C::R2H && C::R2W * C::R2H <= C::NT, C::NT, 0, 0);
  CHECK(C::R1W * C::R1H <= C::NT && C::OWN <= C::NT, C::NT, 0, 0);
  const std::vector<int> wanted = side_wanted(P);
  std::vector<int> g(P.nx * P.ny, 0);  // stores of each node in the iteration before (the initial state: 1)
  g.assign(g.size(), 1);
  std::vector<int> side = wanted, u_stored(P.nx * P.ny, 0);
  for (int it = 0; it < iterations; ++it) {
    std::vector<int> g_new(g.size(), 0), side_new(side.size(), 0);
    for (int tile = 0; tile < ntx * nty; ++tile) {
      const int x0 = tile % ntx * C::TX, y0 = tile / ntx * C::TY;
      std::vector<int> su(C::R2W * C::R2H, 0), sn(C::R1W * C::R1H, 0);
      auto side_read = [&](int layer, int e, int pos) {
        const size_t o = side_entry(P, layer, e, pos) / 4;
        CHECK(o < side.size() && side[o] == 1, layer, e, pos);
      };
      // phase 1: u on R2
      for (int e = 0; e < C::NT; ++e) {
        if (e >= C::OWN + C::NRING) continue;
        int rx, ry;
        resident_pos<C>(e, rx, ry);
        CHECK(rx >= 0 && rx < C::R2W && ry >= 0 && ry < C::R2H, rx, ry, e);
        CHECK((e < C::OWN) == (rx >= 2 && rx < C::TX + 2 && ry >= 2 && ry < C::TY + 2), rx, ry, e);
        int x = x0 - 2 + rx, y = y0 - 2 + ry;
        const bool own = e < C::OWN && x < P.nx && y < P.ny;
        const bool in = locate(P, x, y);
        CHECK(!own || (in && x == x0 - 2 + rx && y == y0 - 2 + ry), x, y, e);
        if (!in) continue;
        CHECK(inside(P, x, y) && g[y * P.nx + x] == 1, x, y, e);
        int sx[9], sy[9], xw, yw;
        sources(P, x, y, sx, sy);
        for (int q = 0; q < 9; ++q) CHECK(inside(P, sx[q], sy[q]) && g[sy[q] * P.nx + sx[q]] == 1, x, y, q);
        walls_of(P, x, y, xw, yw);
        for (int w = 0; w < 2; ++w) {
          const int ed = w == 0 ? xw : yw, pos = w == 0 ? y : x;
          if (ed < 0) continue;
          side_read(0, ed, pos);
          if (!P.extrap) continue;
          int xi, yi;
          inner_node(ed, x, y, xi, yi);
          CHECK(inside(P, xi, yi) && g[yi * P.nx + xi] == 1, xi, yi, ed);
          side_read(1, ed, pos);
        }
        su[ry * C::R2W + rx] += 1;
      }
      for (int v : su) CHECK(v <= 1, v, 0, 0);
      // phase 2: N on R1
      for (int e = 0; e < C::NT; ++e) {
        const int rx = e % C::R1W, ry = e / C::R1W;
        int gx = x0 - 1 + rx, gy = y0 - 1 + ry;
        if (!(e < C::R1W * C::R1H && locate(P, gx, gy))) continue;
        int xa, xb, ya, yb;
        bool onex, oney;
        fd_taps<true>(P, rx + 1, ry + 1, gx, gy, xa, xb, ya, yb, onex, oney);
        const int taps[4] = {(ry + 1) * C::R2W + xa, (ry + 1) * C::R2W + xb, ya * C::R2W + rx + 1, yb * C::R2W + rx + 1};
        for (int t : taps) CHECK(t >= 0 && t < C::R2W * C::R2H && su[t] == 1, gx, gy, t);
        sn[e] = 1;
        if (r1_own_node<C>(P, x0, y0, rx, ry) && (on_wall(P, gx, gy) || P.extrap)) {
          int xw, yw;
          walls_of(P, gx, gy, xw, yw);
          if (xw >= 0) side_new[side_entry(P, 0, xw, gy) / 4] += 1;
          if (yw >= 0) side_new[side_entry(P, 0, yw, gx) / 4] += 1;
          if (P.extrap) {
            int ee[4], pos[4];
            const int n = inner_entries(P, gx, gy, ee, pos);
            for (int k = 0; k < n; ++k) side_new[side_entry(P, 1, ee[k], pos[k]) / 4] += 1;
          }
        }
      }
      // phase 3: own nodes
      for (int e = 0; e < C::OWN; ++e) {
        int rx, ry;
        resident_pos<C>(e, rx, ry);
        const int x = x0 - 2 + rx, y = y0 - 2 + ry;
        if (x >= P.nx || y >= P.ny) continue;
        int xa, xb, ya, yb;
        bool onex, oney;
        fd_taps<true>(P, rx - 1, ry - 1, x, y, xa, xb, ya, yb, onex, oney);
        const int taps[4] = {(ry - 1) * C::R1W + xa, (ry - 1) * C::R1W + xb, ya * C::R1W + rx - 1, yb * C::R1W + rx - 1};
        for (int t : taps) CHECK(t >= 0 && t < C::R1W * C::R1H && sn[t] == 1, x, y, t);
        g_new[y * P.nx + x] += 1;
        if (it == iterations - 1) u_stored[y * P.nx + x] += 1;
      }
    }
    for (size_t i = 0; i < g_new.size(); ++i) CHECK(g_new[i] == 1, (int)i, g_new[i], it);
    for (size_t i = 0; i < side_new.size(); ++i) CHECK(side_new[i] == wanted[i], (int)i, side_new[i], it);
    g = g_new;
    side = side_new;
  }
  for (size_t i = 0; i < u_stored.size(); ++i) CHECK(u_stored[i] == 1, (int)i, u_stored[i], 0);
  ++g_cases;
}

template <int TX, int TY>
void shape(const std::vector<int> &sizes) {
  for (int nx : sizes)
    for (int ny : sizes)
      for (int per = 0; per < 4; ++per)
        for (int extrap = 0; extrap < 2; ++extrap) {
          Lat P{nx, ny, (nx + 31) / 32 * 32, per & 1, (per >> 1) & 1, nx > ny ? nx : ny, extrap};
          char buf[120];
          snprintf(buf, sizeof buf, "resident tile %dx%d, lattice %dx%d, periodic x %d y %d, linear %d", TX, TY, nx, ny,
                   P.per_x, P.per_y, extrap);
          g_ctx = buf;
          resident<ResGeom<TX, TY>>(P, 3);
        }
}

}  // namespace

int main() {
  for (int nx : {3, 4, 5, 8, 33})
    for (int ny : {3, 4, 6, 9, 17})
      for (int per = 0; per < 4; ++per) {
        Lat P{nx, ny, (nx + 31) / 32 * 32, per & 1, (per >> 1) & 1, nx > ny ? nx : ny, 0};
        g_ctx = "sides and masks";
        sides_and_masks(P);
      }
  // one node more and less than the tiles, the smallest lattices, strips
  const std::vector<int> sizes = {3, 4, 5, 7, 8, 9, 13, 14, 15, 16, 17, 29, 31, 32, 33, 34, 65};
  shape<8, 8>(sizes);    // double precision
  shape<16, 16>(sizes);
  shape<16, 8>(sizes);   // single precision, half-precision storage
  shape<32, 14>(sizes);
  // the longest strips of 152 tiles
  for (int n : {152 * 32, 152 * 32 - 5}) {
    g_ctx = "longest strips";
    resident<ResGeom<32, 14>>(Lat{n, 14, (n + 31) / 32 * 32, 0, 0, n, 0}, 1);
    resident<ResGeom<32, 14>>(Lat{3, 152 * 14, 32, 0, 1, 152 * 14, 1}, 1);
  }
  if (g_fail) {
    fprintf(stderr, "%ld failures\n", g_fail);
    return 1;
  }
  printf("ok %ld\n", g_cases);
  return 0;
}
