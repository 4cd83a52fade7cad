// Host-side bounds audit of the warp columns' index arithmetic (the column
// section of paper_2502_00920_gb300/csrc/lbs_tiles.h, which step_column_kernel
// takes its strips, segments, rows and columns from).  For one and two
// iterations per launch, over periodic lattices (rows and columns wrap) and
// interior regions of walled ones, odd widths and padded rows among them:
//   - every row, pair of populations and displacement record read lies in the
//     state's allocation, the pairs on even columns; a pair may hold one word
//     of a row's padding only where the kernel replaces it;
//   - within 3 T nodes of what a block stores, a wrapped read is the node
//     modulo the lattice and an unwrapped one the node itself;
//   - the steps reach every row of the segment, and every node of the region
//     is stored exactly once;
//   - offsets are exact on lattices of 2^31 nodes and more (the largest sizes
//     that are accepted), where a plane's elements do not fit 32 bits.
// Prints "ok <cases>" and exits 0, or lists the first failures and exits 1.
#include <stdio.h>

#include <string>
#include <vector>

#include "lbs_tiles.h"

using namespace lbs;

namespace {

struct Lat {
  int nx, ny, pitch, per_x, per_y;
};

long g_fail = 0, g_cases = 0;
std::string g_ctx;
#define CHECK(cond, ...)                                                             \
  do {                                                                               \
    if (!(cond) && g_fail++ < 25) fprintf(stderr, "FAIL [%s] %s\n", g_ctx.c_str(), #cond); \
  } while (0)

int64_t mod(int64_t a, int64_t n) { return (a % n + n) % n; }

// one block: `stored` (if any) counts the stores of each node
template <int T>
void block(const Lat &P, const ColumnRegion &R, int b, std::vector<int> *stored, bool ends_only) {
  // of the nine planes of g and of u, in elements, from 64-bit products
  const uint64_t plane = (uint64_t)P.ny * (uint64_t)P.pitch;
  CHECK((uint64_t)plane_of(P) == plane);
  int xo, ya, yb;
  column_block<T>(R, b, xo, ya, yb);
  CHECK(xo >= R.x0 && xo < R.x1 && ya >= R.y0 && ya < yb && yb <= R.y1);
  const int r0 = ya - 3 * T, n = column_steps<T>(ya, yb);
  for (int j = 0; j < n; ++j) {
    if (ends_only && j > 2 && j < n - 3) continue;
    const int row = column_row(P, R, r0 + j);
    CHECK(row >= 0 && row < P.ny);
    if (r0 + j >= ya - 3 * T && r0 + j < yb + 3 * T)
      CHECK(row == (R.wrap ? mod(r0 + j, P.ny) : (r0 + j < P.ny ? r0 + j : P.ny - 1)));
    for (int lane = 0; lane < 32; ++lane) {
      const int xc = xo - kColumnHalo<T> + 2 * lane, xl = column_pair(P, R, xc);
      CHECK(xl >= 0 && xl % 2 == 0 && xl < P.nx && xl + 1 < P.pitch);
      // (the kernel stands the node in for the padding where xl is the last node)
      CHECK(xl + 1 < P.nx || xl == P.nx - 1);
      for (int q = 0; q < 9; q += 8) {
        const uint64_t o = (uint64_t)(q * plane_of(P)) + (uint64_t)((size_t)row * P.pitch) + (uint64_t)xl;
        CHECK(o == (uint64_t)q * plane + (uint64_t)row * (uint64_t)P.pitch + (uint64_t)xl && o + 1 < 9 * plane);
      }
      for (int k = 0; k < 64; k += 32) {
        const int x = xo - kColumnHalo<T> + lane + k, c = column_node(P, R, x);
        CHECK(c >= 0 && c < P.nx);
        CHECK(c == (R.wrap ? mod(x, P.nx) : (x < P.nx ? x : P.nx - 1)));
      }
      if (column_mine<T>(R, lane, xc)) {
        // the pair it stores and the three nodes per iteration around it
        CHECK(xc % 2 == 0 && xc >= R.x0 && xc + 1 < R.x1 && xc + 1 < P.nx && xl == xc);
        CHECK(2 * lane >= 3 * T && 2 * lane + 1 < 64 - 3 * T);
        if (!R.wrap) CHECK(xc - 3 * T >= 0 && xc + 1 + 3 * T < P.nx && ya - 3 * T >= 0 && yb - 1 + 3 * T < P.ny);
      }
    }
  }
  int last = ya - 1;
  for (int j = 0; j < n + n % 2; ++j) {  // (steps go in pairs)
    const int row = column_stored<T>(r0, j);
    if (row < ya || row >= yb) continue;
    CHECK(row == last + 1);
    last = row;
    if (!stored) continue;
    for (int lane = 0; lane < 32; ++lane) {
      const int xc = xo - kColumnHalo<T> + 2 * lane;
      if (column_mine<T>(R, lane, xc) && xc + 1 < P.nx)
        for (int k = 0; k < 2; ++k) (*stored)[(size_t)row * P.nx + xc + k] += 1;
    }
  }
  CHECK(last == yb - 1);
}

template <int T>
void region(const Lat &P, int x0, int x1, int y0, int y1, int wrap, int resident) {
  char buf[160];
  snprintf(buf, sizeof buf, "%d iterations, lattice %dx%d, region [%d, %d) x [%d, %d), %d resident", T, P.nx, P.ny, x0,
           x1, y0, y1, resident);
  g_ctx = buf;
  const ColumnRegion R = column_split<T>(x0, x1, y0, y1, wrap, resident);
  const int nseg = (y1 - y0 + R.seg - 1) / R.seg;
  CHECK(R.seg >= 1 && (int64_t)R.nstrip * nseg < INT32_MAX);
  const bool large = (int64_t)P.nx * P.ny > (int64_t)1 << 24;
  if (large) {
    for (int s : {0, R.nstrip - 1})
      for (int g : {0, nseg - 1}) block<T>(P, R, g * R.nstrip + s, nullptr, true);
  } else {
    std::vector<int> stored((size_t)P.nx * P.ny, 0);
    for (int b = 0; b < R.nstrip * nseg; ++b) block<T>(P, R, b, &stored, false);
    for (int y = 0; y < P.ny; ++y)
      for (int x = 0; x < P.nx; ++x)
        CHECK(stored[(size_t)y * P.nx + x] == (x >= x0 && x < x1 && y >= y0 && y < y1 ? 1 : 0));
  }
  ++g_cases;
}

Lat lattice(int nx, int ny, int per) { return Lat{nx, ny, (nx + 31) / 32 * 32, per, per}; }

void periodic(int nx, int ny, int resident) {
  const Lat P = lattice(nx, ny, 1);
  if (!column_wraps(P)) return;
  region<1>(P, 0, nx, 0, ny, 1, resident);
  region<2>(P, 0, nx, 0, ny, 1, resident);
}

// the interior of a walled (or odd) lattice, as launch_step_column takes it
void interior(int nx, int ny, int resident) {
  const Lat P = lattice(nx, ny, 0);
  int a_lo, a_hi, b_lo, b_hi;
  interior_range(nx, ny, 32, 16, a_lo, a_hi, b_lo, b_hi);
  if (a_hi > a_lo && b_hi > b_lo) region<1>(P, a_lo * 32, a_hi * 32, b_lo * 16, b_hi * 16, 0, resident);
}

}  // namespace

int main() {
  for (int resident : {152 * 6, 152 * 12, 7})
    for (int nx : {128, 130, 154, 156, 158, 168, 170, 224, 260, 390})
      for (int ny : {64, 65, 71, 100, 177, 333}) periodic(nx, ny, resident);
  for (int nx : {67, 70, 96, 97, 99, 100, 131, 160, 161, 193, 227, 500})
    for (int ny : {35, 50, 51, 60, 101, 130, 300}) interior(nx, ny, 152 * 12);
  // 2^31 nodes and more, up to the 2^34 that are accepted
  const int large[][2] = {{46340, 46340}, {46342, 46342}, {46400, 46400}, {1 << 16, 1 << 15}, {128, 1 << 25},
                          {1 << 25, 64}, {1 << 16, 1 << 16}, {1 << 17, 1 << 17}};
  for (auto &s : large) {
    periodic(s[0], s[1], 152 * 6);
    interior(s[0] - 1, s[1], 152 * 12);
  }
  if (g_fail) {
    fprintf(stderr, "%ld failures\n", g_fail);
    return 1;
  }
  printf("ok %ld\n", g_cases);
  return 0;
}
