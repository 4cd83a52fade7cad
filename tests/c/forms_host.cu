// The kernels' node functions (lbs_device.cuh) on the host: the source tensor
// from displacement differences, the collision and the wall rules, in both
// compute types.  Reads cases as numbers from standard input, writes one line
// of results per case; tests/test_node_forms.py holds them against the literal
// formulas.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include "lbs_device.cuh"

using namespace lbs;

static double next() {
  double v;
  if (scanf("%lf", &v) != 1) v = NAN;
  return v;
}

// model lam mu dx, then dxx dxy dyx dyy onex oney
template <class R>
static void stress() {
  Params P;
  memset(&P, 0, sizeof P);
  P.model = (int)next();
  P.lam = next();
  P.mu = next();
  P.inv_dx = 1.0 / next();
  P.cs = P.c = P.rho0 = 1.0;
  const Coef<R> c = make_coef<R, R>(P);
  const R dxx = (R)next(), dxy = (R)next(), dyx = (R)next(), dyy = (R)next();
  const bool onex = next() != 0, oney = next() != 0;
  R N[4];
  stress_n<R>(P, c, dxx, dxy, dyx, dyy, onex, oney, N);
  printf("%.17g %.17g %.17g %.17g\n", (double)N[0], (double)N[1], (double)N[2], (double)N[3]);
}

// omega sigma, nine populations, source
template <class R>
static void collision() {
  const double omega = next(), sigma = next();
  const CollideK<R> K = collide_k<R>((R)omega, (R)sigma, R(1));
  R f[9];
  for (R &v : f) v = (R)next();
  const R s = sizeof(R) == 8 ? K.s9 : R(1);  // (as Coef's idxs and sbxs scale it)
  const R Sx = (R)next() * s, Sy = (R)next() * s;
  collide<R>(f, Sx, Sy, K);
  for (int q = 0; q < 9; ++q) printf("%.17g ", (double)f[q]);
  printf("\n");
}

// xw yw, the four edges' types and prescribed values, 1 / cs^2, c / cs^2, wn,
// nine post-collision populations; writes the populations the rules supply (0
// where they leave what streamed in)
template <class R>
static void walls() {
  Params P;
  memset(&P, 0, sizeof P);
  const int xw = (int)next(), yw = (int)next();
  for (int &t : P.etype) t = (int)next();
  R sev[kEdgeEntries][2];
  for (int e = 0; e < 4; ++e)
    for (int a = 0; a < 2; ++a) sev[e][a] = (R)next();
  // a corner's entry is filled where both its walls are Dirichlet (edge_entry)
  for (int i = 4; i < kEdgeEntries; ++i) {
    const int ex = kLeft + (i & 1), ey = kBottom + ((i >> 1) & 1);
    const bool both = P.etype[ex] == LBS_DIRICHLET && P.etype[ey] == LBS_DIRICHLET;
    for (int a = 0; a < 2; ++a) sev[i][a] = both ? R(0.5) * (sev[ex][a] + sev[ey][a]) : (R)NAN;
  }
  const R ics2 = (R)next(), cj = (R)next();
  R wn[4], g0[9], f[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  for (R &v : wn) v = (R)next();
  for (R &v : g0) v = (R)next();
  wall_rules_own<R>(P, xw, yw, sev, ics2, cj, wn, g0, f);
  for (int q = 0; q < 9; ++q) printf("%.17g ", (double)f[q]);
  printf("\n");
}

int main(int argc, char **argv) {
  if (argc != 4) return 2;
  const bool wide = !strcmp(argv[1], "double");
  for (int n = atoi(argv[3]); n > 0; --n) {
    if (!strcmp(argv[2], "stress")) wide ? stress<double>() : stress<float>();
    else if (!strcmp(argv[2], "collision")) wide ? collision<double>() : collision<float>();
    else wide ? walls<double>() : walls<float>();
  }
  return 0;
}
