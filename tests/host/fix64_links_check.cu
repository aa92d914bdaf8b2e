// Host-side check of which links the fixed-point FP64 hopping sum
// (wd_fix64.cuh) takes: one that holds an infinity, a NaN or a value that does
// not fit sends its site to the FP64 chain whatever the neighbour it meets, a
// vanishing one included.  Prints "OK <hops>".
#include <cmath>
#include <cstdio>

#include "../../paper_0810_5365_gb300/csrc/wd_fix64.cuh"

using namespace wd;

// a zero neighbour (of either sign) at hop `at` of eight, with real `where` of its link set to v
template <int RC, int S, bool FWD>
static bool refused(int at, int where, double v, double zero) {
  FixSite s;
  fix_begin(s);
  for (int k = 0; k < 8; k++) {
    cx<double> h[6];
    for (int j = 0; j < 6; j++) h[j] = {0.3 + 0.1 * j, -0.2 * j};
    double u[RC];
    for (int j = 0; j < RC; j++) u[j] = j % 8 == 0 ? 1 : 0;  // the unit matrix
    if (k == at) {
      u[where] = v;
      for (auto& c : h) c = {zero, -zero};
    }
    fix_hop<S, FWD, RC>(s, k / 2, h, u, false, false);
  }
  return !fix_ok(s);
}

// a site all of whose neighbours vanish, and one of them does: exact zeros, and exact sums
template <int RC>
static bool zeros(double zero) {
  FixSite s, t;
  fix_begin(s), fix_begin(t);
  for (int k = 0; k < 8; k++) {
    cx<double> h[6];
    double u[RC];
    for (int j = 0; j < RC; j++) u[j] = j % 8 == 0 ? 1 : 0;
    for (auto& c : h) c = {zero, -zero};
    fix_hop<1, true, RC>(s, k / 2, h, u, k % 2, false);
    if (k == 3)
      for (int j = 0; j < 6; j++) h[j] = {1.0 + j, -0.5 * j};
    fix_hop<1, true, RC>(t, k / 2, h, u, false, false);
  }
  if (!fix_ok(s) || !fix_ok(t)) return false;
  for (int j = 0; j < 12; j++)
    if (fix_double(s.r[j], s.E) != 0 || fix_double(s.i[j], s.E) != 0) return false;
  for (int j = 0; j < 6; j++)
    if (std::fabs(fix_double(t.r[j], t.E) - (1.0 + j)) > 1e-15 * 8 ||
        std::fabs(fix_double(t.i[j], t.E) + 0.5 * j) > 1e-15 * 8)
      return false;
  return true;
}

template <int RC>
static int check() {
  int n = 0;
  for (int at = 0; at < 8; at++)
    for (int w = 0; w < RC; w++)
      for (double v : {(double)INFINITY, -(double)INFINITY, (double)NAN, 1e200})
        for (double z : {0.0, -0.0}) {
          n++;
          if (!refused<RC, 1, true>(at, w, v, z) || !refused<RC, -1, false>(at, w, v, z)) {
            printf("FAIL recon %d hop %d real %d value %g: taken\n", RC, at, w, v);
            return 0;
          }
        }
  for (double z : {0.0, -0.0})
    if (!zeros<RC>(z)) {
      printf("FAIL recon %d: zero neighbours\n", RC);
      return 0;
    }
  return n;
}

int main() {
  const int a = check<18>(), b = check<12>();
  if (!a || !b) return 1;
  printf("OK %d\n", a + b);
  return 0;
}
