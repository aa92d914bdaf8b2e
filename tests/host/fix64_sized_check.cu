// Host-side check that the fixed-point FP64 hopping sum (wd_fix64.cuh) takes
// 18-real links of any size from 2^-64 to 2^64, none of them sent to the FP64
// chain, and is no less exact than the chain on them (rms relative to the
// site's rms component, against long double); that links of different sizes on
// one site are summed right; and that infinities, NaN and larger links are
// refused.  Prints "OK <largest ratio>".
#define main fix64_check_main
#include "fix64_check.cu"
#undef main

// sizes: the scale of each hop's link
template <int S>
static bool sized(double lo, double hi, int n, double& ef, double& ed) {
  double sf = 0, sd = 0;
  for (int k = 0; k < n; k++) {
    Site st = {};
    fix_begin(st.fx);
    auto hop1 = [&](auto MU, auto SG, auto FW) {
      constexpr int mu = decltype(MU)::value, s = decltype(SG)::value;
      constexpr bool fwd = decltype(FW)::value;
      cx<double> h[6];
      for (auto& v : h) v = {gau(), gau()};
      double u[18];
      su3(u, uni() < 0.5 ? 0.3 : 3.0);
      const double sc = std::exp2(lo + (hi - lo) * uni());
      for (auto& v : u) v *= sc;
      const bool flip = mu == 3 && uni() < 0.5;
      fix_hop<s, fwd, 18, true>(st.fx, mu, h, u, flip, false);
      cx<double> ud[9];
      cx<ld> ul[9];
      for (int j = 0; j < 9; j++) ud[j] = {u[2 * j], u[2 * j + 1]}, ul[j] = {u[2 * j], u[2 * j + 1]};
      chain<double, mu, s, fwd>(st.dp, h, ud, flip, false);
      chain<ld, mu, s, fwd>(st.ex, h, ul, flip, false);
    };
    auto dir = [&](auto MU) {
      hop1(MU, std::integral_constant<int, S>(), std::true_type());
      hop1(MU, std::integral_constant<int, -S>(), std::false_type());
    };
    dir(std::integral_constant<int, 0>());
    dir(std::integral_constant<int, 1>());
    dir(std::integral_constant<int, 2>());
    dir(std::integral_constant<int, 3>());
    if (!fix_ok(st.fx)) return false;
    double nn = 0, f = 0, d = 0;
    for (int j = 0; j < 12; j++) {
      nn += (double)(st.ex[j].r * st.ex[j].r + st.ex[j].i * st.ex[j].i);
      const ld a = fix_double(st.fx.r[j], st.fx.E) - st.ex[j].r, b = fix_double(st.fx.i[j], st.fx.E) - st.ex[j].i;
      const ld p = st.dp[j].r - st.ex[j].r, q = st.dp[j].i - st.ex[j].i;
      f += (double)(a * a + b * b), d += (double)(p * p + q * q);
    }
    sf += f / nn, sd += d / nn;
  }
  ef = std::sqrt(sf / n), ed = std::sqrt(sd / n);
  return true;
}

// one link real v at hop `at`, the others SU(3): whether the site is refused
static bool refused(int at, int where, double v, double h0) {
  FixSite s;
  fix_begin(s);
  for (int k = 0; k < 8; k++) {
    cx<double> h[6];
    for (auto& c : h) c = k == at ? cx<double>{h0, -h0} : cx<double>{gau(), gau()};
    double u[18];
    su3(u, 0.3);
    if (k == at) u[where] = v;
    fix_hop<1, true, 18, true>(s, k / 2, h, u, false, false);
  }
  return !fix_ok(s);
}

int main() {
  double worst = 0;
  const double range[][2] = {{0.029, 0.029}, {0.2, 0.2}, {-0.1, 0.6}, {3, 3.3}, {-3.3, -3}, {-8, -7}, {-6, 6},
                             {-30, 30}, {62, 63}, {-63, -62}};
  for (auto& r : range) {
    double ef, ed, e2, d2;
    if (!sized<1>(r[0], r[1], 1000, ef, ed) || !sized<-1>(r[0], r[1], 1000, e2, d2))
      return printf("FAIL: links of 2^%g to 2^%g refused\n", r[0], r[1]), 1;
    printf("links 2^%g to 2^%g: fixed %.3g chain %.3g\n", r[0], r[1], ef, ed);
    worst = std::fmax(worst, std::fmax(ef / ed, e2 / d2));
  }
  if (worst > 1) return printf("FAIL %.3f\n", worst), 1;
  for (int at = 0; at < 8; at++)
    for (int w = 0; w < 18; w++)
      for (double h0 : {0.0, -0.0, 1.0})
        for (double v : {(double)INFINITY, -(double)INFINITY, (double)NAN, 1e200, -1e25})
          if (!refused(at, w, v, h0)) return printf("FAIL: real %d = %g taken\n", w, v), 1;
  // a link that vanishes adds nothing
  FixSite s;
  fix_begin(s);
  for (int k = 0; k < 8; k++) {
    cx<double> h[6];
    for (auto& c : h) c = {k == 2 ? 1.0 : 3.0, 0.5};
    double u[18] = {};
    if (k == 2) u[0] = u[8] = u[16] = 1;
    fix_hop<1, true, 18, true>(s, k / 2, h, u, false, false);
  }
  if (!fix_ok(s) || fix_double(s.r[0], s.E) != 1.0 || fix_double(s.i[0], s.E) != 0.5)
    return printf("FAIL: vanishing links\n"), 1;
  printf("OK %.3f\n", worst);
  return 0;
}
