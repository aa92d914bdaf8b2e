// Host-side check that the fixed-point FP64 hopping sum (wd_fix64.cuh) gives
// every component of a site the bits that the FP64 chain gives it, whatever
// its size beside the others: sites whose links do not mix the colours
// (diagonal, or nearly), with one colour or one spin of the half spinors
// smaller than the rest by a factor.  The components' errors against long
// double (rms over sites, where a site that fix_ok or fix_resolved refuses
// takes the chain's value) are compared with the chain's.  Also: products near
// the end of the sums' range.  Prints "OK <largest ratio>".
#define main fix64_check_main
#include "fix64_check.cu"
#undef main

// ratio of the two errors, the largest over the components; refused: share of sites
template <int RC, int S>
static double ratio(int form, double f, int n, double& refused) {
  double ef[12] = {}, ed[12] = {};
  int no = 0;
  for (int k = 0; k < n; k++) {
    Site st = {};
    fix_begin(st.fx);
    auto hop1 = [&](auto MU, auto SG, auto FW) {
      constexpr int mu = decltype(MU)::value, s = decltype(SG)::value;
      constexpr bool fwd = decltype(FW)::value;
      cx<double> h[6];
      for (int j = 0; j < 6; j++) {
        const double sc = (form == 1 ? j >= 3 : j % 3 == 1) ? f : 1;
        h[j] = {sc * gau(), sc * gau()};
      }
      double u[18] = {}, ur[RC];
      if (form == 2) {
        su3(u, 1e-25);  // off the diagonal 1e-25
      } else {
        const double a = 6.283185307179586 * uni(), b = 6.283185307179586 * uni(), ph[3] = {a, b, -a - b};
        for (int d = 0; d < 3; d++) u[8 * d] = std::cos(ph[d]), u[8 * d + 1] = std::sin(ph[d]);
      }
      for (int j = 0; j < RC; j++) ur[j] = u[j];
      fix_hop<s, fwd, RC>(st.fx, mu, h, ur, false, false);
      cx<double> ud[9];
      cx<ld> ul[9];
      for (int j = 0; j < 9; j++) ud[j] = {u[2 * j], u[2 * j + 1]}, ul[j] = {u[2 * j], u[2 * j + 1]};
      if (RC == 12)  // the diagonal link's third row as the kernel rebuilds it
        ud[8] = {u[0] * u[8] - u[1] * u[9], -(u[0] * u[9] + u[1] * u[8])},
        ul[8] = {(ld)u[0] * u[8] - (ld)u[1] * u[9], -((ld)u[0] * u[9] + (ld)u[1] * u[8])};
      chain<double, mu, s, fwd>(st.dp, h, ud, false, false);
      chain<ld, mu, s, fwd>(st.ex, h, ul, false, false);
    };
    auto dir = [&](auto MU) {
      hop1(MU, std::integral_constant<int, S>(), std::true_type());
      hop1(MU, std::integral_constant<int, -S>(), std::false_type());
    };
    dir(std::integral_constant<int, 0>());
    dir(std::integral_constant<int, 1>());
    dir(std::integral_constant<int, 2>());
    dir(std::integral_constant<int, 3>());
    const bool take = fix_ok(st.fx) && fix_resolved(st.fx);
    no += !take;
    for (int j = 0; j < 12; j++) {
      const ld p = st.dp[j].r - st.ex[j].r, q = st.dp[j].i - st.ex[j].i;
      const ld a = take ? fix_double(st.fx.r[j], st.fx.E) - st.ex[j].r : p;
      const ld b = take ? fix_double(st.fx.i[j], st.fx.E) - st.ex[j].i : q;
      ef[j] += (double)(a * a + b * b);
      ed[j] += (double)(p * p + q * q);
    }
  }
  double w = 0;
  for (int j = 0; j < 12; j++) w = std::fmax(w, std::sqrt(ef[j] / ed[j]));
  refused = (double)no / n;
  return w;
}

// eight hops of links whose reals are all of size v (not unitary), all products of one sign
template <int RC>
static bool range_kept(double v, double size) {
  FixSite s;
  fix_begin(s);
  cx<double> h[6];
  double u[RC];
  for (auto& c : h) c = {size, -size};
  for (auto& c : u) c = v;
  for (int k = 0; k < 8; k++) fix_hop<-1, true, RC>(s, 3, h, u, false, false);  // all spins: + t
  if (!fix_ok(s)) return true;  // (refused: the chain)
  // rows 0 and 1: eight times six products v size (row 2 vanishes with 12 reals)
  return std::fabs(fix_double(s.r[0], s.E) / (48 * v * size) - 1) < 1e-15;
}

int main() {
  double worst = 0, no;
  for (int form = 0; form < 3; form++)
    for (double lf : {0., 2., 3.5, 4., 4.5, 5., 5.5, 8., 12., 20., 40., 60.}) {
      const double f = std::ldexp(1.0, -(int)lf) * (lf > (int)lf ? std::sqrt(0.5) : 1);
      const double r[2] = {ratio<18, 1>(form, f, 2000, no), ratio<12, -1>(form, f, 2000, no)};
      printf("form %d factor 2^-%g: errors %.3f %.3f of the chain's, refused %.2g\n", form, lf, r[0], r[1], no);
      if (lf == 0 && no > 0) return printf("FAIL: ordinary sites refused\n"), 1;
      worst = std::fmax(worst, std::fmax(r[0], r[1]));
    }
  for (double v : {1.0, 0.99, 0.9, 0.8, 0.7, 0.66, 0.6, 0.5})
    for (double size : {1.0, 1.3, 1.499, 1.5, 1.9999})
      if (!range_kept<18>(v, size) || !range_kept<12>(v, size))
        return printf("FAIL: range, links %g, spinors %g\n", v, size), 1;
  // at the threshold the two errors are equal to a tenth (2000 sites: 2 %)
  if (worst > 1.1) return printf("FAIL %.3f\n", worst), 1;
  printf("OK %.3f\n", worst);
  return 0;
}
