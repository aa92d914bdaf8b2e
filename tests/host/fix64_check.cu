// Host-side check of the fixed-point FP64 hopping sum (wd_fix64.cuh) and of
// the FP64 chain it replaces, both against long double, on sites of random
// neighbours and SU(3) links, over the forms that a site can take.  Prints
// both errors of each form (rms over components, relative to the rms component
// of each site), then "OK <sites> <largest fixed-point error / chain error>".
// Infinities, NaN and links that are not of order one have to be refused.
#include <cmath>
#include <cstdio>
#include <cstdlib>

#include "../../paper_0810_5365_gb300/csrc/wd_fix64.cuh"

using namespace wd;
typedef long double ld;

static unsigned long long sm = 0x1234567;
static double uni() {
  unsigned long long z = (sm += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return ((double)((z ^ (z >> 31)) >> 11) + 0.5) / 9007199254740992.0;
}
static double gau() { return std::sqrt(-2 * std::log(uni())) * std::cos(6.283185307179586 * uni()); }

struct C {
  ld r, i;
};
static C operator*(C a, C b) { return {a.r * b.r - a.i * b.i, a.r * b.i + a.i * b.r}; }
static C operator+(C a, C b) { return {a.r + b.r, a.i + b.i}; }
static C operator-(C a, C b) { return {a.r - b.r, a.i - b.i}; }
static C conj(C a) { return {a.r, -a.i}; }

// rows 0 and 1 orthonormal, row 2 their conjugate cross product (all rounded)
static void su3(double (&u)[18], double eps) {
  C m[3][3];
  for (int r = 0; r < 2; r++)
    for (int c = 0; c < 3; c++) m[r][c] = {(r == c) + eps * gau(), eps * gau()};
  for (int r = 0; r < 2; r++) {
    if (r) {
      C d = {0, 0};
      for (int c = 0; c < 3; c++) d = d + conj(m[0][c]) * m[1][c];
      for (int c = 0; c < 3; c++) m[1][c] = m[1][c] - d * m[0][c];
    }
    ld n = 0;
    for (int c = 0; c < 3; c++) n += m[r][c].r * m[r][c].r + m[r][c].i * m[r][c].i;
    for (int c = 0; c < 3; c++) m[r][c] = {m[r][c].r / sqrtl(n), m[r][c].i / sqrtl(n)};
  }
  for (int c = 0; c < 3; c++)
    m[2][c] = conj(m[0][(c + 1) % 3] * m[1][(c + 2) % 3] - m[0][(c + 2) % 3] * m[1][(c + 1) % 3]);
  for (int k = 0; k < 9; k++) {
    u[2 * k] = (double)m[k / 3][k % 3].r;
    u[2 * k + 1] = (double)m[k / 3][k % 3].i;
  }
}

template <typename R, int MU, int S, bool FWD>
static void chain(cx<R> (&acc)[12], const cx<double> (&hd)[6], const cx<R> (&u)[9], bool flip,
                  bool unit) {
  // the order of operations of the FP64 kernel (hop)
  cx<R> t[6];
  for (int hs = 0; hs < 2; hs++)
    for (int c = 0; c < 3; c++) {
      cx<R> v{0, 0};
      for (int d = 0; d < 3; d++) {
        const cx<R> h{(R)hd[hs * 3 + d].r, (R)hd[hs * 3 + d].i};
        const cx<R> e = FWD ? u[c * 3 + d] : u[d * 3 + c];
        const R s = FWD ? (R)1 : (R)-1;
        v.r = std::fma(e.r, h.r, v.r);
        v.r = std::fma(-s * e.i, h.i, v.r);
        v.i = std::fma(e.r, h.i, v.i);
        v.i = std::fma(s * e.i, h.r, v.i);
      }
      t[hs * 3 + c] = v;
      if (MU == 3 && unit) t[hs * 3 + c] = cx<R>{(R)hd[hs * 3 + c].r, (R)hd[hs * 3 + c].i};
      if (MU == 3 && flip) t[hs * 3 + c] = cx<R>{-t[hs * 3 + c].r, -t[hs * 3 + c].i};
    }
  auto add = [&](int k, cx<R> v, int s) {
    acc[k].r += s * v.r;
    acc[k].i += s * v.i;
  };
  auto addi = [&](int k, cx<R> v, int s) {
    acc[k].r -= s * v.i;
    acc[k].i += s * v.r;
  };
  for (int c = 0; c < 3; c++) {
    add(c, t[c], 1);
    add(3 + c, t[3 + c], 1);
    if (MU == 0) addi(6 + c, t[3 + c], -S), addi(9 + c, t[c], -S);
    if (MU == 1) add(6 + c, t[3 + c], -S), add(9 + c, t[c], S);
    if (MU == 2) addi(6 + c, t[c], -S), addi(9 + c, t[3 + c], S);
    if (MU == 3) add(6 + c, t[c], -S), add(9 + c, t[3 + c], -S);
  }
}

struct Site {
  FixSite fx;
  cx<double> dp[12];
  cx<ld> ex[12];
};

// spread: neighbours' magnitudes spread over 2^(+-spread)
template <int MU, int S, bool FWD, int RC>
static void hop(Site& st, int form, double spread) {
  cx<double> h[6];
  const double sc = std::ldexp(1.0, (int)((2 * uni() - 1) * spread)) * (form == 5 ? 1e200 : form == 6 ? 1e-200 : 1);
  for (int k = 0; k < 6; k++) h[k] = {sc * gau(), sc * gau()};
  if (form == 1 && uni() < 0.7) for (auto& v : h) v = {0, 0};       // sparse neighbourhoods
  if (form == 2) for (int k = 0; k < 6; k++) if (k % 3) h[k] = {0, -0.0};  // one colour
  double u[18];
  su3(u, form == 3 ? 0.0 : form == 4 ? 3.0 : 0.3);  // unit links, near the identity, anywhere
  double ur[RC];
  for (int k = 0; k < RC; k++) ur[k] = u[k];
  const bool flip = MU == 3 && uni() < 0.5, unit = MU == 3 && form == 7 && uni() < 0.5;
  fix_hop<S, FWD, RC>(st.fx, MU, h, ur, flip, unit);
  cx<double> ud[9];
  cx<ld> ul[9];
  for (int k = 0; k < 9; k++) ud[k] = {u[2 * k], u[2 * k + 1]}, ul[k] = {u[2 * k], u[2 * k + 1]};
  if (RC == 12) {
    auto cr = [](auto* v, int o, int a, int b, int c, int d) {
      auto R = [](auto x, auto y, auto p, auto q) { return x * y - p * q; };
      v[o].r = R(v[a].r, v[b].r, v[a].i, v[b].i) - R(v[c].r, v[d].r, v[c].i, v[d].i);
      v[o].i = -((v[a].r * v[b].i + v[a].i * v[b].r) - (v[c].r * v[d].i + v[c].i * v[d].r));
    };
    cr(ud, 6, 1, 5, 2, 4), cr(ud, 7, 2, 3, 0, 5), cr(ud, 8, 0, 4, 1, 3);
    cr(ul, 6, 1, 5, 2, 4), cr(ul, 7, 2, 3, 0, 5), cr(ul, 8, 0, 4, 1, 3);
  }
  chain<double, MU, S, FWD>(st.dp, h, ud, flip, unit);
  chain<ld, MU, S, FWD>(st.ex, h, ul, flip, unit);
}

template <int RC, int S>
static bool sites(int form, int n, double spread, double& ef, double& ed) {
  double sf = 0, sd = 0, norm = 0;
  for (int k = 0; k < n; k++) {
    Site st = {};
    fix_begin(st.fx);
    hop<0, S, true, RC>(st, form, spread);
    hop<0, -S, false, RC>(st, form, spread);
    hop<1, S, true, RC>(st, form, spread);
    hop<1, -S, false, RC>(st, form, spread);
    hop<2, S, true, RC>(st, form, spread);
    hop<2, -S, false, RC>(st, form, spread);
    hop<3, S, true, RC>(st, form, spread);
    hop<3, -S, false, RC>(st, form, spread);
    ld nn = 0, f = 0, d = 0;
    if (form == 1 && st.fx.any == 0)  // an all-zero neighbourhood gives exact zeros
      for (int j = 0; j < 12; j++)
        if (fix_double(st.fx.r[j], st.fx.E) != 0 || fix_double(st.fx.i[j], st.fx.E) != 0) return false;
    for (int j = 0; j < 12; j++) nn += st.ex[j].r * st.ex[j].r + st.ex[j].i * st.ex[j].i;
    if (!fix_ok(st.fx)) {
      printf("FAIL form %d: a site that fits was refused\n", form);
      return false;
    }
    for (int j = 0; j < 12; j++) {
      const ld a = fix_double(st.fx.r[j], st.fx.E) - st.ex[j].r, b = fix_double(st.fx.i[j], st.fx.E) - st.ex[j].i;
      f += a * a + b * b;
      const ld p = st.dp[j].r - st.ex[j].r, q = st.dp[j].i - st.ex[j].i;
      d += p * p + q * q;
    }
    if (nn > 0) sf += (double)(f / nn), sd += (double)(d / nn), norm += 1;
  }
  ef = std::sqrt(sf / norm);
  ed = std::sqrt(sd / norm);
  return true;
}

int main() {
  const int n = 400;
  double worst = 0;
  for (int form = 0; form < 8; form++)
    for (double spread : {0.0, 3.0, 40.0}) {
      double ef[4], ed[4];
      if (!sites<18, 1>(form, n, spread, ef[0], ed[0]) || !sites<18, -1>(form, n, spread, ef[1], ed[1]) ||
          !sites<12, 1>(form, n, spread, ef[2], ed[2]) || !sites<12, -1>(form, n, spread, ef[3], ed[3]))
        return 1;
      for (int j = 0; j < 4; j++) {
        printf("form %d spread %g recon %d: fixed %.3g chain %.3g\n", form, spread, j < 2 ? 18 : 12, ef[j], ed[j]);
        worst = std::fmax(worst, ef[j] / ed[j]);
      }
    }
  // what has to be refused: infinities, NaN, links that are not of order one
  for (int k = 0; k < 7; k++) {
    FixSite s;
    fix_begin(s);
    cx<double> h[6];
    for (auto& v : h) v = {gau(), gau()};
    double u[18];
    su3(u, 0.3);
    if (k == 0) h[3].i = INFINITY;
    if (k == 1) h[3].i = NAN;
    if (k == 2) u[7] = 1.5;
    if (k == 3) for (auto& v : u) v *= 0.01;
    if (k == 4) u[0] = NAN;
    if (k == 5) for (auto& v : h) v = {v.r * 1e-300, v.i * 1e-300};
    if (k == 6) for (auto& v : h) v = {0, 5e-320};
    fix_hop<1, true, 18>(s, 0, h, u, false, false);
    if (fix_ok(s)) {
      printf("FAIL refusal %d\n", k);
      return 1;
    }
  }
  // rows of ordinary size whose row 2 is larger (12-real storage, not SU(3))
  for (double z : {1.0, 0.6, -0.6, -1.0}) {
    double u[12] = {1, 0, 0, z, 0, 0, 0, z, 1, 0, 0, 0};  // row 2 = (0, 0, 1 + z^2)
    FixSite s;
    fix_begin(s);
    cx<double> h[6];
    for (auto& v : h) v = {gau(), gau()};
    fix_hop<1, true, 12>(s, 0, h, u, false, false);
    if (fix_ok(s)) {
      printf("FAIL refusal of row 2 (%g)\n", z);
      return 1;
    }
  }
  printf("OK %d %.3f\n", n, worst);
  return 0;
}
