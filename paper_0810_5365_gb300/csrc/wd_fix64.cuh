// The FP64 hopping sum in 64-bit fixed point on the integer pipe.
//
// GB300 issues FP64 at 1/64 of its FP32 rate (1.7 DADD lanes per SM and clock
// measured) but 64 lanes of 32 x 32 + 64 bit multiply-adds (mad.wide.s32) or
// 64-bit adds.  A hop needs 36 FP64 additions and 72 multiply-adds, so the
// FP64 pipe bounds the FP64 kernel at about 500 clocks per site and SM, seven
// times its memory time.  Here only the 12 additions of the spin projection
// stay on that pipe; the SU(3) product and the sum over the eight hops run on
// integers.
//
// Formats (E: the site's scale, a biased exponent, e = E - 1023; no projected
// component seen so far is 1.5 2^e or more):
//   half spinor  h = H 2^(e-61), |H| < 1.5 2^61
//   link         u = V 2^(el-61), |V| < 2^61 (1 + 2^-20), el 0 for SU(3) (fix_hop)
//   products     t = T 2^(e-58), below 2^60 each (fix_ok; rows of a norm of up
//                to one cannot give more), so that the sum of eight fits 64 bits
// H and V are cut into two signed 32-bit limbs, x = x.h 2^32 + x.l, and
// H V = H.h V.h 2^64 + (H.h V.l + H.l V.h) 2^32 + H.l V.l.  The last product
// is dropped (below 2^-59 of the largest |h|, rms), the middle ones are summed
// and rounded once per component and hop.  The FP64 chain rounds each of
// its 6 + 1 additions per hop at 2^-53 of the partial sum.
//
// Error: a site's sums share one scale, so the fixed-point error, 2^-58 of it
// (rms), is the same for all components, where the chain's goes with each
// component's own products.  Against 64-bit mantissas, relative to the rms
// component of the site: fixed point 0.48e-16, chain 1.42e-16 on Gaussian
// neighbours of one size, and the smaller for every form tried (unit links,
// single colours, sizes spread over 2^+-40: tests/host/fix64_check.cu).  A
// component whose products stay below 2^-5 of the scale would get fewer bits
// than the chain gives it (links that do not mix the colours, a spin that is
// small): its site takes the chain (fix_resolved).  Component by component the
// error is 0.41 of the chain's for products of one size and 0.95 of it at that
// line (tests/host/fix64_small_check.cu; 2^-6 would be 1.5 times the chain's).
//
// A site also falls back to the FP64 chain when a value does not fit: 12-real
// links with |u| above 1 or small throughout (not SU(3)), 18-real ones beyond
// 2^64, infinities, NaN, or exponents near the ends of the range.  Where a site
// falls back its warp pays both (24^3x48, us, every site in the chain / none:
// 660 / 187 with 18-real links, 812 / 212 with 12; the chain alone took 537 and
// 686).  On Gaussian fields no site does, on solutions and residuals of Gaussian
// sources at most one warp in ten thousand (links of mean 0.94) holds one.  On
// the propagator of a point source 0.1 to 2 % of the warps do (216 to 230 us,
// 18-real), on residuals of such a solve most; smoother links have more
// (propagators with exp(0.15 i H): 410 to 560 us).
//
// Instructions per hop: 30 conversions of 11 (a 64-bit shift written on two
// 32-bit words: on a 64-bit variable the compiler took 16), 216 multiply-adds,
// about 150 for the sums and their sizes and 60 for the scale.  The sizes and
// the three bits that T has for the line at 2^-5 (a carry between the halves of
// a row) cost 6 to 9 %: 174 -> 185 us and, with 12-real links, 193 -> 212 (the
// scale of 18-real links another 2); at 2^-3 without those bits the propagators
// above took the chain everywhere.
#pragma once

#include <string.h>

#include "wd_common.cuh"

namespace wd {

struct Limb {
  int h, l;
};

// 64-bit accumulators of a site: the four spins of the output, as T above
struct FixSite {
  long long r[12], i[12];
  int E;          // biased exponent of the scale
  unsigned any;   // non-zero: some neighbour was not zero
  unsigned bad;   // non-zero: a value did not fit
  // how large the hops' products have been (fix_size): of the x and y hops, of
  // the z and t hops, one word per colour, spin 0 in its low half
  unsigned xy[3], zt[3];
};

constexpr int FIX_EMIN = 128;   // smallest and largest scale handled
constexpr int FIX_EMAX = 1980;
// A component is resolved when one of its products reaches 2^-5 of the scale:
// fix_size's bits from T = 2^53 on.
constexpr unsigned FIX_FINE = 0xffc0ffc0u;
// Eight products below T = 2^60 cannot overflow: the bits from there on.
constexpr unsigned FIX_FULL = 0xe000e000u;
// The scale is one bit above the largest component's power of two where that
// component is 1.5 times it or more: a row of norm one then gives less than
// sqrt(6) 1.5 2^58 < 2^60.
constexpr unsigned FIX_ROOM = 0x80000u;
constexpr unsigned FIX_UMAX = 0x3ff00000u;  // high words of |u| < 1 + 2^-20 ...
constexpr unsigned FIX_UMIN = 0x3fc00000u;  // ... and of 1/8 (an SU(3) row has a real >= 0.23)
constexpr int FIX_LINK = 64;  // largest |el| of a link; zero and tiny links count as 2^-64

__host__ __device__ __forceinline__ unsigned long long d_bits(double x) {
  unsigned long long b;
  memcpy(&b, &x, 8);
  return b;
}

// (hi : lo) >> s, 0 for s > 63
__host__ __device__ __forceinline__ void shr_pair(unsigned& hi, unsigned& lo, int s) {
#ifdef __CUDA_ARCH__
  asm("{\n\t.reg .b64 t;\n\tmov.b64 t, {%1, %0};\n\tshr.u64 t, t, %2;\n\tmov.b64 {%1, %0}, t;\n\t}"
      : "+r"(hi), "+r"(lo) : "r"(s));
#else
  const unsigned long long v = s > 63 ? 0 : (((unsigned long long)hi << 32) | lo) >> s;
  hi = (unsigned)(v >> 32);
  lo = (unsigned)v;
#endif
}

__host__ __device__ __forceinline__ Limb fix_split(long long v) {
  Limb o;
  o.l = (int)(unsigned)v;
  o.h = (int)(v >> 32) + (int)((unsigned)o.l >> 31);
  return o;
}

// |x| with its leading bit (of 2^e) at bit 63 - (s - e), truncated, with x's
// sign; a negative value comes out one unit low (x ^ -1 for -x), as
// fix_neg's do
__host__ __device__ __forceinline__ Limb fix_limbs(unsigned long long b, int s) {
  const unsigned hi = (unsigned)(b >> 32), lo = (unsigned)b;
  const unsigned a = hi & 0x7fffffffu;
  const int sh = s - (int)(a >> 20);
  unsigned top = ((a << 11) | (lo >> 21)) | 0x80000000u, bot = lo << 11;
  shr_pair(top, bot, sh);
  const unsigned m = (unsigned)((int)hi >> 31);
  Limb o;
  o.l = (int)(bot ^ m);
  o.h = (int)(top ^ m) + (int)((unsigned)o.l >> 31);
  return o;
}

__host__ __device__ __forceinline__ Limb fix_neg(Limb a) {
  Limb o;
  o.h = -a.h;
  o.l = ~a.l;
  return o;
}

// One real of a sum of products, in two halves of at most four products each
// (their middle terms add up to less than 2^63): fix_carry between them.
struct FixAcc {
  long long A, B;
};
__host__ __device__ __forceinline__ void fix_mac(FixAcc& s, Limb u, Limb h) {
  s.A += (long long)u.h * h.h;
  s.B += (long long)u.h * h.l;
  s.B += (long long)u.l * h.h;
}
__host__ __device__ __forceinline__ void fix_carry(FixAcc& s) {
  s.A += s.B >> 32;
  s.B = (long long)(unsigned)s.B;
}
__host__ __device__ __forceinline__ long long fix_round(const FixAcc& s) {
  return s.A + (s.B >> 32);
}

// conj(a b - c d) as a link element (row 2 of an SU(3) matrix)
__host__ __device__ __forceinline__ void fix_cross(Limb (&o)[2], const Limb (&a)[2],
                                                   const Limb (&b)[2], const Limb (&c)[2],
                                                   const Limb (&d)[2]) {
  const Limb nbi = fix_neg(b[1]), ndr = fix_neg(d[0]), nbr = fix_neg(b[0]);
  FixAcc re = {0, 1LL << 28}, im = {0, 1LL << 28};
  // -(a.r b.i + a.i b.r - c.r d.i - c.i d.r)
  fix_mac(re, a[0], b[0]);
  fix_mac(im, a[0], nbi);
  fix_mac(re, a[1], nbi);
  fix_mac(im, a[1], nbr);
  fix_carry(re);
  fix_carry(im);
  fix_mac(re, c[0], ndr);
  fix_mac(im, c[0], d[1]);
  fix_mac(re, c[1], d[1]);
  fix_mac(im, c[1], d[0]);
  // products 2^-122 -> 2^-61 (up to 2^63 where |u| is up to one: fix_hop's check
  // sees the wrapped value too)
  o[0] = fix_split((long long)((unsigned long long)re.A * 8) + (re.B >> 29));
  o[1] = fix_split((long long)((unsigned long long)im.A * 8) + (im.B >> 29));
}

// Site state before its first hop.
__host__ __device__ __forceinline__ void fix_begin(FixSite& acc) {
#pragma unroll
  for (int k = 0; k < 12; k++) acc.r[k] = acc.i[k] = 0;
#pragma unroll
  for (int c = 0; c < 3; c++) acc.xy[c] = acc.zt[c] = 0;
  acc.E = FIX_EMIN;
  acc.any = acc.bad = 0;
}

__host__ __device__ __forceinline__ unsigned fix_sizes(const FixSite& a) {
  return a.xy[0] | a.xy[1] | a.xy[2] | a.zt[0] | a.zt[1] | a.zt[2];
}

// Raise the site's scale to that of the projected half spinor h when h is
// larger (with some room, so that few of the later hops raise it again: each
// time costs the shift of all sums).  A half spinor that vanishes goes
// through the products like any other: they come out as zero, a link that does
// not fit is seen (0 times NaN is NaN), and the time of a launch, which the
// tuners compare, does not depend on how much of a field is zero.
// el: the link's exponent (fix_hop).
__host__ __device__ __forceinline__ void fix_scale(FixSite& acc, const cx<double> (&h)[6],
                                                   int el) {
  unsigned m = 0;
#pragma unroll
  for (int k = 0; k < 6; k++) {
    const unsigned a = (unsigned)(d_bits(h[k].r) >> 32) & 0x7fffffffu;
    const unsigned b = (unsigned)(d_bits(h[k].i) >> 32) & 0x7fffffffu;
    m = m > a ? m : a;
    m = m > b ? m : b;
  }
  acc.any |= m;
  if (m == 0) {
    // a zero neighbour (point sources), or denormals of up to 2^-1043
    unsigned long long lows = 0;
#pragma unroll
    for (int k = 0; k < 6; k++) lows |= d_bits(h[k].r) | d_bits(h[k].i);
    acc.bad |= (unsigned)lows;
  }
  const int e = (int)((m + FIX_ROOM) >> 20) + el;
  if (e > acc.E) {
    const int d = e - acc.E < 63 ? e - acc.E : 63;
    acc.E = e;
#pragma unroll
    for (int k = 0; k < 12; k++) {
      acc.r[k] >>= d;
      acc.i[k] >>= d;
    }
    const int dw = d < 16 ? d : 16;
    const unsigned keep = (0xffffu >> dw) * 0x10001u;
    acc.bad |= fix_sizes(acc) & FIX_FULL;
#pragma unroll
    for (int c = 0; c < 3; c++) {
      acc.xy[c] = (acc.xy[c] >> dw) & keep;
      acc.zt[c] = (acc.zt[c] >> dw) & keep;
    }
  }
}

// The largest |high word| of n link reals so far, and at the end whether the
// link is one that V can hold.
__host__ __device__ __forceinline__ void fix_link_max(unsigned& um, unsigned long long b) {
  const unsigned a = (unsigned)(b >> 32) & 0x7fffffffu;
  um = um > a ? um : a;
}

// t = (row c of U h) or (row c of U^+ h) for one of the two half spinors:
// v[d] = U[c][d] or U[d][c], H[d] the limbs of h
template <bool FWD>
__host__ __device__ __forceinline__ void fix_row(long long& tr, long long& ti,
                                                 const Limb (&v)[3][2], const Limb (*H)[2]) {
  FixAcc re = {0, 1LL << 31}, im = {0, 1LL << 31};
#pragma unroll
  for (int d = 0; d < 3; d++) {
    fix_mac(re, v[d][0], H[d][0]);
    fix_mac(im, v[d][0], H[d][1]);
  }
  fix_carry(re);
  fix_carry(im);
#pragma unroll
  for (int d = 0; d < 3; d++) {
    const Limb n = fix_neg(H[d][FWD ? 1 : 0]);
    fix_mac(re, v[d][1], FWD ? n : H[d][1]);
    fix_mac(im, v[d][1], FWD ? H[d][0] : n);
  }
  tr = fix_round(re);
  ti = fix_round(im);
}

// The size of two products: the bits at which v's leading 16 differ from the
// bit below, the first in the low half of the word, the second in the high one
// (bit b + 1 of T is set where |T| >= 2^b; the carry from the low half only
// reaches bit 0 of the high one)
__host__ __device__ __forceinline__ unsigned fix_size(long long v0, long long v1) {
  const unsigned a = (unsigned)((unsigned long long)v0 >> 32);
  const unsigned b = (unsigned)((unsigned long long)v1 >> 32);
#ifdef __CUDA_ARCH__
  const unsigned w = __byte_perm(a, b, 0x7632);
#else
  const unsigned w = (a >> 16) | (b & 0xffff0000u);
#endif
  return w ^ (w << 1);
}

// Colour c of the expansion of expand_add: upper spins t0, t1, lower spins
// +-S t or +-S i t (of direction mu).
template <int S>
__host__ __device__ __forceinline__ void fix_expand(FixSite& acc, int mu, int c, long long r0,
                                                    long long i0, long long r1, long long i1) {
  const unsigned w = fix_size(r0, r1) | fix_size(i0, i1);
  if (mu < 2)
    acc.xy[c] |= w;
  else
    acc.zt[c] |= w;
  acc.r[c] += r0;
  acc.i[c] += i0;
  acc.r[3 + c] += r1;
  acc.i[3 + c] += i1;
  auto add = [&](int k, long long r, long long i, int sgn) {
    acc.r[k] = sgn > 0 ? acc.r[k] + r : acc.r[k] - r;
    acc.i[k] = sgn > 0 ? acc.i[k] + i : acc.i[k] - i;
  };
  // sgn * i t = (-sgn t.i, sgn t.r)
  auto add_i = [&](int k, long long r, long long i, int sgn) {
    acc.r[k] = sgn > 0 ? acc.r[k] - i : acc.r[k] + i;
    acc.i[k] = sgn > 0 ? acc.i[k] + r : acc.i[k] - r;
  };
  switch (mu) {
    case 0:  // lower = (-S i t1, -S i t0)
      add_i(6 + c, r1, i1, -S);
      add_i(9 + c, r0, i0, -S);
      break;
    case 1:  // lower = (-S t1, S t0)
      add(6 + c, r1, i1, -S);
      add(9 + c, r0, i0, S);
      break;
    case 2:  // lower = (-S i t0, S i t1)
      add_i(6 + c, r0, i0, -S);
      add_i(9 + c, r1, i1, S);
      break;
    default:  // lower = (-S t0, -S t1)
      add(6 + c, r0, i0, -S);
      add(9 + c, r1, i1, -S);
      break;
  }
}

// One hop of direction mu: the projected half spinor h (six complex doubles)
// times the link u (RC reals as stored; not read when unit), added to the
// site's sums.  Colour by colour, so that only one row of products is live
// beside the sums.
//
// SIZED (18-real links): a link that is not of order one (tadpole-scaled or
// smeared ones, anisotropic actions) is held as 2^el times one that is, and its
// products scale the site: without it each site next to such a link took the
// chain after its fixed-point pass, 24^3x48 651 us a launch where the chain
// alone took 537, and now 188.  12-real links are SU(3), others take the chain: row 2, a
// product of the rows, does not scale with them.
template <int S, bool FWD, int RC, bool SIZED = false>
__host__ __device__ __forceinline__ void fix_hop(FixSite& acc, int mu, const cx<double> (&h)[6],
                                                 const double (&u)[RC], bool flip, bool unit) {
  static_assert(!SIZED || RC == 18, "12-real links have no scale of their own");
  unsigned um = 0;
  int el = 0;
  if (SIZED && !unit) {
#pragma unroll
    for (int k = 0; k < RC; k++) fix_link_max(um, d_bits(u[k]));
    if (um > FIX_UMAX || um < FIX_UMIN) {
      el = (int)((um + 0xfffffu) >> 20) - 1023;
      acc.bad |= el > FIX_LINK ? 1u : 0u;
      el = el > FIX_LINK ? FIX_LINK : el < -FIX_LINK ? -FIX_LINK : el;
    }
  }
  fix_scale(acc, h, el);
  Limb H[6][2];
#pragma unroll
  for (int k = 0; k < 6; k++) {
    H[k][0] = fix_limbs(d_bits(h[k].r), acc.E - el + 2);
    H[k][1] = fix_limbs(d_bits(h[k].i), acc.E - el + 2);
  }
  if (flip) {
#pragma unroll
    for (int k = 0; k < 6; k++) {
      H[k][0] = fix_neg(H[k][0]);
      H[k][1] = fix_neg(H[k][1]);
    }
  }
  if (unit) {
#pragma unroll
    for (int c = 0; c < 3; c++) {
      auto t = [](Limb a) { return ((((long long)a.h << 32) + a.l) + 4) >> 3; };
      fix_expand<S>(acc, mu, c, t(H[c][0]), t(H[c][1]), t(H[3 + c][0]), t(H[3 + c][1]));
    }
    return;
  }
  Limb U[9][2];
  if (RC == 12) {
#pragma unroll
    for (int k = 0; k < RC; k++) {
      fix_link_max(um, d_bits(u[k]));
      U[k >> 1][k & 1] = fix_limbs(d_bits(u[k]), 1023 + 2);
    }
    fix_cross(U[6], U[1], U[5], U[2], U[4]);
    fix_cross(U[7], U[2], U[3], U[0], U[5]);
    fix_cross(U[8], U[0], U[4], U[1], U[3]);
    // (rows that are not orthonormal can give a larger row 2, which the sums
    // have no room for: t or 2 L - t is negative when |V.h| > L)
    constexpr unsigned L = (1u << 29) + 512;
    unsigned big = 0;
#pragma unroll
    for (int k = 6; k < 9; k++)
#pragma unroll
      for (int j = 0; j < 2; j++) {
        const unsigned t = (unsigned)U[k][j].h + L;
        big |= t | (2 * L - t);
      }
    acc.bad |= big >> 31;
  }
#pragma unroll
  for (int c = 0; c < 3; c++) {
    Limb v[3][2];
#pragma unroll
    for (int d = 0; d < 3; d++) {
#pragma unroll
      for (int j = 0; j < 2; j++) {
        const int k = FWD ? c * 3 + d : d * 3 + c;
        if (RC == 12) {
          v[d][j] = U[k][j];
        } else {
          if (!SIZED) fix_link_max(um, d_bits(u[2 * k + j]));
          v[d][j] = fix_limbs(d_bits(u[2 * k + j]), 1023 + el + 2);
        }
      }
    }
    long long r0, i0, r1, i1;
    fix_row<FWD>(r0, i0, v, &H[0]);
    fix_row<FWD>(r1, i1, v, &H[3]);
    fix_expand<S>(acc, mu, c, r0, i0, r1, i1);
  }
  if (!SIZED) acc.bad |= (um > FIX_UMAX || um < FIX_UMIN) ? 1u : 0u;
}

// whether the site's sums are valid (else: the FP64 chain)
__host__ __device__ __forceinline__ bool fix_ok(const FixSite& a) {
  return (a.bad | (fix_sizes(a) & FIX_FULL)) == 0 && a.E < FIX_EMAX && (a.E > FIX_EMIN || a.any == 0);
}

// Whether every component of the site has as many bits as the FP64 chain would
// give it.  The sums of a site share one scale, so a component all of whose
// products are small keeps fewer bits (none, 2^-55 below the scale), where the
// chain rounds each relative to its own products.  With links that mix the
// colours the products of a component are of the size of its neighbours; with
// links that do not (unit, diagonal) a colour can stay small.  Spins 0 and 1
// add the products of their own rows; spins 2 and 3 those of spins 1 and 0
// along x and y, of 0 and 1 along z and t.
__host__ __device__ __forceinline__ bool fix_resolved(const FixSite& a) {
  bool all = true;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const unsigned up = (a.xy[c] | a.zt[c]) & FIX_FINE;
    const unsigned low = (((a.xy[c] << 16) | (a.xy[c] >> 16)) | a.zt[c]) & FIX_FINE;
    all = all && (up & 0xffffu) && (up >> 16) && (low & 0xffffu) && (low >> 16);
  }
  return all || a.any == 0;
}

// T 2^(E - 1023 - 58) as a double, rounded to nearest
__host__ __device__ __forceinline__ double fix_double(long long t, int E) {
  const long long s = t >> 63;
  const unsigned long long m = (unsigned long long)((t ^ s) - s);
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)m);
#else
  const int lz = m ? __builtin_clzll(m) : 64;
#endif
  const unsigned long long n = m << (lz & 63);
  unsigned long long b = ((unsigned long long)(E + 4 - lz) << 52) + (n >> 11) + ((n >> 10) & 1);
  b |= (unsigned long long)s & 0x8000000000000000ull;
  if (m == 0) b = 0;
  double d;
  memcpy(&d, &b, 8);
  return d;
}

}  // namespace wd
