// Device-side building blocks shared by the libwd kernels: lattice geometry,
// the site-blocked packed field formats, complex arithmetic and the
// deterministic FP64 block reduction.
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <stdint.h>
#include <stddef.h>
#include <string.h>

#include <type_traits>

#include "../../include/wd.h"

namespace wd {

// ---------------------------------------------------------------------------
// geometry
// ---------------------------------------------------------------------------

// Sites per block of the site-blocked structure-of-arrays layout.  A block of
// 32 consecutive checkerboard sites stores component group k of all its sites
// contiguously, so one warp reading one group issues a single 512-byte (FP32)
// or 1024-byte (FP64) fully coalesced request of 128-bit vectors.
constexpr int SB = 32;

// Exact division by an invariant d for 0 <= n < 2^31 by one 64-bit multiply
// and a shift (Granlund and Montgomery, "Division by invariant integers using
// multiplication", PLDI 1994): with s = ceil(log2 d) and M = ceil(2^(32+s)/d),
// floor(n/d) = (n * M) >> (32 + s), since the rounding error of M contributes
// less than n / 2^(32+s) < 1/(2d).
struct FastDiv {
  unsigned long long M;
  int shift;  // 32 + s
  int d;
};

inline FastDiv make_fastdiv(int d) {
  FastDiv f;
  int s = 0;
  while ((1LL << s) < d) s++;
  unsigned __int128 num = (unsigned __int128)1 << (32 + s);
  f.M = (unsigned long long)((num + (unsigned)d - 1) / (unsigned)d);
  f.shift = 32 + s;
  f.d = d;
  return f;
}

__host__ __device__ __forceinline__ int fdiv(int n, const FastDiv& f) {
  return (int)(((unsigned long long)(unsigned)n * f.M) >> f.shift);
}

struct Geom {
  int L[4];    // extents
  int Lh0;     // L0 / 2
  int Vh;      // sites per parity
  int Vh_pad;  // Vh rounded up to a multiple of SB
  int S1;      // checkerboard stride of +y  (Lh0)
  int S2;      // checkerboard stride of +z  (Lh0 * L1)
  int S3;      // checkerboard stride of +t  (Lh0 * L1 * L2)
  FastDiv dLh0, dL1, dL2;
};

inline Geom make_geom(const int d[4]) {
  Geom g;
  for (int i = 0; i < 4; i++) g.L[i] = d[i];
  g.Lh0 = d[0] / 2;
  long long V = (long long)d[0] * d[1] * d[2] * d[3];
  g.Vh = (int)(V / 2);
  g.Vh_pad = (g.Vh + SB - 1) / SB * SB;
  g.S1 = g.Lh0;
  g.S2 = g.Lh0 * d[1];
  g.S3 = g.Lh0 * d[1] * d[2];
  g.dLh0 = make_fastdiv(g.Lh0);
  g.dL1 = make_fastdiv(d[1]);
  g.dL2 = make_fastdiv(d[2]);
  return g;
}

// Checkerboard site cb of parity p -> coordinates (x0..x3).
__host__ __device__ __forceinline__ void cb_coords(int cb, int p, const Geom& g, int& x0, int& x1, int& x2,
                                          int& x3) {
  const int r0 = fdiv(cb, g.dLh0);
  const int xh = cb - r0 * g.Lh0;
  const int r1 = fdiv(r0, g.dL1);
  x1 = r0 - r1 * g.L[1];
  x3 = fdiv(r1, g.dL2);
  x2 = r1 - x3 * g.L[2];
  x0 = 2 * xh + ((p + x1 + x2 + x3) & 1);
}

// vector index of component group k (of NC) of checkerboard site cb
__host__ __device__ __forceinline__ size_t sbi(int cb, int k, int NC) {
  return ((size_t)(cb >> 5) * NC + k) * SB + (cb & (SB - 1));
}

// ---------------------------------------------------------------------------
// complex arithmetic
// ---------------------------------------------------------------------------

template <typename R>
struct cx {
  R r, i;
};

template <typename R>
__device__ __forceinline__ cx<R> mk(R r, R i) { cx<R> c; c.r = r; c.i = i; return c; }
template <typename R>
__device__ __forceinline__ cx<R> operator+(cx<R> a, cx<R> b) { return mk(a.r + b.r, a.i + b.i); }
template <typename R>
__device__ __forceinline__ cx<R> operator-(cx<R> a, cx<R> b) { return mk(a.r - b.r, a.i - b.i); }
template <typename R>
__device__ __forceinline__ cx<R> operator*(R s, cx<R> a) { return mk(s * a.r, s * a.i); }
// i * a
template <typename R>
__device__ __forceinline__ cx<R> ti(cx<R> a) { return mk(-a.i, a.r); }
// a * b
template <typename R>
__device__ __forceinline__ cx<R> cmul(cx<R> a, cx<R> b) {
  return mk(a.r * b.r - a.i * b.i, a.r * b.i + a.i * b.r);
}
// acc + a * b
template <typename R>
__device__ __forceinline__ cx<R> cmadd(cx<R> a, cx<R> b, cx<R> acc) {
  acc.r = fma(a.r, b.r, acc.r);
  acc.r = fma(-a.i, b.i, acc.r);
  acc.i = fma(a.r, b.i, acc.i);
  acc.i = fma(a.i, b.r, acc.i);
  return acc;
}
// acc + conj(a) * b
template <typename R>
__device__ __forceinline__ cx<R> cjmadd(cx<R> a, cx<R> b, cx<R> acc) {
  acc.r = fma(a.r, b.r, acc.r);
  acc.r = fma(a.i, b.i, acc.r);
  acc.i = fma(a.r, b.i, acc.i);
  acc.i = fma(-a.i, b.r, acc.i);
  return acc;
}
// conj(a * b - c * d)
template <typename R>
__device__ __forceinline__ cx<R> conj_cross(cx<R> a, cx<R> b, cx<R> c, cx<R> d) {
  R re = a.r * b.r - a.i * b.i - (c.r * d.r - c.i * d.i);
  R im = a.r * b.i + a.i * b.r - (c.r * d.i + c.i * d.r);
  return mk(re, -im);
}

// ---------------------------------------------------------------------------
// per-site reductions: the 24 terms of one site are summed in the working
// precision R.  The kernels that fuse a reduction keep summing in R over the
// sites of a warp or block, and the per-block (or per-warp) partials are
// summed in FP64.  GB300 issues FP64 at 1/64 of its FP32 rate: a sum over
// sites in FP64 (a shuffle tree of DADDs per warp) costs more than the
// memory traffic of the kernels that fuse these reductions.
// ---------------------------------------------------------------------------

// the arithmetic type of a storage precision (FP32 for FP16 storage)
template <int P>
using real_of = typename std::conditional<P == WD_F64, double, float>::type;

template <typename T = double, typename R>
__device__ __forceinline__ T site_norm2(const cx<R> (&v)[12]) {
  R t = (R)0;
#pragma unroll
  for (int k = 0; k < 12; k++) {
    t = fma(v[k].r, v[k].r, t);
    t = fma(v[k].i, v[k].i, t);
  }
  return (T)t;
}

// re + i im += sum_k conj(a_k) b_k
template <typename R, typename T>
__device__ __forceinline__ void site_cdot(const cx<R> (&a)[12], const cx<R> (&b)[12], T& re,
                                          T& im) {
  R r = (R)0, i = (R)0;
#pragma unroll
  for (int k = 0; k < 12; k++) {
    r = fma(a[k].r, b[k].r, r);
    r = fma(a[k].i, b[k].i, r);
    i = fma(a[k].r, b[k].i, i);
    i = fma(-a[k].i, b[k].r, i);
  }
  re += (T)r;
  im += (T)i;
}

// ---------------------------------------------------------------------------
// packed spinor formats (per parity; Vh_pad sites)
//   WD_F64: NC = 12 double2, group k = complex component k = spin*3 + colour
//   WD_F32: NC =  6 float4,  group k = components 2k, 2k+1
//   WD_F16: NC =  3 int4,    group k = components 4k..4k+3 as half2 (re, im),
//           followed by float scale[Vh_pad]; value = half * scale
// ---------------------------------------------------------------------------

template <int P> struct SpinorFmt;
template <> struct SpinorFmt<WD_F64> { static constexpr size_t bytes_per_site = 192; };
template <> struct SpinorFmt<WD_F32> { static constexpr size_t bytes_per_site = 96; };
template <> struct SpinorFmt<WD_F16> { static constexpr size_t bytes_per_site = 52; };

inline size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

inline size_t spinor_half_bytes(const Geom& g, int prec) {
  size_t per = prec == WD_F64 ? 192 : prec == WD_F32 ? 96 : 52;
  return round_up((size_t)g.Vh_pad * per, 256);
}

// Programmatic dependent launch.  wait blocks until the previous kernel of the
// stream has completed and its writes are visible; launch_dependents lets the
// next kernel be scheduled once every CTA of this grid has got here (its CTAs
// then fill the SM slots that this grid's last wave frees).  A kernel calls
// this before its first global memory access, so it never reads or writes
// anything its predecessor may still touch.  Both are no-ops for a launch
// without the programmatic-serialisation attribute.
// In this order one grid at most waits behind a running one.  The other way
// round several small grids queue up on the SMs, their CTAs land unevenly, and
// a launch takes up to half again as long.  us per hopping launch in a stream,
// launch_dependents first / wait first: FP32 14x10x18x22 6.1 / 4.2, 16^4 5.8 /
// 4.7 (with a fused norm 7.9 / 5.7), FP16 16^4 4.4 / 4.0 (7.1 / 5.5); 8^4 (3.1)
// and grids of more than a wave (24^4 FP32 15.2) do not change.
__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.wait;\n\tgriddepcontrol.launch_dependents;\n" ::: "memory");
}

// Bring bytes (a multiple of 16, at a 16-byte boundary) into L2; nothing waits
// for it.
__device__ __forceinline__ void prefetch_l2(const void* p, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(p), "r"(bytes) : "memory");
}

// The FP16 links of directions mu < nmu that the n output sites from c0 on
// (parity p) will read, brought into L2 by the first 4 nmu lanes of a warp, one
// region and part each.  Backward links are taken at the shifted sites without
// the wrap at the lattice's edge.  n and c0 even, c0 + n <= Vh.
__device__ __forceinline__ void prefetch_links_f16(const void* gauge, const Geom& g, int p, int c0,
                                                   int n, int nmu, int lane) {
  if (lane >= 4 * nmu) return;
  const int r = lane >> 1, mu = r >> 1;
  const bool bwd = r & 1;
  const int shift = !bwd || mu == 0 ? 0 : mu == 1 ? g.S1 : mu == 2 ? g.S2 : g.S3;
  const int s = (c0 > shift ? c0 - shift : 0) & ~1;  // (8-byte part: 16-byte boundary)
  const size_t at = (size_t)(2 * mu + (bwd ? 1 - p : p)) * g.Vh_pad + s;
  const char* b = (const char*)gauge;
  if (lane & 1)
    prefetch_l2(b + (size_t)8 * g.Vh_pad * 16 + at * 8, n * 8);
  else
    prefetch_l2(b + at * 16, n * 16);
}

// A load of an input field.  COH = false: the read-only data path (the field
// is not written while the kernel runs).  COH = true: an ordinary coherent
// load, for a kernel that reads fields written earlier in the same launch by
// other CTAs (after a grid barrier).
template <bool COH, typename T>
__device__ __forceinline__ T ldin(const T* p) {
  if constexpr (COH)
    return __ldca(p);
  else
    return __ldg(p);
}

// float <-> double on the integer pipe, with the results of the conversion
// instructions (round to nearest even).  Those run on GB300's FP64 pipe, at
// 1/64 of the FP32 rate: the 24 of a site took longer than its memory traffic
// (packing links to FP32: 64 % of that pipe busy, also where they were
// predicated off).  Normal numbers and zeros are done here; a site that holds
// anything else takes the instructions, in a branch of its own.
__host__ __device__ __forceinline__ bool narrows(double d) {  // zero, or in [2^-126, 2^128)
  unsigned long long r;
  memcpy(&r, &d, 8);
  const unsigned a = (unsigned)(r >> 32) & 0x7fffffffu;
  return a - 0x38100000u < 0x0fe00000u || (a | (unsigned)r) == 0u;
}
__host__ __device__ __forceinline__ float narrow(double d) {
  unsigned long long r;
  memcpy(&r, &d, 8);
  const unsigned hi = (unsigned)(r >> 32), lo = (unsigned)r, a = hi & 0x7fffffffu;
  const unsigned m = ((a - 0x38000000u) << 3) | (lo >> 29), rem = lo << 3;
  const unsigned up = (rem > 0x80000000u || (rem == 0x80000000u && (m & 1u))) ? 1u : 0u;
  const unsigned b = (hi & 0x80000000u) | ((a | lo) == 0u ? 0u : m + up);
  float f;
  memcpy(&f, &b, 4);
  return f;
}
__host__ __device__ __forceinline__ bool widens(float f) {  // zero or normal
  unsigned b;
  memcpy(&b, &f, 4);
  b &= 0x7fffffffu;
  return b - 0x00800000u < 0x7f000000u || b == 0u;
}
__host__ __device__ __forceinline__ double widen(float f) {
  unsigned b;
  memcpy(&b, &f, 4);
  const unsigned a = b & 0x7fffffffu;
  const unsigned hi = a == 0u ? b : (b & 0x80000000u) | ((a >> 3) + 0x38000000u), lo = b << 29;
  const unsigned long long r = ((unsigned long long)hi << 32) | lo;
  double d;
  memcpy(&d, &r, 8);
  return d;
}
template <int N>
__host__ __device__ __forceinline__ void convert(cx<float> (&o)[N], const cx<double> (&s)[N]) {
  bool plain = true;
#pragma unroll
  for (int k = 0; k < N; k++) plain = plain && narrows(s[k].r) && narrows(s[k].i);
  if (plain) {
#pragma unroll
    for (int k = 0; k < N; k++) o[k].r = narrow(s[k].r), o[k].i = narrow(s[k].i);
  } else {
#pragma unroll
    for (int k = 0; k < N; k++) o[k].r = (float)s[k].r, o[k].i = (float)s[k].i;
  }
}
template <int N>
__host__ __device__ __forceinline__ void convert(cx<double> (&o)[N], const cx<float> (&s)[N]) {
  bool plain = true;
#pragma unroll
  for (int k = 0; k < N; k++) plain = plain && widens(s[k].r) && widens(s[k].i);
  if (plain) {
#pragma unroll
    for (int k = 0; k < N; k++) o[k].r = widen(s[k].r), o[k].i = widen(s[k].i);
  } else {
#pragma unroll
    for (int k = 0; k < N; k++) o[k].r = (double)s[k].r, o[k].i = (double)s[k].i;
  }
}
// The array that values of type T go through on their way to or from s: s
// itself when it has that type (then the conversion is nothing), else tmp.
template <typename T, int N>
__host__ __device__ __forceinline__ cx<T> (&through(cx<T> (&s)[N], cx<T> (&)[N]))[N] {
  return s;
}
template <typename T, typename R, int N>
__host__ __device__ __forceinline__ cx<T> (&through(cx<R> (&)[N], cx<T> (&tmp)[N]))[N] {
  return tmp;
}
template <typename R, int N>
__host__ __device__ __forceinline__ void convert(cx<R> (&)[N], const cx<R> (&)[N]) {}

// Load the 12 complex components of site cb as type R.
template <int P, typename R, bool COH = false>
__device__ __forceinline__ void load_spinor(cx<R> (&s)[12], const void* base, int cb, int Vh_pad) {
  if constexpr (P == WD_F64) {
    const double2* p = (const double2*)base;
#pragma unroll
    for (int k = 0; k < 12; k++) {
      double2 v = ldin<COH>(p + sbi(cb, k, 12));
      s[k] = mk<R>((R)v.x, (R)v.y);
    }
  } else if constexpr (P == WD_F32) {
    const float4* p = (const float4*)base;
#pragma unroll
    for (int k = 0; k < 6; k++) {
      float4 v = ldin<COH>(p + sbi(cb, k, 6));
      s[2 * k] = mk<R>((R)v.x, (R)v.y);
      s[2 * k + 1] = mk<R>((R)v.z, (R)v.w);
    }
  } else {
    const int4* p = (const int4*)base;
    const float* sc = (const float*)((const char*)base + (size_t)Vh_pad * 48);
    float scale = ldin<COH>(sc + cb);
#pragma unroll
    for (int k = 0; k < 3; k++) {
      int4 v = ldin<COH>(p + sbi(cb, k, 3));
      const __half2* h = reinterpret_cast<const __half2*>(&v);
#pragma unroll
      for (int j = 0; j < 4; j++) {
        float2 f = __half22float2(h[j]);
        s[4 * k + j] = mk<R>((R)(f.x * scale), (R)(f.y * scale));
      }
    }
  }
}

// Plain (cached) load variant for fields that this kernel also writes
// (x, y operands that may alias out): no read-only path.
template <int P, typename R>
__device__ __forceinline__ void load_spinor_rw(cx<R> (&s)[12], const void* base, int cb, int Vh_pad) {
  if constexpr (P == WD_F64) {
    const double2* p = (const double2*)base;
    cx<double> tmp[12];
    auto& w = through<double>(s, tmp);
#pragma unroll
    for (int k = 0; k < 12; k++) {
      double2 v = p[sbi(cb, k, 12)];
      w[k] = mk<double>(v.x, v.y);
    }
    convert(s, w);
  } else if constexpr (P == WD_F32) {
    const float4* p = (const float4*)base;
    cx<float> tmp[12];
    auto& w = through<float>(s, tmp);
#pragma unroll
    for (int k = 0; k < 6; k++) {
      float4 v = p[sbi(cb, k, 6)];
      w[2 * k] = mk<float>(v.x, v.y);
      w[2 * k + 1] = mk<float>(v.z, v.w);
    }
    convert(s, w);
  } else {
    const int4* p = (const int4*)base;
    const float* sc = (const float*)((const char*)base + (size_t)Vh_pad * 48);
    float scale = sc[cb];
    cx<float> tmp[12];
    auto& w = through<float>(s, tmp);
#pragma unroll
    for (int k = 0; k < 3; k++) {
      int4 v = p[sbi(cb, k, 3)];
      const __half2* h = reinterpret_cast<const __half2*>(&v);
#pragma unroll
      for (int j = 0; j < 4; j++) {
        float2 f = __half22float2(h[j]);
        w[4 * k + j] = mk<float>(f.x * scale, f.y * scale);
      }
    }
    convert(s, w);
  }
}

// One site of a packed field as it sits in memory (the format load_spinor_rw
// reads), so that a kernel can issue the loads of its next site before it
// computes the current one.
template <int P>
struct RawSite;
template <>
struct RawSite<WD_F16> {
  int4 v[3];
  float s;
};
template <>
struct RawSite<WD_F32> {
  float4 v[6];
};
template <>
struct RawSite<WD_F64> {
  double2 v[12];
};

template <int P>
__device__ __forceinline__ void load_raw(RawSite<P>& o, const void* base, int cb, int Vh_pad) {
  if constexpr (P == WD_F16) {
    const int4* p = (const int4*)base;
#pragma unroll
    for (int k = 0; k < 3; k++) o.v[k] = p[sbi(cb, k, 3)];
    o.s = ((const float*)((const char*)base + (size_t)Vh_pad * 48))[cb];
  } else if constexpr (P == WD_F32) {
    const float4* p = (const float4*)base;
#pragma unroll
    for (int k = 0; k < 6; k++) o.v[k] = p[sbi(cb, k, 6)];
  } else {
    const double2* p = (const double2*)base;
#pragma unroll
    for (int k = 0; k < 12; k++) o.v[k] = p[sbi(cb, k, 12)];
  }
}

// the values of a raw site, with the arithmetic of load_spinor_rw
template <int P, typename R>
__device__ __forceinline__ void unpack_raw(cx<R> (&s)[12], const RawSite<P>& o) {
  if constexpr (P == WD_F16) {
    cx<float> tmp[12];
    auto& w = through<float>(s, tmp);
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const __half2* h = reinterpret_cast<const __half2*>(&o.v[k]);
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const float2 f = __half22float2(h[j]);
        w[4 * k + j] = mk<float>(f.x * o.s, f.y * o.s);
      }
    }
    convert(s, w);
  } else if constexpr (P == WD_F32) {
    cx<float> tmp[12];
    auto& w = through<float>(s, tmp);
#pragma unroll
    for (int k = 0; k < 6; k++) {
      w[2 * k] = mk<float>(o.v[k].x, o.v[k].y);
      w[2 * k + 1] = mk<float>(o.v[k].z, o.v[k].w);
    }
    convert(s, w);
  } else {
    cx<double> tmp[12];
    auto& w = through<double>(s, tmp);
#pragma unroll
    for (int k = 0; k < 12; k++) w[k] = mk<double>(o.v[k].x, o.v[k].y);
    convert(s, w);
  }
}

// An FP16 site: the values scaled by the site's largest |real component| m,
// rounded to half, and m as the site scale.  KEEP: s is overwritten with
// what was stored (the rounded values times m, as load_spinor_rw would read
// them back), for a norm or dot product of the stored field.
template <typename R, bool KEEP>
__device__ __forceinline__ void store_spinor_f16(void* base, int cb, int Vh_pad, cx<R> (&s)[12]) {
  float m = 0.f;
  cx<float> tmp[12];
  auto& w = through<float>(s, tmp);
  convert(w, s);
#pragma unroll
  for (int k = 0; k < 12; k++) m = fmaxf(m, fmaxf(fabsf(w[k].r), fabsf(w[k].i)));
  float inv = m > 0.f ? 1.0f / m : 0.f;
  int4* p = (int4*)base;
  float* sc = (float*)((char*)base + (size_t)Vh_pad * 48);
#pragma unroll
  for (int k = 0; k < 3; k++) {
    int4 v;
    __half2* h = reinterpret_cast<__half2*>(&v);
#pragma unroll
    for (int j = 0; j < 4; j++) {
      h[j] = __floats2half2_rn(w[4 * k + j].r * inv, w[4 * k + j].i * inv);
      if constexpr (KEEP) {
        const float2 f = __half22float2(h[j]);
        s[4 * k + j] = mk<R>((R)(f.x * m), (R)(f.y * m));
      }
    }
    p[sbi(cb, k, 3)] = v;
  }
  sc[cb] = m;
}

template <int P, typename R>
__device__ __forceinline__ void store_spinor(void* base, int cb, int Vh_pad,
                                             const cx<R> (&site)[12]) {
  cx<R>(&s)[12] = const_cast<cx<R>(&)[12]>(site);  // (not written)
  if constexpr (P == WD_F64) {
    double2* p = (double2*)base;
    cx<double> tmp[12];
    auto& w = through<double>(s, tmp);
    convert(w, s);
#pragma unroll
    for (int k = 0; k < 12; k++) p[sbi(cb, k, 12)] = make_double2(w[k].r, w[k].i);
  } else if constexpr (P == WD_F32) {
    float4* p = (float4*)base;
    cx<float> tmp[12];
    auto& w = through<float>(s, tmp);
    convert(w, s);
#pragma unroll
    for (int k = 0; k < 6; k++)
      p[sbi(cb, k, 6)] = make_float4(w[2 * k].r, w[2 * k].i, w[2 * k + 1].r, w[2 * k + 1].i);
  } else {
    store_spinor_f16<R, false>(base, cb, Vh_pad, s);
  }
}

// ---------------------------------------------------------------------------
// packed gauge formats: 8 regions (mu, parity of the base site), region
// r = 2*mu + par holds Vh_pad sites.
//   (F64,18): 9 double2 (row-major entries)     (F64,12): 6 double2 (rows 0,1)
//   (F32,18): 9 float2                           (F32,12): 3 float4 (rows 0,1)
//   (F16,12): 1 int4 (U00 U01 U02 U10 as half2) in the first 8 regions, then
//             1 int2 (U11 U12) in 8 more regions
// ---------------------------------------------------------------------------

inline size_t link_bytes(int prec, int recon) {
  if (prec == WD_F64) return recon == 18 ? 144 : 96;
  if (prec == WD_F32) return recon == 18 ? 72 : 48;
  if (prec == WD_F16 && recon == 12) return 24;
  return 0;
}

inline size_t gauge_bytes(const Geom& g, int prec, int recon) {
  return round_up((size_t)8 * g.Vh_pad * link_bytes(prec, recon), 256);
}

// rebuild row 2 of an SU(3) matrix from rows 0 and 1: row2 = conj(row0 x row1)
template <typename R>
__device__ __forceinline__ void reconstruct_row2(cx<R> (&u)[9]) {
  u[6] = conj_cross(u[1], u[5], u[2], u[4]);
  u[7] = conj_cross(u[2], u[3], u[0], u[5]);
  u[8] = conj_cross(u[0], u[4], u[1], u[3]);
}

template <int P, int RC, typename R>
__device__ __forceinline__ void load_link(cx<R> (&u)[9], const void* gauge, int region, int cb,
                                          int Vh_pad) {
  if constexpr (P == WD_F64) {
    constexpr int NC = RC == 18 ? 9 : 6;
    const double2* p = (const double2*)gauge + (size_t)region * Vh_pad * NC;
#pragma unroll
    for (int k = 0; k < NC; k++) {
      double2 v = __ldg(p + sbi(cb, k, NC));
      u[k] = mk<R>((R)v.x, (R)v.y);
    }
  } else if constexpr (P == WD_F32) {
    if constexpr (RC == 18) {
      const float2* p = (const float2*)gauge + (size_t)region * Vh_pad * 9;
#pragma unroll
      for (int k = 0; k < 9; k++) {
        float2 v = __ldg(p + sbi(cb, k, 9));
        u[k] = mk<R>((R)v.x, (R)v.y);
      }
    } else {
      const float4* p = (const float4*)gauge + (size_t)region * Vh_pad * 3;
#pragma unroll
      for (int k = 0; k < 3; k++) {
        float4 v = __ldg(p + sbi(cb, k, 3));
        u[2 * k] = mk<R>((R)v.x, (R)v.y);
        u[2 * k + 1] = mk<R>((R)v.z, (R)v.w);
      }
    }
  } else {
    const int4* pa = (const int4*)gauge + (size_t)region * Vh_pad;
    const int2* pb = (const int2*)((const char*)gauge + (size_t)8 * Vh_pad * 16) + (size_t)region * Vh_pad;
    int4 a = __ldg(pa + sbi(cb, 0, 1));
    int2 b = __ldg(pb + sbi(cb, 0, 1));
    const __half2* ha = reinterpret_cast<const __half2*>(&a);
    const __half2* hb = reinterpret_cast<const __half2*>(&b);
#pragma unroll
    for (int j = 0; j < 4; j++) {
      float2 f = __half22float2(ha[j]);
      u[j] = mk<R>((R)f.x, (R)f.y);
    }
#pragma unroll
    for (int j = 0; j < 2; j++) {
      float2 f = __half22float2(hb[j]);
      u[4 + j] = mk<R>((R)f.x, (R)f.y);
    }
  }
  if constexpr (RC == 12) reconstruct_row2(u);
}

// ---------------------------------------------------------------------------
// deterministic FP64 reduction: block tree -> per-block partials -> the last
// block to finish sums the partials in a fixed order and calls `fin`.
// ---------------------------------------------------------------------------

struct RedScratch {
  double* partials;    // >= gridDim.x * N doubles
  unsigned* counter;   // zero between kernels; reset by the last block
};

// Sum over the BS threads of a block (1-, 2- or 3-dimensional; warps are
// taken in linear thread order), in the type T.  The total is in every
// thread of warp 0.
template <int N, int BS, typename T = double>
__device__ __forceinline__ void block_sum(T (&v)[N], T* smem /* N * BS/32 */) {
  const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
  const int lane = tid & 31, warp = tid >> 5;
#pragma unroll
  for (int j = 0; j < N; j++) {
    T t = v[j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    v[j] = t;
  }
  __syncthreads();
  if (lane == 0) {
#pragma unroll
    for (int j = 0; j < N; j++) smem[j * (BS / 32) + warp] = v[j];
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int j = 0; j < N; j++) {
      T t = lane < BS / 32 ? smem[j * (BS / 32) + lane] : (T)0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      v[j] = t;
    }
  }
}

// Sum over the BS threads of a block in FP64, in a fixed order, with few
// additions per scheduler: halves of the block are folded through shared
// memory until one warp is left.  The total is in thread 0.
template <int N, int BS>
__device__ __forceinline__ void sum_threads(double (&v)[N], double (*smem)[BS]) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int half = BS / 2; half >= 32; half /= 2) {
    if (tid >= half && tid < 2 * half) {
#pragma unroll
      for (int j = 0; j < N; j++) smem[j][tid] = v[j];
    }
    __syncthreads();
    if (tid < half) {
#pragma unroll
      for (int j = 0; j < N; j++) v[j] += smem[j][tid + half];
    }
  }
  if (tid < 32) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int j = 0; j < N; j++) v[j] += __shfl_xor_sync(0xffffffffu, v[j], o);
  }
}

// v[j] = sum over k < n of p[k stride + j], this thread's k = threadIdx.x + i BS,
// loaded twelve at a time before they are added.  (A jump into the additions,
// not a condition on each: an FP64 addition that is predicated off still takes
// its 64 cycles.)
template <int N, int BS>
__device__ __forceinline__ void sum_strided(double (&v)[N], const double* __restrict__ p, int n,
                                            int stride) {
#pragma unroll
  for (int j = 0; j < N; j++) v[j] = 0.0;
  for (int k0 = threadIdx.x; k0 < n; k0 += 12 * BS) {
    double w[12][N];
#pragma unroll
    for (int c = 0; c < 12; c++)
#pragma unroll
      for (int j = 0; j < N; j++)
        if (k0 + c * BS < n) w[c][j] = __ldcg(p + (size_t)(k0 + c * BS) * stride + j);
    auto add = [&](int c) {
#pragma unroll
      for (int j = 0; j < N; j++) v[j] += w[c][j];
    };
    const int here = (n - k0 + BS - 1) / BS;
    if (k0 < BS) {
#pragma unroll
      for (int j = 0; j < N; j++) v[j] = w[0][j];
    } else {
      add(0);
    }
    switch (here < 12 ? here : 12) {
      case 12: add(11); [[fallthrough]];
      case 11: add(10); [[fallthrough]];
      case 10: add(9); [[fallthrough]];
      case 9: add(8); [[fallthrough]];
      case 8: add(7); [[fallthrough]];
      case 7: add(6); [[fallthrough]];
      case 6: add(5); [[fallthrough]];
      case 5: add(4); [[fallthrough]];
      case 4: add(3); [[fallthrough]];
      case 3: add(2); [[fallthrough]];
      case 2: add(1); [[fallthrough]];
      default: break;
    }
  }
}

// The block's share of a grid sum, without the cross-block step: the block
// sums v in T and thread 0 stores its N totals as FP64 partials.  A separate
// launch that follows the kernel in its stream (sum_block_partials) adds the
// partials in block order.  Unlike grid_reduce, no block waits for an atomic
// round trip before it exits.
template <int N, int BS, typename T>
__device__ __forceinline__ void block_partials(T (&v)[N], double* partials) {
  __shared__ T smem[N * (BS / 32)];
  block_sum<N, BS, T>(v, smem);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int j = 0; j < N; j++) partials[(size_t)blockIdx.x * N + j] = (double)v[j];
  }
}

// Returns true in every thread of the last block; there `tot` holds the grid
// total in thread 0.  The block sums in T (the
// kernel's working precision), the block partials in FP64.
template <int N, int BS, typename T = double>
__device__ __forceinline__ bool grid_reduce(T (&v)[N], RedScratch rs, double (&tot)[N]) {
  // (more than four sums do not get a word per thread of shared memory)
  constexpr bool FOLD = N <= 4;
  __shared__ double smem[N][FOLD ? BS : BS / 32];
  __shared__ bool last;
  if constexpr (FOLD && std::is_same<T, double>::value)
    sum_threads<N, BS>(v, smem);
  else
    block_sum<N, BS, T>(v, reinterpret_cast<T*>(smem));
  if (threadIdx.x == 0) {
#pragma unroll
    for (int j = 0; j < N; j++) rs.partials[(size_t)blockIdx.x * N + j] = (double)v[j];
    // one acquire-release arrival: it orders the partials written above
    // before it for the last block, and that block's reads after it
    unsigned t;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;"
                 : "=r"(t) : "l"(rs.counter) : "memory");
    last = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double acc[N];
  if constexpr (FOLD) {
    sum_strided<N, BS>(acc, rs.partials, (int)gridDim.x, N);
  } else {
#pragma unroll
    for (int j = 0; j < N; j++) acc[j] = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += BS)
#pragma unroll
      for (int j = 0; j < N; j++) acc[j] += __ldcg(rs.partials + (size_t)b * N + j);
  }
  if constexpr (FOLD)
    sum_threads<N, BS>(acc, smem);
  else
    block_sum<N, BS>(acc, &smem[0][0]);
#pragma unroll
  for (int j = 0; j < N; j++) tot[j] = acc[j];
  if (threadIdx.x == 0) *rs.counter = 0u;
  return true;
}

}  // namespace wd
