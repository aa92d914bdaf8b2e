// Field layout conversions (canonical FP64 <-> packed, precision changes) and
// the BLAS-like vector kernels with FP64 reductions.  The paper's solver is a
// sequence of kernels: Dslash, a dot product whose global sum is done on the
// GPU in double precision by parallel reduction, and BLAS-like updates
// (section "Wilson inverter: Main features").  Reductions here are two-level
// and deterministic: fixed grid, fixed tree inside a block, and a fixed-order
// sum of the per-block partials, either by the last block to finish
// (grid_reduce: wd_norm2, wd_cdot) or by a one-CTA launch that follows the
// kernel in its stream (sum_block_partials: the fused norms of the solvers).
#include "wd_internal.h"

namespace wd {

// ---------------------------------------------------------------------------
// library state shared by the translation units
// ---------------------------------------------------------------------------

State& state() {
  static State s;
  return s;
}

int num_sms() {
  State& s = state();
  if (s.num_sms == 0) {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    s.num_sms = n > 0 ? n : 1;
  }
  return s.num_sms;
}

size_t l2_bytes() {
  State& s = state();
  if (s.l2_bytes == 0) {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrL2CacheSize, dev);
    s.l2_bytes = n > 0 ? (size_t)n : 1;
  }
  return s.l2_bytes;
}

int blas_grid(long long n, int bs) {
  long long need = (n + bs - 1) / bs;
  long long cap = (long long)num_sms() * (2048 / bs);
  if (need < 1) need = 1;
  return (int)(need < cap ? need : cap);
}

cudaError_t ensure_scratch(size_t doubles) {
  State& s = state();
  if (!s.counter) {
    cudaError_t e = device_malloc(&s.counter, 256);
    if (e != cudaSuccess) return e;
    e = cudaMemset(s.counter, 0, 256);
    if (e != cudaSuccess) return e;
  }
  if (doubles <= s.partials_cap) return cudaSuccess;
  size_t cap = doubles < 65536 ? 65536 : doubles;
  if (s.partials) {
    cudaDeviceSynchronize();
    cudaFree(s.partials);
    s.partials = nullptr;
    s.partials_cap = 0;
  }
  cudaError_t e = device_malloc(&s.partials, cap * sizeof(double));
  if (e != cudaSuccess) return e;
  s.partials_cap = cap;
  return cudaSuccess;
}

bool drop_nn_scratch() {
  State& s = state();
  if (s.nn_scratch_taken.exchange(true)) return false;
  const bool had = s.nn_scratch != nullptr;
  if (had) cudaFree(s.nn_scratch);
  s.nn_scratch = nullptr;
  s.nn_scratch_bytes = 0;
  s.nn_scratch_taken.store(false);
  return had;
}

cudaError_t device_malloc(void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes);
  if (e == cudaErrorMemoryAllocation && drop_nn_scratch()) e = cudaMalloc(p, bytes);
  if (e != cudaSuccess) cudaGetLastError();  // (returned here: not to the next launch's check)
  return e;
}

cudaError_t device_flag(int** flag, cudaStream_t st) {
  State& s = state();
  if (!s.dev_flag) {
    cudaError_t e = device_malloc(&s.dev_flag, 256);
    if (e != cudaSuccess) return e;
  }
  *flag = s.dev_flag;
  return cudaMemsetAsync(s.dev_flag, 0, sizeof(int), st);
}

// The cross-block step of block_partials: one CTA, a fixed order.  FP64
// additions bound it: each of a warp holds its scheduler for 64 cycles, and
// the two warps of a scheduler take turns.  So the partials are loaded first,
// a thread adds only what it holds (sum_strided), and the threads' sums
// meet through shared memory (one addition per halving, by half of the warps)
// before the last warp's tree.  2592 partials: 26 additions on a scheduler's
// path, where zero-initialised chains and a tree in every warp took 54; CG
// iteration (three such sums), FP16: 24^3x48 115.5 -> 111.8 us, 16^3x32 38.0 ->
// 35.2, 8^4 26.9 -> 24.7.
template <int N>
__global__ void __launch_bounds__(256) sum_blocks_kernel(const double* __restrict__ partials,
                                                         int nblocks, SumOut out) {
  constexpr int BS = 256;
  __shared__ double smem[N][BS];
  pdl_begin();
  double acc[N];
  sum_strided<N, BS>(acc, partials, nblocks, N);
  sum_threads<N, BS>(acc, smem);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int j = 0; j < N; j++)
      if (out.p[j]) *out.p[j] = acc[j];
  }
}

cudaError_t sum_block_partials(int n, const double* partials, int nblocks, SumOut out,
                               cudaStream_t st, bool plain) {
  const dim3 g(1), b(256);
  switch (n) {
    case 1: return launch_with(!plain, sum_blocks_kernel<1>, g, b, st, partials, nblocks, out);
    case 2: return launch_with(!plain, sum_blocks_kernel<2>, g, b, st, partials, nblocks, out);
    case 3: return launch_with(!plain, sum_blocks_kernel<3>, g, b, st, partials, nblocks, out);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t sum_block_partials(int n, const double* partials, int nblocks, double* out,
                               cudaStream_t st, bool plain) {
  SumOut o = {{out, n > 1 ? out + 1 : nullptr, n > 2 ? out + 2 : nullptr}};
  return sum_block_partials(n, partials, nblocks, o, st, plain);
}

RedScratch scratch() {
  RedScratch r;
  r.partials = state().partials;
  r.counter = state().counter;
  return r;
}

// ---------------------------------------------------------------------------
// canonical <-> packed spinors
// ---------------------------------------------------------------------------

__device__ __forceinline__ int lex_parity(int i, const Geom& g) {
  const int r0 = fdiv(i >> 1, g.dLh0);  // i / L0 (L0 is even)
  const int r1 = fdiv(r0, g.dL1);
  const int x3 = fdiv(r1, g.dL2);
  return (i + (r0 - r1 * g.L[1]) + (r1 - x3 * g.L[2]) + x3) & 1;
}

// The canonical side of the conversions holds 192 (spinor) or 144 (link)
// consecutive bytes per site, which one thread per site would touch 16 bytes
// at a time, 192 or 144 bytes apart from its neighbour: a warp's request then
// covers 32 sectors half full.  Here a warp moves its 32 sites between
// canonical memory and shared memory in whole lines, and each thread takes
// its site from there (an odd number of 16-byte words per site, so that the
// eight lanes of a phase use different banks).  The packing kernels copy the
// next 32 sites (cp.async, no registers) while they convert the current ones.
//
// 24^3x48, us, one thread per site on canonical memory (and conversions on the
// FP64 pipe, wd_common.cuh) -> now:
//   links   F32 12-real 90 -> 80, 18-real 101 -> 88; F16 90 -> 72;
//           F64 12-real 114 -> 98, 18-real 144 -> 116   (HBM: 75 for F32 12-real)
//   pack    F32 42 -> 35, F16 34 -> 32, F64 46 -> 41     (28 for F32)
//   unpack  F32 88 -> 33, F16 94 -> 29, F64 106 -> 49    (28 for F32)
// Without the asynchronous copies the links of F32 18-real took 127.
constexpr int CANON_BS = 96;  // three warps: two buffers each within 48 KB

__device__ __forceinline__ void cp_async16(double2* dst, const double2* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
// all but the newest N groups of this thread have arrived
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" :: "n"(N) : "memory");
}

// NC of every SW canonical words of the sites i0 .. i0 + 31 (below n), NS
// words apart in w
template <int NC, int SW, int NS>
__device__ __forceinline__ void stage_sites(double2* w, const double2* src, long long i0,
                                            long long n, int lane) {
  if (i0 < n) {
    const int words = NC * (int)(n - i0 < 32 ? n - i0 : 32);
#pragma unroll
    for (int j = 0; j < NC; j++) {
      const int e = lane + 32 * j;
      if (e < words) cp_async16(w + e / NC * NS + e % NC, src + (i0 + e / NC) * SW + e % NC);
    }
  }
  cp_async_commit();
}

// src: canonical complex double [n][12]; half layout (full = 0) indexes by cb,
// full layout (full = 1) by lexicographic site.
template <int P>
__global__ void __launch_bounds__(CANON_BS)
    pack_spinor_kernel(char* dst, const double2* __restrict__ src, Geom g, int full,
                       size_t half_bytes) {
  __shared__ double2 sm[CANON_BS / 32][2][32 * 13];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long n = full ? 2LL * g.Vh : g.Vh;
  const long long step = (long long)gridDim.x * CANON_BS;
  long long i0 = blockIdx.x * (long long)CANON_BS + 32 * warp;
  stage_sites<12, 12, 13>(sm[warp][0], src, i0, n, lane);
  for (int b = 0; i0 < n; i0 += step, b ^= 1) {
    stage_sites<12, 12, 13>(sm[warp][b ^ 1], src, i0 + step, n, lane);
    cp_async_wait<1>();
    __syncwarp();
    const double2* w = sm[warp][b];
    const long long i = i0 + lane;
    if (i < n) {
      const int cb = full ? (int)(i >> 1) : (int)i;
      const int par = full ? lex_parity((int)i, g) : 0;
      cx<double> s[12];
#pragma unroll
      for (int k = 0; k < 12; k++) {
        const double2 q = w[lane * 13 + k];
        s[k] = mk<double>(q.x, q.y);
      }
      store_spinor<P, double>(dst + par * half_bytes, cb, g.Vh_pad, s);
    }
    __syncwarp();  // (the next copy into this buffer follows)
  }
}

template <int P>
__global__ void __launch_bounds__(CANON_BS)
    unpack_spinor_kernel(double2* dst, const char* __restrict__ src, Geom g, int full,
                         size_t half_bytes) {
  __shared__ double2 sm[CANON_BS / 32][32 * 13];
  const int lane = threadIdx.x & 31;
  double2* w = sm[threadIdx.x >> 5];
  const long long n = full ? 2LL * g.Vh : g.Vh;
  const long long step = (long long)gridDim.x * CANON_BS;
  for (long long i0 = blockIdx.x * (long long)CANON_BS + (threadIdx.x & ~31); i0 < n; i0 += step) {
    const int words = 12 * (int)(n - i0 < 32 ? n - i0 : 32);
    const long long i = i0 + lane;
    if (i < n) {
      const int cb = full ? (int)(i >> 1) : (int)i;
      const int par = full ? lex_parity((int)i, g) : 0;
      cx<double> s[12];
      load_spinor_rw<P, double>(s, src + par * half_bytes, cb, g.Vh_pad);
#pragma unroll
      for (int k = 0; k < 12; k++) w[lane * 13 + k] = make_double2(s[k].r, s[k].i);
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 12; j++) {
      const int e = lane + 32 * j;
      if (e < words) dst[i0 * 12 + e] = w[e + e / 12];
    }
    __syncwarp();
  }
}

#define WD_PREC_SWITCH(prec, F, ...)                  \
  switch (prec) {                                      \
    case WD_F64: F<WD_F64><<<__VA_ARGS__; break;       \
    case WD_F32: F<WD_F32><<<__VA_ARGS__; break;       \
    case WD_F16: F<WD_F16><<<__VA_ARGS__; break;       \
    default: return cudaErrorInvalidValue;             \
  }

cudaError_t pack_spinor(void* dst, const double* src, const Geom& g, int parity, int prec,
                        cudaStream_t st) {
  int full = parity == WD_FULL;
  long long n = full ? 2LL * g.Vh : g.Vh;
  int grid = blas_grid(n, CANON_BS);
  size_t hb = spinor_half_bytes(g, prec);
  WD_PREC_SWITCH(prec, pack_spinor_kernel, grid, CANON_BS, 0, st>>>((char*)dst, (const double2*)src, g,
                                                                full, hb))
  return cudaGetLastError();
}

cudaError_t unpack_spinor(double* dst, const void* src, const Geom& g, int parity, int prec,
                          cudaStream_t st) {
  int full = parity == WD_FULL;
  long long n = full ? 2LL * g.Vh : g.Vh;
  int grid = blas_grid(n, CANON_BS);
  size_t hb = spinor_half_bytes(g, prec);
  WD_PREC_SWITCH(prec, unpack_spinor_kernel, grid, CANON_BS, 0, st>>>((double2*)dst, (const char*)src,
                                                                  g, full, hb))
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// gauge packing
// ---------------------------------------------------------------------------

// the RC / 2 stored entries of a link
template <int P, int RC>
__device__ __forceinline__ void store_link(char* gauge, int region, int cb, int Vh_pad,
                                           const cx<double> (&u)[RC / 2]) {
  if constexpr (P == WD_F64) {
    constexpr int NC = RC / 2;
    double2* p = (double2*)gauge + (size_t)region * Vh_pad * NC;
#pragma unroll
    for (int k = 0; k < NC; k++) p[sbi(cb, k, NC)] = make_double2(u[k].r, u[k].i);
    return;
  }
  cx<float> w[RC / 2];
  convert(w, u);
  if constexpr (P == WD_F32) {
    if constexpr (RC == 18) {
      float2* p = (float2*)gauge + (size_t)region * Vh_pad * 9;
#pragma unroll
      for (int k = 0; k < 9; k++) p[sbi(cb, k, 9)] = make_float2(w[k].r, w[k].i);
    } else {
      float4* p = (float4*)gauge + (size_t)region * Vh_pad * 3;
#pragma unroll
      for (int k = 0; k < 3; k++)
        p[sbi(cb, k, 3)] = make_float4(w[2 * k].r, w[2 * k].i, w[2 * k + 1].r, w[2 * k + 1].i);
    }
  } else if constexpr (P == WD_F16) {
    int4* pa = (int4*)gauge + (size_t)region * Vh_pad;
    int2* pb = (int2*)(gauge + (size_t)8 * Vh_pad * 16) + (size_t)region * Vh_pad;
    int4 a;
    int2 b;
    __half2* ha = reinterpret_cast<__half2*>(&a);
    __half2* hb = reinterpret_cast<__half2*>(&b);
#pragma unroll
    for (int j = 0; j < 4; j++) ha[j] = __floats2half2_rn(w[j].r, w[j].i);
#pragma unroll
    for (int j = 0; j < 2; j++) hb[j] = __floats2half2_rn(w[4 + j].r, w[4 + j].i);
    pa[sbi(cb, 0, 1)] = a;
    pb[sbi(cb, 0, 1)] = b;
  }
}

// src: canonical [4][V][3][3] complex double; one thread per (mu, site), the
// warp's links staged as the spinors above (of 12-real storage the first two
// rows only)
template <int P, int RC>
__global__ void __launch_bounds__(CANON_BS)
    pack_gauge_kernel(char* dst, const double2* __restrict__ src, Geom g) {
  constexpr int NC = RC / 2, NS = NC | 1;  // words read per link, words between links
  __shared__ double2 sm[CANON_BS / 32][2][32 * NS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long V = 2LL * g.Vh, n = 4 * V;
  const long long step = (long long)gridDim.x * CANON_BS;
  long long t0 = blockIdx.x * (long long)CANON_BS + 32 * warp;
  stage_sites<NC, 9, NS>(sm[warp][0], src, t0, n, lane);
  for (int b = 0; t0 < n; t0 += step, b ^= 1) {
    stage_sites<NC, 9, NS>(sm[warp][b ^ 1], src, t0 + step, n, lane);
    cp_async_wait<1>();
    __syncwarp();
    const double2* w = sm[warp][b];
    const long long t = t0 + lane;
    if (t < n) {
      const int mu = (int)(t / V);
      const int i = (int)(t - mu * V);
      const int par = lex_parity(i, g);
      cx<double> u[NC];
#pragma unroll
      for (int k = 0; k < NC; k++) {
        const double2 q = w[lane * NS + k];
        u[k] = mk<double>(q.x, q.y);
      }
      store_link<P, RC>(dst, 2 * mu + par, i >> 1, g.Vh_pad, u);
    }
    __syncwarp();  // (the next copy into this buffer follows)
  }
}

cudaError_t pack_gauge(void* dst, const double* src, const Geom& g, int prec, int recon,
                       cudaStream_t st) {
  int grid = blas_grid(8LL * g.Vh, CANON_BS);
  const double2* s = (const double2*)src;
  char* d = (char*)dst;
  if (prec == WD_F64 && recon == 18) pack_gauge_kernel<WD_F64, 18><<<grid, CANON_BS, 0, st>>>(d, s, g);
  else if (prec == WD_F64 && recon == 12) pack_gauge_kernel<WD_F64, 12><<<grid, CANON_BS, 0, st>>>(d, s, g);
  else if (prec == WD_F32 && recon == 18) pack_gauge_kernel<WD_F32, 18><<<grid, CANON_BS, 0, st>>>(d, s, g);
  else if (prec == WD_F32 && recon == 12) pack_gauge_kernel<WD_F32, 12><<<grid, CANON_BS, 0, st>>>(d, s, g);
  else if (prec == WD_F16 && recon == 12) pack_gauge_kernel<WD_F16, 12><<<grid, CANON_BS, 0, st>>>(d, s, g);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// precision conversion, BLAS and reductions (nh halves of Vh sites each)
// ---------------------------------------------------------------------------

template <int PD, int PS>
__global__ void convert_kernel(char* dst, const char* __restrict__ src, Geom g, int nh,
                               size_t dhb, size_t shb) {
  long long n = (long long)nh * g.Vh;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    int h = (int)(i / g.Vh), cb = (int)(i - (long long)h * g.Vh);
    using R = typename std::conditional<PD == WD_F64 || PS == WD_F64, double, float>::type;
    cx<R> s[12];
    load_spinor_rw<PS, R>(s, src + h * shb, cb, g.Vh_pad);
    store_spinor<PD, R>(dst + h * dhb, cb, g.Vh_pad, s);
  }
}

cudaError_t convert_spinor(void* dst, int dprec, const void* src, int sprec, const Geom& g, int nh,
                           cudaStream_t st) {
  int grid = blas_grid((long long)nh * g.Vh, 256);
  size_t dhb = spinor_half_bytes(g, dprec), shb = spinor_half_bytes(g, sprec);
  char* d = (char*)dst;
  const char* s = (const char*)src;
#define WD_CV(A, B)                                                                 \
  if (dprec == A && sprec == B) {                                                   \
    convert_kernel<A, B><<<grid, 256, 0, st>>>(d, s, g, nh, dhb, shb);              \
    return cudaGetLastError();                                                      \
  }
  WD_CV(WD_F64, WD_F64) WD_CV(WD_F64, WD_F32) WD_CV(WD_F64, WD_F16)
  WD_CV(WD_F32, WD_F64) WD_CV(WD_F32, WD_F32) WD_CV(WD_F32, WD_F16)
  WD_CV(WD_F16, WD_F64) WD_CV(WD_F16, WD_F32) WD_CV(WD_F16, WD_F16)
#undef WD_CV
  return cudaErrorInvalidValue;
}

// The reductions and axpby stream their fields once on a grid of resident
// CTAs (resident_grid); each thread loads its next site, as raw words, before
// it computes the current one.  Sums over sites are FP64: one conversion and
// one addition per site, and the block tree once per thread, which with a
// thread per site was most of the time (GB300's FP64 rate is 1/64 of FP32's).
// They overlap their launch with the previous kernel's end (pdl_begin).
// us per call on 24^3x48, FP32: norm2 13.1 -> 7.7, cdot 20.6 -> 9.5, axpby 10.3
// -> 7.7; on 8^4 7.0 -> 4.6, 8.4 -> 5.9, 4.5 -> 4.3.

// site i of nh halves
template <int P>
__device__ __forceinline__ void load_site(RawSite<P>& o, const char* x, long long i, const Geom& g,
                                          size_t hb) {
  const bool odd = i >= g.Vh;
  load_raw<P>(o, odd ? x + hb : x, (int)(odd ? i - g.Vh : i), g.Vh_pad);
}

constexpr int RED_BS = 256;

template <int P>
__global__ void __launch_bounds__(RED_BS) norm2_kernel(double* res, const char* __restrict__ x,
                                                       Geom g, int nh, size_t hb, RedScratch rs) {
  using R = real_of<P>;
  pdl_begin();
  const long long n = (long long)nh * g.Vh, step = (long long)gridDim.x * RED_BS;
  double acc[1] = {0.0};
  long long i = blockIdx.x * (long long)RED_BS + threadIdx.x;
  RawSite<P> a;
  if (i < n) load_site<P>(a, x, i, g, hb);
  for (; i < n; i += step) {
    RawSite<P> na;
    if (i + step < n) load_site<P>(na, x, i + step, g, hb);
    asm volatile("" ::: "memory");  // the next site's loads are issued here
    cx<R> s[12];
    unpack_raw<P, R>(s, a);
    acc[0] += site_norm2(s);
    a = na;
  }
  double tot[1];
  if (grid_reduce<1, RED_BS>(acc, rs, tot) && threadIdx.x == 0) res[0] = tot[0];
}

template <int P>
__global__ void __launch_bounds__(RED_BS) cdot_kernel(double* res, const char* __restrict__ x,
                                                      const char* __restrict__ y, Geom g, int nh,
                                                      size_t hb, RedScratch rs) {
  using R = real_of<P>;
  pdl_begin();
  const long long n = (long long)nh * g.Vh, step = (long long)gridDim.x * RED_BS;
  double acc[2] = {0.0, 0.0};
  long long i = blockIdx.x * (long long)RED_BS + threadIdx.x;
  RawSite<P> a, b;
  if (i < n) {
    load_site<P>(a, x, i, g, hb);
    load_site<P>(b, y, i, g, hb);
  }
  for (; i < n; i += step) {
    RawSite<P> na, nb;
    if (i + step < n) {
      load_site<P>(na, x, i + step, g, hb);
      load_site<P>(nb, y, i + step, g, hb);
    }
    asm volatile("" ::: "memory");
    cx<R> u[12], v[12];
    unpack_raw<P, R>(u, a);
    unpack_raw<P, R>(v, b);
    site_cdot(u, v, acc[0], acc[1]);
    a = na;
    b = nb;
  }
  double tot[2];
  if (grid_reduce<2, RED_BS>(acc, rs, tot) && threadIdx.x == 0) {
    res[0] = tot[0];
    res[1] = tot[1];
  }
}

template <int P>
__global__ void __launch_bounds__(RED_BS) axpby_kernel(double a, const char* __restrict__ x,
                                                       double b, char* y, Geom g, int nh,
                                                       size_t hb) {
  using R = real_of<P>;
  pdl_begin();
  const long long n = (long long)nh * g.Vh, step = (long long)gridDim.x * RED_BS;
  const R ra = (R)a, rb = (R)b;
  // b = 0: y is output only and never read (BLAS convention), so an
  // uninitialised y cannot leak NaN or Inf through 0 * y
  const bool read_y = b != 0.0;
  auto update = [&](cx<R>(&u)[12], cx<R>(&v)[12]) {
    if (read_y) {
#pragma unroll
      for (int k = 0; k < 12; k++) {
        v[k].r = ra * u[k].r + rb * v[k].r;
        v[k].i = ra * u[k].i + rb * v[k].i;
      }
    } else {
#pragma unroll
      for (int k = 0; k < 12; k++) v[k] = mk<R>(ra * u[k].r, ra * u[k].i);
    }
  };
  long long i = blockIdx.x * (long long)RED_BS + threadIdx.x;
  RawSite<P> p, q;
  if (i < n) {
    load_site<P>(p, x, i, g, hb);
    if (read_y) load_site<P>(q, y, i, g, hb);
  }
  for (; i < n; i += step) {
    RawSite<P> np, nq;
    if (i + step < n) {
      load_site<P>(np, x, i + step, g, hb);
      if (read_y) load_site<P>(nq, y, i + step, g, hb);
    }
    cx<R> u[12], v[12];
    unpack_raw<P, R>(u, p);
    if (read_y) unpack_raw<P, R>(v, q);
    update(u, v);
    const bool odd = i >= g.Vh;
    store_spinor<P, R>(odd ? y + hb : y, (int)(odd ? i - g.Vh : i), g.Vh_pad, v);
    p = np;
    q = nq;
  }
}

// FP64 axpby: bound by the FP64 pipe, and fastest with the site's elements
// loaded as they are used (34 registers, eight CTAs per SM): loading ahead
// takes 210 registers and 45 us on 24^3x48, a site at a time 106 and 39,
// against 35.  It does not overlap its launch: the next grid's CTAs then crowd
// on the SMs that have room (16^3x32: 22 us against 10).
__global__ void axpby_f64_kernel(double a, const char* __restrict__ x, double b, char* y, Geom g,
                                 int nh, size_t hb) {
  const long long n = (long long)nh * g.Vh;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int h = (int)(i / g.Vh), cb = (int)(i - (long long)h * g.Vh);
    cx<double> u[12], v[12];
    load_spinor_rw<WD_F64, double>(u, x + h * hb, cb, g.Vh_pad);
    if (b != 0.0) {
      load_spinor_rw<WD_F64, double>(v, y + h * hb, cb, g.Vh_pad);
#pragma unroll
      for (int k = 0; k < 12; k++) {
        v[k].r = a * u[k].r + b * v[k].r;
        v[k].i = a * u[k].i + b * v[k].i;
      }
    } else {
#pragma unroll
      for (int k = 0; k < 12; k++) v[k] = mk<double>(a * u[k].r, a * u[k].i);
    }
    store_spinor<WD_F64, double>(y + h * hb, cb, g.Vh_pad, v);
  }
}

template <int P>
static cudaError_t norm2_p(double* res, const void* x, const Geom& g, int nh, cudaStream_t st) {
  static const int per_sm = ctas_per_sm(norm2_kernel<P>);
  const int grid = resident_grid(per_sm, (long long)nh * g.Vh);
  cudaError_t e = ensure_scratch((size_t)grid * 2);
  if (e != cudaSuccess) return e;
  // (FP64 on a part-filled GPU: 11.5 us overlapped, 10.4 plain on 16^3x32)
  return launch_with(P != WD_F64 || grid == per_sm * num_sms(), norm2_kernel<P>, dim3(grid),
                     dim3(RED_BS), st, res, (const char*)x, g, nh, spinor_half_bytes(g, P),
                     scratch());
}
template <int P>
static cudaError_t cdot_p(double* res, const void* x, const void* y, const Geom& g, int nh,
                          cudaStream_t st) {
  static const int per_sm = ctas_per_sm(cdot_kernel<P>);
  const int grid = resident_grid(per_sm, (long long)nh * g.Vh);
  cudaError_t e = ensure_scratch((size_t)grid * 2);
  if (e != cudaSuccess) return e;
  return launch_pdl(cdot_kernel<P>, dim3(grid), dim3(RED_BS), st, res, (const char*)x,
                    (const char*)y, g, nh, spinor_half_bytes(g, P), scratch());
}
template <int P>
static cudaError_t axpby_p(double a, const void* x, double b, void* y, const Geom& g, int nh,
                           cudaStream_t st) {
  static const int per_sm = ctas_per_sm(axpby_kernel<P>);
  const int grid = resident_grid(per_sm, (long long)nh * g.Vh);
  return launch_pdl(axpby_kernel<P>, dim3(grid), dim3(RED_BS), st, a, (const char*)x, b, (char*)y,
                    g, nh, spinor_half_bytes(g, P));
}

cudaError_t norm2(double* res, const void* x, const Geom& g, int prec, int nh, cudaStream_t st) {
  switch (prec) {
    case WD_F64: return norm2_p<WD_F64>(res, x, g, nh, st);
    case WD_F32: return norm2_p<WD_F32>(res, x, g, nh, st);
    case WD_F16: return norm2_p<WD_F16>(res, x, g, nh, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t cdot(double* res, const void* x, const void* y, const Geom& g, int prec, int nh,
                 cudaStream_t st) {
  switch (prec) {
    case WD_F64: return cdot_p<WD_F64>(res, x, y, g, nh, st);
    case WD_F32: return cdot_p<WD_F32>(res, x, y, g, nh, st);
    case WD_F16: return cdot_p<WD_F16>(res, x, y, g, nh, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t axpby(double a, const void* x, double b, void* y, const Geom& g, int prec, int nh,
                  cudaStream_t st) {
  switch (prec) {
    case WD_F64:
      axpby_f64_kernel<<<blas_grid((long long)nh * g.Vh, 256), 256, 0, st>>>(
          a, (const char*)x, b, (char*)y, g, nh, spinor_half_bytes(g, WD_F64));
      return cudaGetLastError();
    case WD_F32: return axpby_p<WD_F32>(a, x, b, y, g, nh, st);
    case WD_F16: return axpby_p<WD_F16>(a, x, b, y, g, nh, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace wd
