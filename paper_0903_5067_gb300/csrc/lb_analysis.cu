// Chain observables of Sec. III A/B computed on the GPU from a device trajectory of unwrapped
// bead positions traj[t][n][3] (FP64): g1, g2, g3 (monomer, monomer-in-CM and centre-of-mass
// mean-square displacements), Rouse modes X_p and their time correlation, static and dynamic
// structure factors S(k), S(k, t) (isotropic: exp(i k.r) averaged over the directions of k is
// sin(kr)/(kr)).
//
// Every output element is a fixed-order sum of one thread block or one or two clusters of
// blocks: threads stride over the summation domain in a fixed pattern and combine in a fixed
// tree, so results are reproducible bit for bit.  No kernel allocates memory; outputs are caller-owned device
// arrays.  All arithmetic is FP64.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/lb.h"
#include "lb_cluster.h"
#include "lb_shared.h"

namespace {

constexpr int kThreads = 256;

// fixed-order block reduction of NV values per thread (result valid in thread 0)
template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV], double (*sh)[kThreads]) {
  const int t = threadIdx.x;
#pragma unroll
  for (int q = 0; q < NV; ++q) sh[q][t] = v[q];
  __syncthreads();
  for (int s = kThreads / 2; s > 0; s >>= 1) {
    if (t < s) {
#pragma unroll
      for (int q = 0; q < NV; ++q) sh[q][t] += sh[q][t + s];
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < NV; ++q) v[q] = sh[q][0];
}

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cluster_blocks() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the double at the same shared-memory location in block `rank` of the cluster
__device__ __forceinline__ double cluster_load(const double* p, unsigned rank) {
  unsigned a, b;
  double v;
  a = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(a), "r"(rank));
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(b) : "memory");
  return v;
}

// two neighbouring doubles (16-byte aligned) in the shared memory of block `rank`; four such loads
// in flight together
struct RemotePair {
  unsigned at;  // shared::cluster address
  __device__ __forceinline__ RemotePair(const double* p, unsigned rank) {
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  }
};
__device__ __forceinline__ void cluster_load4(const RemotePair (&p)[4], double2 (&v)[4]) {
  asm volatile(
      "ld.shared::cluster.v2.f64 {%0, %1}, [%8];\n\tld.shared::cluster.v2.f64 {%2, %3}, [%9];\n\t"
      "ld.shared::cluster.v2.f64 {%4, %5}, [%10];\n\tld.shared::cluster.v2.f64 {%6, %7}, [%11];"
      : "=d"(v[0].x), "=d"(v[0].y), "=d"(v[1].x), "=d"(v[1].y), "=d"(v[2].x), "=d"(v[2].y), "=d"(v[3].x), "=d"(v[3].y)
      : "r"(p[0].at), "r"(p[1].at), "r"(p[2].at), "r"(p[3].at)
      : "memory");
}

__device__ __forceinline__ void centre(const double* __restrict__ f, int N, double c[3]) {
  double s0 = 0, s1 = 0, s2 = 0;
  for (int n = 0; n < N; ++n) {
    s0 += f[3 * n];
    s1 += f[3 * n + 1];
    s2 += f[3 * n + 2];
  }
  c[0] = s0 / N;
  c[1] = s1 / N;
  c[2] = s2 / N;
}

// g1, g2, g3 of one origin pair: frames a and b with centres ca, cb
__device__ __forceinline__ void add_displacements(const double* ca, const double* cb, const double* a0,
                                                  const double* b0, const double* a1, const double* b1, double v[3]) {
  double dcm[3], s3 = 0;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    dcm[q] = cb[q] - ca[q];
    s3 += dcm[q] * dcm[q];
  }
  v[2] += s3;
  double s1 = 0, s2 = 0;
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    const double *fa = w ? a1 : a0, *fb = w ? b1 : b0;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const double d = fb[q] - fa[q];
      s1 += d * d;
      const double dr = d - dcm[q];
      s2 += dr * dr;
    }
  }
  v[0] += s1;
  v[1] += s2;
}

__device__ __forceinline__ void write_msd(const double v[3], int norig, int lag, int nlag, double* out) {
  const bool any = norig > 0;
  out[lag] = any ? v[0] / (2.0 * norig) : 0.0;
  out[nlag + lag] = any ? v[1] / (2.0 * norig) : 0.0;
  out[2 * nlag + lag] = any ? v[2] / norig : 0.0;
}

// The whole run staged in shared memory (kMsdFrames frames at most): a cluster of blocks forms the
// centres of mass once, a warp per frame, each block a share of the frames, and every block
// takes the full series of the centre and the two inner beads (9 doubles per frame) from its
// peers through distributed shared memory.  Then the cluster's lags, one after the other per
// block, origins strided over the threads.  At T = 1000, N = 128, 501 lags 115 us
// (k_msd below, two centres of N beads for every lag and origin with frame-strided reads: 1233 us;
// 19 clusters instead of the 15 that fit at a time: 184 us).
constexpr int kMsdFrames = 3000;
constexpr int kMsdCluster = 8;
constexpr int kMsdThreads = 512;
__global__ void __launch_bounds__(kMsdThreads) k_msd_staged(const double* __restrict__ traj, int T, int N, int i0, int i1,
                                                         double* __restrict__ out, int nlag, int nclusters) {
  extern __shared__ __align__(16) double series[];  // [T][9]: centre, bead i0, bead i1
  __shared__ double ws[3][kMsdThreads / 32];
  const int rank = (int)cluster_rank(), G = (int)cluster_blocks();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = ((T + G - 1) / G + 1) & ~1;  // frames of a block, an even number
  const int f0 = rank * per < T ? rank * per : T, f1 = f0 + per < T ? f0 + per : T;
  for (int t = f0 + warp; t < f1; t += kMsdThreads / 32) {
    const double* f = traj + (size_t)t * N * 3;
    double s[3] = {0, 0, 0};  // s[j]: elements lane + 32 j + 96 m, component (lane + 2 j) mod 3
    for (int e = lane; e < 3 * N; e += 96) {
#pragma unroll
      for (int j = 0; j < 3; ++j)
        if (e + 32 * j < 3 * N) s[j] += f[e + 32 * j];
    }
    double c[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int j = (2 * q + lane) % 3;  // (lane + 2 j) mod 3 = q for j = 2 (q - lane) = 2 q + lane mod 3
      c[q] = j == 0 ? s[0] : (j == 1 ? s[1] : s[2]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) c[q] += __shfl_xor_sync(0xffffffffu, c[q], o);
    }
    if (lane < 9) {
      const int q = lane % 3;
      series[9 * t + lane] = lane < 3 ? (q == 0 ? c[0] : (q == 1 ? c[1] : c[2])) / N : f[3 * (lane < 6 ? i0 : i1) + q];
    }
  }
  cluster_barrier();
  // pairs of doubles, a block's share a whole number of them (`per` is even)
  const int npair = (9 * T + 1) / 2;
  for (int e0 = threadIdx.x; e0 < npair; e0 += 4 * kMsdThreads) {
    const int last = npair - 1;
    const int e[4] = {e0, min(e0 + kMsdThreads, last), min(e0 + 2 * kMsdThreads, last), min(e0 + 3 * kMsdThreads, last)};
    int owner[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) owner[j] = 2 * e[j] / 9 / per;
    const RemotePair from[4] = {{series + 2 * e[0], (unsigned)owner[0]}, {series + 2 * e[1], (unsigned)owner[1]},
                                {series + 2 * e[2], (unsigned)owner[2]}, {series + 2 * e[3], (unsigned)owner[3]}};
    double2 v[4];
    cluster_load4(from, v);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (owner[j] != rank) reinterpret_cast<double2*>(series)[e[j]] = v[j];
  }
  cluster_barrier();  // every share has been read; also the block's barrier
  for (int lag = (int)(blockIdx.x / G) + nclusters * rank; lag < nlag; lag += nclusters * G) {
    const int norig = T - lag;
    double v[3] = {0, 0, 0};
    for (int t0 = threadIdx.x; t0 < norig; t0 += kMsdThreads) {
      const double *a = series + 9 * t0, *b = a + 9 * lag;
      add_displacements(a, b, a + 3, b + 3, a + 6, b + 6, v);
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
      if (lane == 0) ws[q][warp] = v[q];
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        v[q] = 0.0;
        for (int w = 0; w < kMsdThreads / 32; ++w) v[q] += ws[q][w];
      }
      write_msd(v, norig, lag, nlag, out);
    }
    __syncthreads();
  }
}

// Longer runs, and short chains with few lags: one block per lag, origins t0 strided over the threads,
// the centres of both frames formed by each thread
__global__ void __launch_bounds__(kThreads) k_msd(const double* __restrict__ traj, int T, int N, int i0, int i1,
                                                  double* __restrict__ out, int nlag) {
  __shared__ double sh[3][kThreads];
  const int lag = blockIdx.x;
  const int norig = T - lag;
  double v[3] = {0, 0, 0};
  for (int t0 = threadIdx.x; t0 < norig; t0 += kThreads) {
    const double* fa = traj + (size_t)t0 * N * 3;
    const double* fb = traj + (size_t)(t0 + lag) * N * 3;
    double ca[3], cb[3];
    centre(fa, N, ca);
    centre(fb, N, cb);
    add_displacements(ca, cb, fa + 3 * i0, fb + 3 * i0, fa + 3 * i1, fb + 3 * i1, v);
  }
  block_sum<3>(v, sh);
  if (threadIdx.x == 0) write_msd(v, norig, lag, nlag, out);
}

// Rouse modes: X_p(t) = (1/N) sum_n r_n(t) cos(p pi (n - 1/2)/N).  The angles are multiples of
// pi/2N, p (2n - 1) of them, so a table of 4N cosines holds every factor (one cospi each).  66 us
// at T = 1000, N = 128; one cospi per term took 3045 us.  The terms n and N + 1 - n
// have the same factor up to (-1)^p: even modes take the sums of the two beads, odd modes the
// differences, which halves the FP64 operations.  A block takes kRouseFrames frames, a thread
// a mode p of one frame after the other, its three components sharing the factor.
constexpr int kRouseFrames = 4;
__global__ void __launch_bounds__(kThreads) k_rouse_modes(const double* __restrict__ traj, int T, int N, int P,
                                                          double* __restrict__ X) {
  extern __shared__ __align__(16) double rsm[];
  const int H = (N + 1) / 2;  // pairs (n, N + 1 - n), the middle bead of an odd N last
  double* tab = rsm;          // 4N cosines of m pi / 2N
  double* sd = tab + 4 * N;   // [frame][parity][n][3]: sums and differences
  const int t0 = blockIdx.x * kRouseFrames, nf = T - t0 < kRouseFrames ? T - t0 : kRouseFrames;
  for (int m = threadIdx.x; m < 4 * N; m += kThreads) tab[m] = cospi((double)m / (2.0 * (double)N));
  for (int e = threadIdx.x; e < nf * 3 * H; e += kThreads) {
    const int f = e / (3 * H), r = e - f * 3 * H, n = r / 3, q = r - 3 * n;
    const double* fr = traj + (size_t)(t0 + f) * N * 3;
    const double lo = fr[r], hi = fr[3 * (N - 1 - n) + q];
    // the middle bead is its own partner: its difference is 0, or NaN where it is not finite
    sd[(2 * f) * 3 * H + r] = 2 * n + 1 == N ? lo : lo + hi;
    sd[(2 * f + 1) * 3 * H + r] = lo - hi;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < nf * P; e += kThreads) {
    const int f = e / P, p = e - f * P + 1;
    const double* v = sd + (2 * f + (p & 1)) * 3 * H;
    double s0 = 0, s1 = 0, s2 = 0;
    int m = p;  // p (2n - 1) mod 4N
    for (int n = 0; n < H; ++n) {
      const double c = tab[m];
      s0 = fma(v[3 * n], c, s0);
      s1 = fma(v[3 * n + 1], c, s1);
      s2 = fma(v[3 * n + 2], c, s2);
      m += 2 * p;
      if (m >= 4 * N) m -= 4 * N;
    }
    double* x = X + ((size_t)(t0 + f) * P + (p - 1)) * 3;
    x[0] = s0 / N;
    x[1] = s1 / N;
    x[2] = s2 / N;
  }
}
// Longer chains (the table and the frames exceed shared memory): one block per frame, one cospi per
// term
__global__ void __launch_bounds__(kThreads) k_rouse_modes_long(const double* __restrict__ traj, int N, int P,
                                                               double* __restrict__ X) {
  const int t = blockIdx.x;
  const double* f = traj + (size_t)t * N * 3;
  for (int e = threadIdx.x; e < 3 * P; e += kThreads) {
    const int p = 1 + e / 3, q = e % 3;
    double s = 0;
    for (int n = 1; n <= N; ++n) s += f[3 * (n - 1) + q] * cospi((double)p * ((double)n - 0.5) / (double)N);
    X[(size_t)t * P * 3 + e] = s / N;
  }
}

// Correlation of mode p at kCorrLags lags from its series X_p(t) staged in shared memory (three
// component planes; kCorrFrames frames at most): a warp's lanes take 32 consecutive lags, so that
// they read consecutive words and share X_p(t0), and the block's 8 warps an eighth of the origins
// each, added in warp order.  FP64-bound: three multiply-adds per origin and lag, 282 us at T = 1000,
// P = 127, 501 lags (227 us of FP64 pipe; a block per (p, lag) with strided reads 642 us).
constexpr int kCorrLags = 64;
constexpr int kCorrFrames = 9000;
__global__ void __launch_bounds__(kThreads) k_rouse_corr_staged(const double* __restrict__ X, int T, int P,
                                                                double* __restrict__ c, int nlag) {
  extern __shared__ __align__(16) double csm[];  // [3][T]
  __shared__ double part[kThreads / 32][32];
  const int p = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int e = threadIdx.x; e < 3 * T; e += kThreads) {
    const int t = e / 3, q = e - 3 * t;
    csm[q * T + t] = X[((size_t)t * P + p) * 3 + q];
  }
  __syncthreads();
  const int l1 = (int)(blockIdx.y + 1) * kCorrLags < nlag ? (int)(blockIdx.y + 1) * kCorrLags : nlag;
  for (int l0 = blockIdx.y * kCorrLags; l0 < l1; l0 += 32) {
    const int lag = l0 + lane;
    const int longest = T - l0;  // origins of the smallest lag; a lane beyond its own adds nothing
    const int a = warp * longest / (kThreads / 32), b = (warp + 1) * longest / (kThreads / 32);
    const int own = T - lag < b ? T - lag : b;
    double s = 0.0;
    for (int t0 = a; t0 < own; ++t0) {
      const double* x = csm + t0;
      s = fma(x[0], x[lag], s);
      s = fma(x[T], x[T + lag], s);
      s = fma(x[2 * T], x[2 * T + lag], s);
    }
    part[warp][lane] = s;
    __syncthreads();
    if (warp == 0 && lag < l1) {
      s = 0.0;
#pragma unroll
      for (int w = 0; w < kThreads / 32; ++w) s += part[w][lane];
      c[(size_t)p * nlag + lag] = T - lag > 0 ? s / (T - lag) : 0.0;
    }
    __syncthreads();
  }
}

// Longer runs, few lags or few modes: one block per (p, lag)
__global__ void __launch_bounds__(kThreads) k_rouse_corr(const double* __restrict__ X, int T, int P,
                                                         double* __restrict__ c, int nlag) {
  __shared__ double sh[1][kThreads];
  const int p = blockIdx.x, lag = blockIdx.y;
  const int norig = T - lag;
  double v[1] = {0};
  for (int t0 = threadIdx.x; t0 < norig; t0 += kThreads) {
    const double* a = X + ((size_t)t0 * P + p) * 3;
    const double* b = X + ((size_t)(t0 + lag) * P + p) * 3;
    v[0] += b[0] * a[0] + b[1] * a[1] + b[2] * a[2];
  }
  block_sum<1>(v, sh);
  if (threadIdx.x == 0) c[(size_t)p * nlag + lag] = norig > 0 ? v[0] / norig : 0.0;
}

// ---------------------------------------------------------------------------------------
// structure factors and hydrodynamic radius
//
// These sums are bound by the FP64 pipe (2 fused multiply-adds per clock and SM: a warp's
// instruction holds it for 16 clocks), so a pair costs what its FP64 operations cost and
// index arithmetic, conversions by integer operations and table lookups in shared memory are
// nearly free beside them.  Measured at T = 1000, N = 128 (before: one block per output, sqrt,
// sine and division per pair and wave number): S(k) at 16 wave numbers 144.0 -> 6.5 ms, S(k, t) at
// 4 wave numbers and 101 lags 29.1 -> 11.4 ms (83 % of the FP64 pipe's cycles), <1/R_H> 70.4 ->
// 0.86 ms.  A pair takes its distance once for a group of wave numbers (14
// operations: difference, square, 1/r, r) and 14 operations per wave number:
//   sum of sin(k r)/(k r) = (1/k) sum of sin(k r) (1/r),
// the sine from a table of 1024 angles and short polynomials.
//
// Every output is the sum of one cluster of blocks, or of two: each thread walks its pairs in a
// fixed order, each block adds its threads in a fixed tree, and block 0 of the cluster adds the
// blocks in rank order through distributed shared memory.  Two clusters add their sums to the
// zeroed output atomically (0 + a + b in either order is the same number).  So results are
// reproducible and no scratch memory is needed.
// ---------------------------------------------------------------------------------------

// sin and cos of 2 pi n / 1024 for n = 0 .. 511 (n + 512: the negatives)
constexpr int kAngles = 1024;
struct SinTab {
  double2 a[kAngles / 2];  // (sin, cos)
};

// Fill the table with a block of at least 48 threads: 32 coarse and 16 fine angles by
// sincospi, the products by angle addition (four operations per entry instead of a sincospi).
// Ends with a barrier.
__device__ __forceinline__ void fill_sin_table(SinTab* tab, double2* seed /* 48 */) {
  const int t = threadIdx.x;
  if (t < 48) {
    double s, c;
    sincospi(t < 32 ? (double)t / 32.0 : (double)(t - 32) / 512.0, &s, &c);
    seed[t] = make_double2(s, c);
  }
  __syncthreads();
  for (int n = t; n < kAngles / 2; n += blockDim.x) {
    const double2 A = seed[n >> 4], B = seed[32 + (n & 15)];
    tab->a[n] = make_double2(fma(A.x, B.y, A.y * B.x), fma(A.y, B.y, -(A.x * B.x)));
  }
  __syncthreads();
}

// sin(2 pi p / 1024) for |p| < 2^31: p = n + f with n the nearest integer (the sum with
// 1.5 2^52 leaves n in the low mantissa bits; f is exact), sin(n) cos(f) + cos(n) sin(f) with
// the Taylor series of sin and cos - 1 in f (|angle| <= pi/1024: truncation below 2e-18).
__device__ __forceinline__ double sin_turns(double p, const SinTab* __restrict__ tab) {
  constexpr double kMagic = 6755399441055744.0;  // 1.5 2^52
  constexpr double u = 2.0 * M_PI / kAngles;
  const double t = p + kMagic;
  const int n = __double2loint(t);
  const double f = p - (t - kMagic);
  const double2 e = tab->a[n & (kAngles / 2 - 1)];
  const double z = f * f;
  const double sf = f * fma(z, fma(z, u * u * u * u * u / 120.0, -(u * u * u) / 6.0), u);
  const double cf = z * fma(z, u * u * u * u / 24.0, -(u * u) / 2.0);
  const double v = e.x + fma(e.x, cf, e.y * sf);
  return __hiloint2double(__double2hiint(v) ^ (int)(((unsigned)n << 22) & 0x80000000u), __double2loint(v));
}

// 1/sqrt(x) for x in [2^-100, 2^100) (rsqrt_range): the single-precision reciprocal square root of x
// truncated to single precision (rounding and truncation by integer operations: |e| < 1e-6
// below) and one third-order step y (1 + e/2 + 3 e^2/8), e = 1 - x y^2 (next term below 4e-19).
__device__ __forceinline__ double rsqrt_pos(double x) {
  const int hi = __double2hiint(x);
  const unsigned bits = ((unsigned)(hi - (896 << 20)) << 3) | ((unsigned)__double2loint(x) >> 29);
  const unsigned yb = __float_as_uint(rsqrtf(__uint_as_float(bits)));
  const double y = __hiloint2double((int)((yb >> 3) + (896u << 20)), (int)(yb << 29));
  const double e = fma(-(x * y), y, 1.0);
  return fma(y * e, fma(e, 0.375, 0.5), y);
}
constexpr int kRangeLo = (1023 - 100) << 20, kRangeHi = (1023 + 100) << 20;  // high words of the range
__device__ __forceinline__ bool rsqrt_range(double x) {  // also false for NaN and negative x
  return (unsigned)(__double2hiint(x) - kRangeLo) < (unsigned)(kRangeHi - kRangeLo);
}

constexpr int kKGroup = 4;           // most wave numbers of one pass over the pairs
constexpr double kFastArg = 1.0e6;   // largest k r of the table path

// sin(k r)/(k r), and k times it (sin(k r)/r) as the sums of the table path need it; general arguments
__device__ __forceinline__ double sinc(double k, double r2) {
  const double x = k * sqrt(r2);
  return x == 0.0 ? 1.0 : sin(x) / x;
}
__device__ __noinline__ double sinc_general(double k, double r2) { return sinc(k, r2) * k; }

// Wave numbers g0 .. g0 + KG - 1 (the last group repeats the last one) and the squared distances
// [2^-100, r2_end) that take the table path for all of them, as a span of high words: compared
// by integer operations (a comparison in FP64 would cost as much as any other operation).
template <int KG>
struct WaveNumbers {
  double k[KG], kt[KG];
  unsigned span;
  __device__ __forceinline__ WaveNumbers(const double* __restrict__ ks, int nk, int g0) {
    double kmax = 0.0;
#pragma unroll
    for (int g = 0; g < KG; ++g) {
      k[g] = ks[g0 + g < nk ? g0 + g : nk - 1];
      kt[g] = k[g] * (kAngles / (2.0 * M_PI));
      kmax = fabs(k[g]) > 0.0 ? fmax(kmax, fabs(k[g])) : INFINITY;  // k = 0 and NaN: the general path
    }
    const double rmax = kFastArg / kmax;
    const int end = __double2hiint(rmax * rmax);
    span = end <= kRangeLo ? 0u : (unsigned)((end < kRangeHi ? end : kRangeHi) - kRangeLo);
  }
};

// acc[g] += sin(k_g r)/r of one pair at squared distance r2 (k_g where k_g r = 0)
template <int KG>
__device__ __forceinline__ void add_pair(double r2, const WaveNumbers<KG>& w, const SinTab* __restrict__ tab,
                                         double (&acc)[KG]) {
  if ((unsigned)(__double2hiint(r2) - kRangeLo) < w.span) {
    const double y = rsqrt_pos(r2);
    const double s = r2 * y;
    const double r = fma(0.5 * y, fma(-s, s, r2), s);
#pragma unroll
    for (int g = 0; g < KG; ++g) acc[g] = fma(sin_turns(w.kt[g] * r, tab), y, acc[g]);
  } else {
#pragma unroll
    for (int g = 0; g < KG; ++g) acc[g] += sinc_general(w.k[g], r2);
  }
}

// sum of v over the threads of every block of the cluster, in a fixed order; the result in
// thread 0 of block 0.  Every thread of every block calls it once; no block returns before
// block 0 has read its sums.
template <int NV>
__device__ __forceinline__ void cluster_sum(double (&v)[NV], double* warp_sums /* NV x 32 */, double* block_sums /* NV */) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int q = 0; q < NV; ++q) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
    if (lane == 0) warp_sums[q * 32 + warp] = v[q];
  }
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      double s = lane < nw ? warp_sums[q * 32 + lane] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
      if (lane == 0) block_sums[q] = s;
    }
  }
  cluster_barrier();
  if (cluster_rank() == 0 && threadIdx.x == 0) {
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      v[q] = 0.0;
      for (unsigned b = 0; b < cluster_blocks(); ++b) v[q] += cluster_load(block_sums + q, b);
    }
  }
  cluster_barrier();
}

// The pairs i < j of a frame as q = 0 .. N (N - 1)/2 - 1: j = i + d mod N with d = q / N + 1
// and i = q mod N (the last d of an even N has N/2 of them), so that consecutive q read
// consecutive beads.
__device__ __forceinline__ double pair_r2(const double* __restrict__ f, int N, unsigned q) {
  const unsigned d = q / (unsigned)N + 1, i = q % (unsigned)N;
  const unsigned j = i + d < (unsigned)N ? i + d : i + d - (unsigned)N;
  const double dx = f[3 * i] - f[3 * j], dy = f[3 * i + 1] - f[3 * j + 1], dz = f[3 * i + 2] - f[3 * j + 2];
  return fma(dx, dx, fma(dy, dy, dz * dz));
}

// Walk T frames of `per` pairs: the pairs at + m nt, m = 0, 1, ..., of all frames one after the other:
// f(frame, pair in the frame) for each.  Where a frame has fewer pairs than there are threads, a thread
// steps over dt whole frames and dq pairs at a time, so that all have a pair in every turn (a loop over
// the frames with one over a frame's pairs in it runs the threads of a warp one after the other there:
// S(k) of 16 wave numbers at T = 1000, N = 2 302 us, now 10); else that loop, whose turns cost
// less (S(k) of 4 at N = 128: 2.92 ms, 3.06 without it).  FEW: the former alone.
template <bool FEW, class F>
__device__ __forceinline__ void walk_frames(int T, unsigned per, unsigned nt, unsigned at, F&& f) {
  if (!FEW && per >= nt) {
    unsigned q = at;
    for (int t = 0; t < T; ++t) {
      for (; q < per; q += nt) f(t, q);
      q -= per;  // the walk goes on in the next frame where it would have
    }
  } else if (per > 0) {
    const unsigned dt = nt / per, dq = nt % per;
    unsigned t = at / per, q = at % per;
    while (t < (unsigned)T) {
      f((int)t, q);
      t += dt;
      q += dq;
      if (q >= per) {
        q -= per;
        ++t;
      }
    }
  }
}

// The pairs i < j of all frames by the nt threads of which this is number `at`: f(r2) for each
template <bool FEW, class F>
__device__ __forceinline__ void walk_pairs(const double* __restrict__ traj, int T, int N, unsigned nt, unsigned at, F&& f) {
  walk_frames<FEW>(T, (unsigned)N * (unsigned)(N - 1) / 2, nt, at,
                   [&](int t, unsigned q) { f(pair_r2(traj + 3 * (size_t)N * t, N, q)); });
}
// The ordered pairs (i, j) at the origins 0, s, 2s, ... of which a later frame exists
template <bool FEW, class F>
__device__ __forceinline__ void walk_origins(const double* __restrict__ traj, int norig, int N, int stride, int lag,
                                             unsigned nt, unsigned at, F&& f) {
  walk_frames<FEW>(norig, (unsigned)N * (unsigned)N, nt, at, [&](int o, unsigned q) {
    const double* fa = traj + 3 * (size_t)N * ((size_t)o * (unsigned)stride);
    const double* fb = fa + 3 * (size_t)N * (unsigned)lag;
    const unsigned i = q / (unsigned)N, j = q % (unsigned)N;
    const double dx = fb[3 * i] - fa[3 * j], dy = fb[3 * i + 1] - fa[3 * j + 1], dz = fb[3 * i + 2] - fa[3 * j + 2];
    f(fma(dx, dx, fma(dy, dy, dz * dz)));
  });
}
__device__ __forceinline__ int origins(int T, int lag, int stride) { return T - lag > 0 ? (T - lag + stride - 1) / stride : 0; }

// `parts` clusters per group of KG wave numbers; two add their sums to S, zeroed
template <int KG>
__global__ void __launch_bounds__(kThreads) k_static_sk(const double* __restrict__ traj, int T, int N,
                                                        const double* __restrict__ ks, int nk, double* __restrict__ S,
                                                        int parts) {
  __shared__ SinTab tab;
  __shared__ double2 seed[48];
  __shared__ double ws[KG * 32], bs[KG];
  fill_sin_table(&tab, seed);
  const unsigned cluster = blockIdx.x / cluster_blocks(), part = cluster % (unsigned)parts;
  const int g0 = (int)(cluster / (unsigned)parts) * KG;
  const WaveNumbers<KG> w(ks, nk, g0);
  double acc[KG] = {};
  walk_pairs<false>(traj, T, N, parts * cluster_blocks() * kThreads, (part * cluster_blocks() + cluster_rank()) * kThreads + threadIdx.x,
             [&](double r2) { add_pair<KG>(r2, w, &tab, acc); });
  cluster_sum<KG>(acc, ws, bs);
  if (cluster_rank() == 0 && threadIdx.x == 0) {
#pragma unroll
    for (int g = 0; g < KG; ++g)
      if (g0 + g < nk) {
        // the N diagonal terms of every frame and each pair twice, over N T; at k = 0 a sum of 0, or
        // NaN where a distance is not finite
        const double pairs = w.k[g] == 0.0 ? 0.5 / parts * (double)N * (N - 1) * T + acc[g] : acc[g] / w.k[g];
        const double v = (part ? 0.0 : 1.0) + 2.0 * pairs / ((double)N * T);
        if (parts == 1) S[g0 + g] = v;
        else atomicAdd(S + g0 + g, v);
      }
  }
}
// Few pairs: one block per wave number, without a table
__global__ void __launch_bounds__(kThreads) k_static_sk_few(const double* __restrict__ traj, int T, int N,
                                                            const double* __restrict__ ks, double* __restrict__ S) {
  __shared__ double sh[1][kThreads];
  const double k = ks[blockIdx.x];
  double v[1] = {0};
  walk_pairs<true>(traj, T, N, kThreads, threadIdx.x, [&](double r2) { v[0] += sinc(k, r2); });
  block_sum<1>(v, sh);
  if (threadIdx.x == 0) S[blockIdx.x] = ((double)N * T + 2.0 * v[0]) / ((double)N * T);
}

// One cluster per lag (blockIdx.y) and group of KG wave numbers: all ordered pairs (i, j) at the
// origins t0 = 0, s, 2s, ...
template <int KG>
__global__ void __launch_bounds__(kThreads) k_dynamic_sk(const double* __restrict__ traj, int T, int N,
                                                         const double* __restrict__ ks, int nk, int stride,
                                                         double* __restrict__ S, int nlag) {
  __shared__ SinTab tab;
  __shared__ double2 seed[48];
  __shared__ double ws[KG * 32], bs[KG];
  fill_sin_table(&tab, seed);
  const int g0 = (int)(blockIdx.x / cluster_blocks()) * KG;
  const int lag = blockIdx.y;
  const int norig = origins(T, lag, stride);
  const WaveNumbers<KG> w(ks, nk, g0);
  double acc[KG] = {};
  walk_origins<false>(traj, norig, N, stride, lag, cluster_blocks() * kThreads, cluster_rank() * kThreads + threadIdx.x,
               [&](double r2) { add_pair<KG>(r2, w, &tab, acc); });
  cluster_sum<KG>(acc, ws, bs);
  if (cluster_rank() == 0 && threadIdx.x == 0) {
#pragma unroll
    for (int g = 0; g < KG; ++g)
      if (g0 + g < nk) {
        const double pairs = w.k[g] == 0.0 ? (double)N * N * norig + acc[g] : acc[g] / w.k[g];  // (as above)
        S[(size_t)(g0 + g) * nlag + lag] = norig > 0 ? pairs / ((double)N * norig) : 0.0;
      }
  }
}
// Few pairs: one block per wave number and lag, without a table
__global__ void __launch_bounds__(kThreads) k_dynamic_sk_few(const double* __restrict__ traj, int T, int N,
                                                             const double* __restrict__ ks, int stride,
                                                             double* __restrict__ S, int nlag) {
  __shared__ double sh[1][kThreads];
  const double k = ks[blockIdx.x];
  const int lag = blockIdx.y, norig = origins(T, lag, stride);
  double v[1] = {0};
  walk_origins<true>(traj, norig, N, stride, lag, kThreads, threadIdx.x, [&](double r2) { v[0] += sinc(k, r2); });
  block_sum<1>(v, sh);
  if (threadIdx.x == 0) S[(size_t)blockIdx.x * nlag + lag] = norig > 0 ? v[0] / ((double)N * norig) : 0.0;
}

// One block, or two clusters that add to `out`, zeroed: 1/r_ij over the pairs i < j of every frame
__global__ void __launch_bounds__(2 * kThreads) k_inverse_radius(const double* __restrict__ traj, int T, int N,
                                                                 double* __restrict__ out) {
  __shared__ double ws[32], bs[1];
  double acc[1] = {0.0};
  walk_pairs<false>(traj, T, N, gridDim.x * blockDim.x, blockIdx.x * blockDim.x + threadIdx.x,
             [&](double r2) { acc[0] += rsqrt_range(r2) ? rsqrt_pos(r2) : 1.0 / sqrt(r2); });
  cluster_sum<1>(acc, ws, bs);
  if (cluster_rank() == 0 && threadIdx.x == 0) {
    const double v = 2.0 * acc[0] / ((double)N * N * T);
    if (gridDim.x == 1) *out = v;
    else atomicAdd(out, v);
  }
}

constexpr size_t kMaxShared = 227 * 1024;  // dynamic and static shared memory of a block
// Dynamic shared memory that keeps a second block off the SM: a cluster's blocks are otherwise
// placed two or three to an SM while other SMs idle, and these kernels fill an SM's FP64 pipe
// with one block.
constexpr size_t kOnePerSM = 116 * 1024;
// Clusters of each size that fit the chip at one block per SM (cudaOccupancyMaxActiveClusters on a
// GB300: 152 SMs, whose groups do not hold a whole number of larger clusters), and how many of them
// S(k) puts on a group of wave numbers
struct ClusterFit {
  int parts, size, fit;
};
constexpr ClusterFit kClusterFit[] = {{2, 16, 7}, {2, 10, 13}, {2, 9, 15}, {2, 6, 23}, {2, 4, 36},
                                      {1, 8, 15}, {1, 4, 36},  {1, 2, 76}, {1, 1, 152}};
// What a structure factor takes in us, for the choice between its forms.  A turn, in which each thread of
// a block takes one pair, is bound by the FP64 pipe of the block's SM: 1 us for the distance and 1.08
// for each sine by the table, 3.4 with the general sine.  A launch takes 4 us and a block's table and
// cluster sum 2 to 4.4 (each wave of blocks).  Measured, S(k) of T frames of N beads, by a block per
// wave number without a table and in groups of 1 and 3 on clusters of 4: T = 1, N = 32 (two turns of
// a block) 10.5, 10.5, 16.7; T = 100, N = 32 (194) 604, 117, 222.  S(k, t) in groups of 1 on a
// block, 2 on 2, 4 on 8 at T = 1000, N = 8, 100 lags: 55.6, 51.4, 68.4 (65.1 without a table; by this
// 61, 52, 67 (69)).
double us_by_table(double waves, int kg, int cs, double turns) {
  return 4.0 + 0.25 * cs + waves * (2.0 + 0.6 * kg + (1 + 1.08 * kg) * fmax(1.0, turns));
}
double us_without_table(double blocks, double turns) { return 4.0 + 3.4 * ceil(blocks / 152) * fmax(1.0, turns); }
constexpr double kClear = 0.85;  // a table has to be this much faster by these estimates, which are that rough

template <class K>
bool allow_shared(K* kernel, size_t bytes) {
  if (bytes <= 40 * 1024) return true;
  if (gblb::allow_all_shared((const void*)kernel) == cudaSuccess) return true;
  cudaGetLastError();
  return false;
}

int status_of(cudaError_t e) {
  return e == cudaSuccess ? LB_OK : (e == cudaErrorMemoryAllocation ? LB_ERR_OOM : LB_ERR_CUDA);
}

// a launch of grid.x clusters of cs blocks along x (smaller ones where those have no place), grid.y of
// them along y
template <class... A, class... B>
int launch_cluster(void (*kernel)(A...), dim3 grid, int threads, int cs, size_t smem, cudaStream_t s, B... args) {
  if (!allow_shared(kernel, smem)) return LB_ERR_CUDA;
  return status_of(gblb::launch_in_clusters(cs, [&](int size) {
    cudaError_t e = cudaSuccess;
    if (size > 8) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) {
      cudaLaunchConfig_t lc = {};
      lc.gridDim = dim3(grid.x * size, grid.y);
      lc.blockDim = dim3(threads);
      lc.dynamicSmemBytes = smem;
      lc.stream = s;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = (unsigned)size;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      lc.attrs = at;
      lc.numAttrs = 1;
      e = cudaLaunchKernelEx(&lc, kernel, (A)args...);
    }
    if (e != cudaSuccess) cudaGetLastError();
    return e;
  }));
}

// Blocks per cluster for `items` pairs per cluster, at most `most`: no more than leave each thread
// eight pairs.
int cluster_for(unsigned long long items, int threads, int most) {
  const unsigned long long by_work = items / (8ull * threads);
  return by_work < 1 ? 1 : (by_work < (unsigned long long)most ? (int)by_work : most);
}

int launch_status() {
  return status_of(cudaGetLastError());
}

}  // namespace

extern "C" {

int lb_analysis_msd(const double* traj, int T, int N, int max_lag, int i0, int i1, double* out, void* stream) {
  if (!traj || !out || T < 1 || N < 1 || max_lag < 0 || i0 < 0 || i1 < 0 || i0 >= N || i1 >= N) return LB_ERR_ARG;
  // Short chains and few lags leave the staged form's exchange of series with nothing to save (us, with the
  // host's share, staged and plain: T = 200, N = 8, 51 lags 72, 65; T = 1000, N = 8, 61 lags 105, 93;
  // T = 400, N = 16, 151 lags 86, 80; T = 400, N = 32, 61 lags 78, 101; T = 1000, N = 8, 501 lags 156, 180).
  const bool plain = (long long)T * (N - 12) <= 4000 && max_lag < 304;
  if (T <= kMsdFrames && !plain) {
    // as many clusters as fit the chip with one block per SM (15 of 8), no more than the lags need
    int nc = (max_lag + kMsdCluster) / kMsdCluster;
    nc = nc < 15 ? nc : 15;
    size_t smem = ((size_t)T * 9 + 1) * sizeof(double);
    smem = smem < kOnePerSM ? kOnePerSM : smem;
    return launch_cluster(k_msd_staged, dim3(nc), kMsdThreads, kMsdCluster, smem,
                          (cudaStream_t)stream, traj, T, N, i0, i1, out, max_lag + 1, nc);
  }
  k_msd<<<max_lag + 1, kThreads, 0, (cudaStream_t)stream>>>(traj, T, N, i0, i1, out, max_lag + 1);
  return launch_status();
}

int lb_analysis_rouse_modes(const double* traj, int T, int N, int P, double* X, void* stream) {
  if (!traj || !X || T < 1 || N < 2 || P < 1 || P > N - 1) return LB_ERR_ARG;
  const size_t smem = (4 * (size_t)N + kRouseFrames * 6 * ((size_t)N + 1) / 2) * sizeof(double);
  if (smem > kMaxShared) {
    k_rouse_modes_long<<<T, kThreads, 0, (cudaStream_t)stream>>>(traj, N, P, X);
    return launch_status();
  }
  if (!allow_shared(k_rouse_modes, smem)) return LB_ERR_CUDA;
  k_rouse_modes<<<(T + kRouseFrames - 1) / kRouseFrames, kThreads, smem, (cudaStream_t)stream>>>(traj, T, N, P, X);
  return launch_status();
}

int lb_analysis_rouse_correlation(const double* X, int T, int P, int max_lag, double* c, void* stream) {
  if (!X || !c || T < 1 || P < 1 || max_lag < 0 || max_lag > 65535) return LB_ERR_ARG;
  // What the two forms take, in us.  The staged form walks all origins for 32 lags at a time, however few
  // are asked for, in blocks of kCorrLags lags; the form with a block per lag and mode takes its share
  // of each, more where the modes of a frame lie in few of the cache's sets.  Measured, staged and
  // plain (and by this): T = 1000, P = 127, 501 lags 282, 642; P = 128, 1 lag 31, 8.5 (30, 8), 12 lags 31, 39
  // (30, 40); P = 13, 281 lags 54, 47 (55, 50); T = 3100, P = 300, 1 lag 158, 17 (156, 14), 16 lags
  // 158, 169 (156, 149); T = 100, P = 128, 2 lags 7.8, 6.4 (8, 6.5), P = 32, 11 lags 7.7, 6.2 (8, 7.0).
  const double lags = max_lag + 1.0, blocks = P * ceil(lags / kCorrLags);
  const double waves = blocks <= 152 ? 1.0 : (blocks <= 304 ? fmax(1.4, blocks / 152) : ceil(blocks / 152));
  const double staged = 5.5 + waves * 0.0246 * T * (lags > 32 ? 2 : 1);
  const double plain = 5.0 + P * lags * (0.0038 + 8.5e-6 * T * (P % 16 == 0 ? 2.2 : (P % 8 == 0 ? 1.3 : 1.0)));
  if (T <= kCorrFrames && plain > 0.95 * staged) {
    const size_t smem = 3 * (size_t)T * sizeof(double);
    if (!allow_shared(k_rouse_corr_staged, smem)) return LB_ERR_CUDA;
    k_rouse_corr_staged<<<dim3(P, (max_lag + kCorrLags) / kCorrLags), kThreads, smem, (cudaStream_t)stream>>>(
        X, T, P, c, max_lag + 1);
    return launch_status();
  }
  k_rouse_corr<<<dim3(P, max_lag + 1), kThreads, 0, (cudaStream_t)stream>>>(X, T, P, c, max_lag + 1);
  return launch_status();
}

int lb_analysis_static_sk(const double* traj, int T, int N, const double* k, int nk, double* S, void* stream) {
  if (!traj || !k || !S || T < 1 || N < 1 || nk < 1) return LB_ERR_ARG;
  // The group size and cluster with the shortest time, all clusters in one wave where possible.  16
  // wave numbers: groups of 3 on 12 clusters of 10 (6.8 ms at T = 1000, N = 128; groups of 2 on 16
  // clusters of 8, two waves, 11.5 ms; one block per wave number 144 ms).  Few pairs: a block per wave
  // number without a table (a frame of 8 beads 6.2 us, with a table 10).
  const double pairs = 0.5 * N * (N - 1.0) * T;
  const cudaStream_t s = (cudaStream_t)stream;
  double best = kClear * us_without_table(nk, pairs / kThreads);
  int kg = 0;
  ClusterFit c = {};
  for (int g = 1; g <= kKGroup; ++g)
    for (const ClusterFit& f : kClusterFit) {
      const int clusters = f.parts * ((nk + g - 1) / g), waves = (clusters + f.fit - 1) / f.fit;
      const double t = us_by_table(waves, g, f.size, ceil(pairs / (f.parts * f.size * kThreads))) + f.parts;
      if (t < best) {
        best = t;
        kg = g;
        c = f;
      }
    }
  if (kg == 0) {
    k_static_sk_few<<<nk, kThreads, 0, s>>>(traj, T, N, k, S);
    return launch_status();
  }
  const size_t apart = c.size > 1 ? kOnePerSM : 0;
  const dim3 grid((nk + kg - 1) / kg * c.parts);
  if (c.parts > 1 && cudaMemsetAsync(S, 0, nk * sizeof(double), s) != cudaSuccess) return launch_status();
  if (kg == 1) return launch_cluster(k_static_sk<1>, grid, kThreads, c.size, apart, s, traj, T, N, k, nk, S, c.parts);
  if (kg == 2) return launch_cluster(k_static_sk<2>, grid, kThreads, c.size, apart, s, traj, T, N, k, nk, S, c.parts);
  if (kg == 3) return launch_cluster(k_static_sk<3>, grid, kThreads, c.size, apart, s, traj, T, N, k, nk, S, c.parts);
  return launch_cluster(k_static_sk<kKGroup>, grid, kThreads, c.size, apart, s, traj, T, N, k, nk, S, c.parts);
}

int lb_analysis_inverse_radius(const double* traj, int T, int N, double* out, void* stream) {
  if (!traj || !out || T < 1 || N < 2) return LB_ERR_ARG;
  const cudaStream_t s = (cudaStream_t)stream;
  const unsigned long long pairs = (unsigned long long)N * (N - 1) / 2 * T;
  if (pairs <= 2 * 2 * kThreads)  // two pairs of a thread take less than the zeroing
    return launch_cluster(k_inverse_radius, dim3(1), 2 * kThreads, 1, 0, s, traj, T, N, out);
  const int cs = cluster_for(pairs / 2, 2 * kThreads, 16);
  if (cudaMemsetAsync(out, 0, sizeof(double), s) != cudaSuccess) return launch_status();
  return launch_cluster(k_inverse_radius, dim3(2), 2 * kThreads, cs, 0, s, traj, T, N, out);
}

int lb_analysis_dynamic_sk(const double* traj, int T, int N, const double* k, int nk, int max_lag,
                           int origin_stride, double* S, void* stream) {
  if (!traj || !k || !S || T < 1 || N < 1 || nk < 1 || max_lag < 0 || max_lag > 65535 || origin_stride < 1)
    return LB_ERR_ARG;
  // As for S(k); clusters of up to 8, of which several share an SM: one more wave than blocks fill
  // (84 blocks take 1.5 to 1.7 times a turn, 404 3.6, 808 5.5)
  const double pairs = (double)N * N * ((T + origin_stride - 1) / origin_stride), nlag = max_lag + 1.0;
  const cudaStream_t s = (cudaStream_t)stream;
  double best = kClear * us_without_table(nk * nlag, pairs / kThreads);
  int kg = 0, cs = 0;
  for (int g = nk < kKGroup ? nk : kKGroup; g >= 1; --g)
    for (int c = 8; c >= 1; c -= c > 4 ? 2 : 1) {
      const double blocks = (nk + g - 1) / g * nlag * c, turns = pairs / (c * kThreads);
      const double t = us_by_table(1.0 + blocks / 152, g, c, blocks <= 152 ? ceil(turns) : turns);
      if (t < best) {
        best = t;
        kg = g;
        cs = c;
      }
    }
  if (kg == 0) {
    k_dynamic_sk_few<<<dim3(nk, max_lag + 1), kThreads, 0, s>>>(traj, T, N, k, origin_stride, S, max_lag + 1);
    return launch_status();
  }
  const dim3 grid((nk + kg - 1) / kg, max_lag + 1);
  if (kg == 1) return launch_cluster(k_dynamic_sk<1>, grid, kThreads, cs, 0, s, traj, T, N, k, nk, origin_stride, S, max_lag + 1);
  if (kg == 2) return launch_cluster(k_dynamic_sk<2>, grid, kThreads, cs, 0, s, traj, T, N, k, nk, origin_stride, S, max_lag + 1);
  if (kg == 3) return launch_cluster(k_dynamic_sk<3>, grid, kThreads, cs, 0, s, traj, T, N, k, nk, origin_stride, S, max_lag + 1);
  return launch_cluster(k_dynamic_sk<kKGroup>, grid, kThreads, cs, 0, s, traj, T, N, k, nk, origin_stride, S, max_lag + 1);
}

}  // extern "C"
