// Brownian dynamics of bead-spring chains with hydrodynamic interaction (Sec. II C): the
// Ito-Euler update r += (D/kT) F dt + sqrt(2 dt) B.W, D/kT = zeta^-1 on the diagonal blocks and
// the regularised Rotne-Prager-Yamakawa mobility off the diagonal, B.W from Fixman's truncated
// Chebyshev expansion of sqrt(D) applied to the noise vector.  The chain model is that of the
// LB runs (FENE bonds, WCA between all pairs, Sec. II A), in an infinite medium.
//
// One thread block per chain (replica) runs many steps per launch with the chain on chip:
// positions, forces and the Chebyshev vectors in shared memory, the 3N x 3N mobility matrix in
// registers (FP32, N <= 64: k_bd_steps_reg) or in shared memory (symmetric: mat-vecs read it by
// columns, so that consecutive threads read consecutive words; k_bd_steps).  Per step: forces,
// the matrix, the noise, power iterations for the spectral bounds of D, the Chebyshev
// recurrence, the update.  Positions are kept in FP64 between launches; the arithmetic type R is
// FP32 or FP64.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <memory>
#include <vector>

#include "../../include/lb.h"
#include "d3q19.cuh"
#include "lb_engine.h"
#include "lb_shared.h"
#include "philox.cuh"

namespace gblb {
namespace {

constexpr int kBDThreads = 256;
constexpr int kBDMaxDegree = 64;
constexpr uint32_t kTagBD = 3;

template <class R>
struct BDK {
  int N;
  R kT, zeta, eta, radius, dt, kfene, R0sq, eps, sig2, rc2;
  int hi, degree, piters;
  uint32_t k0;
  double* x;  // [replica][3N], unwrapped positions
  unsigned* status;
};

template <class R>
__device__ __forceinline__ R rcp(R v) {
  return R(1) / v;
}

// block-wide sum of one value per thread (fixed order); every thread gets the result
template <class R>
__device__ R block_sum(R v, R* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) red[warp] = v;
  __syncthreads();
  R s = R(0);
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
  __syncthreads();
  return s;
}

// out = a * (M v) + b * v + c * u (M symmetric, n x n, leading dimension n; u may be null),
// and, with y, also y += cy * out.  Two neighbouring threads per output row, each over half
// the columns with two partial sums (M read by columns: consecutive rows are consecutive
// words), combined by a shuffle; the pair's even thread writes.
template <class R>
__device__ __forceinline__ void matvec(const R* __restrict__ M, int n, const R* __restrict__ v, R a, R b, R c,
                                       const R* __restrict__ u, R* __restrict__ out, R* __restrict__ y = nullptr,
                                       R cy = R(0)) {
  const int half = threadIdx.x & 1, h0 = half ? n / 2 : 0, h1 = half ? n : n / 2;
  for (int row = threadIdx.x >> 1; row < n; row += blockDim.x >> 1) {
    R s0 = R(0), s1 = R(0);
    int col = h0;
    for (; col + 1 < h1; col += 2) {
      s0 += M[col * n + row] * v[col];
      s1 += M[(col + 1) * n + row] * v[col + 1];
    }
    if (col < h1) s0 += M[col * n + row] * v[col];
    R sum = s0 + s1;
    sum += __shfl_xor_sync(__activemask(), sum, 1);  // the pair (2k, 2k+1) is active together
    if (!half) {
      R o = a * sum + b * v[row];
      if (u) o += c * u[row];
      out[row] = o;
      if (y) y[row] += cy * o;
    }
  }
}

// FENE (bonded) + WCA force coefficient of a pair: force on i = coef (x_i - x_j)
template <class R>
__device__ __forceinline__ R bd_pair_coef(R r2, bool bonded, const BDK<R>& P) {
  R coefv = R(0);
  if (r2 < P.rc2) {
    const R s2 = P.sig2 / r2, s6 = s2 * s2 * s2;
    coefv += R(24) * P.eps / r2 * (R(2) * s6 * s6 - s6);
  }
  if (bonded) {
    if (r2 >= P.R0sq)
      atomicOr(P.status, 1u);
    else
      coefv -= P.kfene / (R(1) - r2 / P.R0sq);
  }
  return coefv;
}

// Conservative force on bead i < N by `lanes` neighbouring threads (a power of two, lane: this
// one's), which split the partners and combine in a fixed tree; whole warps call it
template <class R>
__device__ __forceinline__ void bd_force(const R* __restrict__ x, const BDK<R>& P, int i, int lane, int lanes, R f[3]) {
  f[0] = f[1] = f[2] = R(0);
  if (i < P.N)
    for (int j = lane; j < P.N; j += lanes) {
      if (j == i) continue;
      const R d0 = x[3 * i] - x[3 * j], d1 = x[3 * i + 1] - x[3 * j + 1], d2 = x[3 * i + 2] - x[3 * j + 2];
      const R c = bd_pair_coef<R>(d0 * d0 + d1 * d1 + d2 * d2, j == i - 1 || j == i + 1, P);
      f[0] += c * d0;
      f[1] += c * d1;
      f[2] += c * d2;
    }
  for (int o = lanes / 2; o > 0; o /= 2)
#pragma unroll
    for (int q = 0; q < 3; ++q) f[q] += __shfl_xor_sync(0xffffffffu, f[q], o, lanes);
}

// Coefficients of the regularised RPY mobility of a pair: ci on the diagonal, cr on d d^T / r2
template <class R>
__device__ __forceinline__ void rpy(R r2, const BDK<R>& P, R& ci, R& cr) {
  const R r = sqrt(r2);
  if (r >= R(2) * P.radius) {
    const R a2 = P.radius * P.radius / r2;
    const R pre = rcp(R(8) * R(M_PI) * P.eta * r);
    ci = pre * (R(1) + R(2) * a2 / R(3));
    cr = pre * (R(1) - R(2) * a2);
  } else {
    const R q = r / P.radius;
    const R pre = rcp(R(6) * R(M_PI) * P.eta * P.radius);
    ci = pre * (R(1) - R(9) * q / R(32));
    cr = pre * (R(3) * q / R(32));
  }
}

// ---------------------------------------------------------------------------------------
// FP32 chains of up to 64 beads: the mobility matrix in registers
// ---------------------------------------------------------------------------------------
// A step is a chain of some 62 dependent products with the 3N x 3N matrix, each between two block
// barriers, so what counts is the latency of one.  Eight neighbouring threads share two rows, each
// with the 3B columns of B beads in registers for the whole step: a product reads only the
// vector (16-byte shared loads; a load serves both rows, since the 128 bytes per clock that
// shared memory returns to the registers bound a product with one row per thread), multiplies,
// and adds the eight by three shuffles, the first of which leaves either half with one of the two
// rows.  So a quad of threads holds a row's results: its values (the recurrences' earlier vectors,
// the sum, the position in FP64) stay there.  Normalising the power iterate is folded into the
// next product as a factor.  64 chains per launch, us per step, before (the matrix in shared memory,
// one load per multiply-add) and now: N = 8 35 -> 9.5, N = 32 61.7 -> 17.5 (one row per thread: 24.4),
// N = 64 200 -> 39.
template <int B>
struct BDReg {  // sizes, and the layout of k_bd_steps_reg's dynamic shared memory in floats
  static constexpr int kCols = 3 * B;                               // columns per thread
  static constexpr int kSeg = (((kCols + 3) / 4) | 1) * 4;          // words per segment of a vector: an odd number of
                                                                    // 16-byte units, so that eight segments' loads
                                                                    // hit different banks
  static constexpr int kVec = 8 * kSeg;
  static constexpr int kThreads = (12 * 8 * B + 31) / 32 * 32;      // of the longest chain, 8B beads
  int x, F, v, cheb, f, coef, part, pairs, total;
  __host__ __device__ BDReg(int N, int K) {
    int off = 0;
    auto take = [&](int n) {
      const int o = off;
      off += (n + 3) / 4 * 4;
      return o;
    };
    pairs = take(5 * 8 * B * N);  // {ci, cr/r2, d0, d1}, and d2, of the pairs (i, j) at pair_at(i, j)
    x = take(3 * N);
    F = take(kVec);
    v = take(2 * kVec);  // two product operands
    cheb = take(K * K);  // cos(k theta_j)
    f = take(K);
    coef = take(K);
    part = take(2 * 32);
    total = off;
  }
  // place of element c in a vector: segment c / 3B
  __device__ __forceinline__ static int vec_at(int c) { return c / kCols * kSeg + c % kCols; }
  // of pair (i, j): the same bead of the eight segments side by side, as eight threads read them
  __device__ __forceinline__ static int pair_at(int i, int j) { return i * 8 * B + j % B * 8 + j / B; }
};

template <int B>
__global__ void __launch_bounds__(BDReg<B>::kThreads) k_bd_steps_reg(const BDK<float> P, uint32_t step0, int nsteps) {
  using R = float;
  using Z = BDReg<B>;
  extern __shared__ __align__(16) unsigned char bsm[];
  const int N = P.N, n = 3 * N, tid = threadIdx.x, nt = blockDim.x, K = P.degree + 1;
  const int lane = tid & 31, warp = tid >> 5;
  const Z L(N, K);
  R* const sm = reinterpret_cast<R*>(bsm);
  R *const x = sm + L.x, *const sF = sm + L.F, *const v0 = sm + L.v, *const v1 = v0 + Z::kVec;
  R *const cheb = sm + L.cheb, *const fj = sm + L.f, *const coef = sm + L.coef, *const part = sm + L.part;
  float4* const pa = reinterpret_cast<float4*>(sm + L.pairs);
  R* const pb = sm + L.pairs + 4 * 8 * B * N;
  const int row = tid >> 2, seg = tid & 7;  // the row whose results this quad holds; its columns' segment
  const bool writes = row < n && (tid & 3) == 0, live = row < n;
  const int at = Z::vec_at(row);
  double* const gx = P.x + (size_t)blockIdx.x * n;
  const uint32_t k1 = kTagBD | ((uint32_t)blockIdx.x << 8);
  double xd = live ? gx[row] : 0.0;
  if (tid < 32) part[tid] = part[32 + tid] = R(0);
  for (int i = tid; i < Z::kVec; i += nt) v0[i] = v1[i] = sF[i] = R(0);  // padding and columns past n stay zero
  for (int i = tid; i < K * K; i += nt) {
    const int k = i / K, j = i - k * K;
    const R th = R(M_PI) * (R(j) + R(0.5)) / R(K);
    cheb[i] = cos(R(k) * th);
  }
  if (writes) x[row] = (R)xd;
  __syncthreads();
  R m[2][3 * B];  // this thread's columns of rows 2 (tid / 8) and the next
  // (M v) of the quad's row, in its four threads
  auto product = [&](const R* v) {
    const float4* p = reinterpret_cast<const float4*>(v + seg * Z::kSeg);
    R s[2][2] = {{R(0), R(0)}, {R(0), R(0)}};
#pragma unroll
    for (int k = 0; k < 3 * B; k += 4) {
      const float4 q = p[k / 4];
      const R e[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (k + j < 3 * B) {
          s[0][j & 1] = fmaf(m[0][k + j], e[j], s[0][j & 1]);
          s[1][j & 1] = fmaf(m[1][k + j], e[j], s[1][j & 1]);
        }
    }
    const R a = s[0][0] + s[0][1], b = s[1][0] + s[1][1];
    const bool second = tid & 4;
    R r = second ? b : a;
    r += __shfl_xor_sync(0xffffffffu, second ? a : b, 4);
    r += __shfl_xor_sync(0xffffffffu, r, 2);
    r += __shfl_xor_sync(0xffffffffu, r, 1);
    return r;
  };
  // sums over the rows: each warp's eight rows now, all warps' after the next barrier
  int turn = 0;
  auto sum_rows = [&](R s) {
    s = live ? s : R(0);
    s += __shfl_xor_sync(0xffffffffu, s, 4);
    s += __shfl_xor_sync(0xffffffffu, s, 8);
    s += __shfl_xor_sync(0xffffffffu, s, 16);
    turn ^= 32;
    if (lane == 0) part[turn + warp] = s;
  };
  auto total = [&]() {
    const float4* p = reinterpret_cast<const float4*>(part + turn);
    R s = R(0);
#pragma unroll
    for (int w = 0; w < (Z::kThreads / 32 + 3) / 4; ++w) {
      const float4 q = p[w];
      s += (q.x + q.y) + (q.z + q.w);
    }
    return s;
  };
  const R inv = rcp(sqrt(R(n)));
  // Rayleigh quotient of a M + b after the power iterations from the uniform vector.  The iterate is
  // normalised every fourth iteration and after the last (the direction, and so the quotient,
  // does not depend on it; four unnormalised iterations change the norm by at most lam_max^4).
  auto quotient = [&](R a, R b) {
    R* cur = v0;
    R* nxt = v1;
    if (writes) cur[at] = inv;
    R own = inv, scale = R(1);  // the row's value; the vector in shared memory is 1/scale times it
    __syncthreads();
    for (int k = 0; k < P.piters; ++k) {
      const R o = a * (scale * product(cur)) + b * own;
      if (writes) nxt[at] = o;
      const bool norm = (k & 3) == 3 || k == P.piters - 1;
      if (norm) sum_rows(o * o);
      __syncthreads();
      scale = norm ? rcp(sqrt(total())) : R(1);
      own = o * scale;
      R* sw = cur;
      cur = nxt;
      nxt = sw;
    }
    sum_rows(own * (a * (scale * product(cur)) + b * own));
    __syncthreads();
    return total();
  };
  for (int it = 0; it < nsteps; ++it) {
    const uint32_t step = step0 + (uint32_t)it;
    const R self = rcp(P.zeta);
    // forces by eight threads per bead, noise (3 standard normals per bead from one Philox call,
    // counter (step, bead, 0, 0)) by the other four's first; pairs by all
    {
      R f[3];
      const int i = tid >> 3;
      bd_force<R>(x, P, i, tid & 7, 8, f);
      if (i < N && (tid & 7) < 3) {
        const int q = tid & 7, r = 3 * i + q;
        sF[Z::vec_at(r)] = q == 0 ? f[0] : (q == 1 ? f[1] : f[2]);
      }
    }
    for (int i = tid - 8 * N; i >= 0 && i < N; i += nt) {
      R g[4];
      gauss4<R>(step, (uint32_t)i, 0u, P.k0, k1, g);
#pragma unroll
      for (int q = 0; q < 3; ++q) v1[Z::vec_at(3 * i + q)] = g[q];
    }
    if (P.hi) {
      for (int q = tid; q < N * (N + 1) / 2; q += nt) {  // (i, i + d), d = 0 .. N/2: each pair once
        const int d = q / N, i = q - d * N, j = i + d < N ? i + d : i + d - N;
        const R d0 = x[3 * i] - x[3 * j], d1 = x[3 * i + 1] - x[3 * j + 1], d2 = x[3 * i + 2] - x[3 * j + 2];
        R ci = self, cr = R(0);
        if (d > 0) {
          const R r2 = d0 * d0 + d1 * d1 + d2 * d2;
          rpy<R>(r2, P, ci, cr);
          cr /= r2;
        }
        const int ij = Z::pair_at(i, j), ji = Z::pair_at(j, i);
        pa[ij] = pa[ji] = make_float4(ci, cr, d0, d1);
        pb[ij] = pb[ji] = d2;
      }
    }
    __syncthreads();
    const R w = live ? v1[at] : R(0);  // the row's noise
    R y, drift;
    if (P.hi) {
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int mine = 2 * (tid >> 3) + r, i = mine / 3, comp = mine - 3 * (mine / 3);
#pragma unroll
        for (int k = 0; k < B; ++k) {
          float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
          R d2 = R(0);
          if (mine < n && seg * B + k < N) {
            q = pa[i * 8 * B + k * 8 + seg];
            d2 = pb[i * 8 * B + k * 8 + seg];
          }
          const R c = q.y * (comp == 0 ? q.z : (comp == 1 ? q.w : d2));
          m[r][3 * k] = (comp == 0 ? q.x : R(0)) + c * q.z;
          m[r][3 * k + 1] = (comp == 1 ? q.x : R(0)) + c * q.w;
          m[r][3 * k + 2] = (comp == 2 ? q.x : R(0)) + c * d2;
        }
      }
      drift = P.dt * product(sF);
      __syncthreads();  // every row has its noise: v1 is overwritten
      // spectral bounds of D = kT M: lam_max on D, lam_min on lam_max I - D
      const R lam_max = R(1.05) * quotient(P.kT, R(0));
      const R mu = quotient(-P.kT, lam_max);
      R lam_min = R(0.5) * (lam_max - mu);
      if (lam_min < lam_max / R(1000)) lam_min = lam_max / R(1000);
      // Chebyshev coefficients of sqrt on [lam_min, lam_max] from the degree + 1 nodes, and the
      // recurrence y = sum_k c_k T_k(Dt) W, Dt = s D - t I
      for (int j = tid; j < K; j += nt)
        fj[j] = sqrt(R(0.5) * (lam_max + lam_min) + R(0.5) * (lam_max - lam_min) * cheb[K + j]);
      const R sc = R(2) / (lam_max - lam_min), tc = (lam_max + lam_min) / (lam_max - lam_min);
      if (writes) v0[at] = w;
      __syncthreads();
      for (int k = tid; k < K; k += nt) {
        R s = R(0);
        for (int j = 0; j < K; ++j) s += fj[j] * cheb[k * K + j];
        coef[k] = (k == 0 ? R(1) : R(2)) / R(K) * s;
      }
      R tp = w, tc1 = sc * P.kT * product(v0) - tc * w;  // T_{k-1}, T_k of the row
      R* cur = v1;
      R* nxt = v0;
      if (writes) cur[at] = tc1;
      __syncthreads();
      y = coef[0] * w + coef[1] * tc1;
      for (int k = 2; k < K; ++k) {
        const R tn = R(2) * sc * P.kT * product(cur) - R(2) * tc * tc1 - tp;
        if (writes) nxt[at] = tn;
        y += coef[k] * tn;
        tp = tc1;
        tc1 = tn;
        __syncthreads();
        R* sw = cur;
        cur = nxt;
        nxt = sw;
      }
    } else {
      drift = live ? P.dt * (self * sF[at]) : R(0);
      y = sqrt(P.kT / P.zeta) * w;
      __syncthreads();
    }
    // update: r += M F dt + sqrt(2 dt) B W (drift through the same mobility)
    xd += (double)(drift + sqrt(R(2) * P.dt) * y);
    if (writes) x[row] = (R)xd;
    __syncthreads();
  }
  if (writes) gx[row] = xd;
}

// Other chains: the matrix in shared memory
template <class R>
__global__ void __launch_bounds__(kBDThreads) k_bd_steps(const BDK<R> P, uint32_t step0, int nsteps) {
  extern __shared__ __align__(16) unsigned char bsm[];
  const int N = P.N, n = 3 * N, tid = threadIdx.x, nt = blockDim.x;
  R* M = reinterpret_cast<R*>(bsm);  // n x n
  R* x = M + n * n;                  // positions (arithmetic copy)
  R* F = x + n;                      // forces
  R* W = F + n;                      // noise
  R* y = W + n;                      // B.W
  R* t0 = y + n;                     // Chebyshev / power-iteration vectors
  R* t1 = t0 + n;
  R* t2 = t1 + n;
  R* red = t2 + n;                   // 32 partial sums
  R* coef = red + 32;                // Chebyshev coefficients
  R* scal = coef + kBDMaxDegree + 1; // [0] lam_min, [1] lam_max
  double* gx = P.x + (size_t)blockIdx.x * n;
  const uint32_t k1 = kTagBD | ((uint32_t)blockIdx.x << 8);
  for (int t = tid; t < n; t += nt) x[t] = (R)gx[t];
  int lanes = 1;  // (more than N would add zeros: N = 2, free draining, FP64, 400 chains 21.6 us per step, now 17.7)
  while (lanes < 32 && lanes < N && lanes * 2 * N <= nt) lanes *= 2;
  __syncthreads();
  for (int it = 0; it < nsteps; ++it) {
    const uint32_t step = step0 + (uint32_t)it;
    // forces: FENE on bonds, WCA on all pairs, as many threads per bead as fit
    for (int base = 0; base < N; base += nt / lanes) {
      const int i = base + tid / lanes;
      R f[3];
      bd_force<R>(x, P, i, tid % lanes, lanes, f);
      if (i < N && tid % lanes == 0) {
        F[3 * i] = f[0];
        F[3 * i + 1] = f[1];
        F[3 * i + 2] = f[2];
      }
    }
    // mobility D/kT: zeta^-1 on the diagonal blocks, regularised RPY elsewhere
    const R self = rcp(P.zeta);
    for (int pr = tid; pr < N * N; pr += nt) {  // consecutive threads: consecutive i (store stride 3)
      const int j = pr / N, i = pr - (pr / N) * N;
      R blk[3][3];
      if (i == j || !P.hi) {
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
          for (int b = 0; b < 3; ++b) blk[a][b] = (i == j && a == b) ? self : R(0);
      } else {
        const R d[3] = {x[3 * i] - x[3 * j], x[3 * i + 1] - x[3 * j + 1], x[3 * i + 2] - x[3 * j + 2]};
        const R r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
        R ci, cr;
        rpy<R>(r2, P, ci, cr);
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
          for (int b = 0; b < 3; ++b) blk[a][b] = (a == b ? ci : R(0)) + cr * d[a] * d[b] / r2;
      }
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) M[(3 * j + b) * n + 3 * i + a] = blk[a][b];
    }
    // noise: 3 standard normals per bead from one Philox call, counter (step, bead, 0, 0)
    for (int i = tid; i < N; i += nt) {
      R g[4];
      gauss4<R>(step, (uint32_t)i, 0u, P.k0, k1, g);
      W[3 * i] = g[0];
      W[3 * i + 1] = g[1];
      W[3 * i + 2] = g[2];
    }
    __syncthreads();
    if (P.hi) {
      // spectral bounds of D = kT M by power iterations (lam_max: on D; lam_min: on lam_max I - D)
      const R inv = rcp(sqrt(R(n)));
      for (int t = tid; t < n; t += nt) t0[t] = inv;
      __syncthreads();
      // the iterate is normalised every fourth iteration and after the last (the direction,
      // and so the Rayleigh quotient below, does not depend on it; four unnormalised
      // iterations change the norm by at most lam_max^4)
      R* pa = t0;  // the iterate
      R* pb = t1;
      for (int k = 0; k < P.piters; ++k) {
        matvec<R>(M, n, pa, P.kT, R(0), R(0), nullptr, pb);
        __syncthreads();
        if ((k & 3) == 3 || k == P.piters - 1) {
          R part = R(0);
          for (int t = tid; t < n; t += nt) part += pb[t] * pb[t];
          const R nrm = rcp(sqrt(block_sum<R>(part, red)));
          for (int t = tid; t < n; t += nt) pb[t] *= nrm;
          __syncthreads();
        }
        R* sw = pa;
        pa = pb;
        pb = sw;
      }
      if (pa != t0) {  // the iterate back into t0
        for (int t = tid; t < n; t += nt) t0[t] = pa[t];
        __syncthreads();
      }
      matvec<R>(M, n, t0, P.kT, R(0), R(0), nullptr, t1);
      __syncthreads();
      R part = R(0);
      for (int t = tid; t < n; t += nt) part += t0[t] * t1[t];
      const R lam_max = R(1.05) * block_sum<R>(part, red);
      for (int t = tid; t < n; t += nt) t0[t] = inv;
      __syncthreads();
      pa = t0;
      pb = t1;
      for (int k = 0; k < P.piters; ++k) {
        matvec<R>(M, n, pa, -P.kT, lam_max, R(0), nullptr, pb);  // (lam_max I - D) v
        __syncthreads();
        if ((k & 3) == 3 || k == P.piters - 1) {
          R pp = R(0);
          for (int t = tid; t < n; t += nt) pp += pb[t] * pb[t];
          const R nrm = rcp(sqrt(block_sum<R>(pp, red)));
          for (int t = tid; t < n; t += nt) pb[t] *= nrm;
          __syncthreads();
        }
        R* sw = pa;
        pa = pb;
        pb = sw;
      }
      if (pa != t0) {
        for (int t = tid; t < n; t += nt) t0[t] = pa[t];
        __syncthreads();
      }
      matvec<R>(M, n, t0, -P.kT, lam_max, R(0), nullptr, t1);
      __syncthreads();
      R pq = R(0);
      for (int t = tid; t < n; t += nt) pq += t0[t] * t1[t];
      const R mu = block_sum<R>(pq, red);
      R lam_min = R(0.5) * (lam_max - mu);
      if (lam_min < lam_max / R(1000)) lam_min = lam_max / R(1000);
      // Chebyshev coefficients of sqrt on [lam_min, lam_max] from the degree+1 nodes
      const int K = P.degree + 1;
      for (int k = tid >> 5; k < K; k += nt >> 5) {  // a warp per coefficient
        R s = R(0);
        for (int j = tid & 31; j < K; j += 32) {
          const R th = R(M_PI) * (R(j) + R(0.5)) / R(K);
          const R xj = R(0.5) * (lam_max + lam_min) + R(0.5) * (lam_max - lam_min) * cos(th);
          s += sqrt(xj) * cos(R(k) * th);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((tid & 31) == 0) coef[k] = (k == 0 ? R(1) : R(2)) / R(K) * s;
      }
      __syncthreads();
      // recurrence: y = sum_k c_k T_k(Dt) W, Dt = s D - t I
      const R sc = R(2) / (lam_max - lam_min), tc = (lam_max + lam_min) / (lam_max - lam_min);
      matvec<R>(M, n, W, sc * P.kT, -tc, R(0), nullptr, t1);  // T_1 W
      __syncthreads();
      for (int t = tid; t < n; t += nt) y[t] = coef[0] * W[t] + coef[1] * t1[t];
      __syncthreads();  // y and t1 are next touched by other threads (the mat-vecs' rows)
      R* tp = W;   // T_{k-1}
      R* tcur = t1;  // T_k
      R* tn = t2;
      for (int k = 2; k < K; ++k) {
        // 2 Dt T_k - T_{k-1}, added to y times c_k by the thread that forms each row
        matvec<R>(M, n, tcur, R(2) * sc * P.kT, R(-2) * tc, R(-1), tp, tn, y, coef[k]);
        __syncthreads();
        R* sw = tp;
        tp = tcur;
        tcur = tn;
        tn = (sw == W) ? t0 : sw;  // never overwrite W before the recurrence is done
      }
    } else {
      const R amp = sqrt(P.kT / P.zeta);
      for (int t = tid; t < n; t += nt) y[t] = amp * W[t];
      __syncthreads();
    }
    // update: r += M F dt + sqrt(2 dt) B W (drift through the same mobility)
    matvec<R>(M, n, F, P.dt, R(0), R(0), nullptr, t1);
    __syncthreads();
    const R nz = sqrt(R(2) * P.dt);
    for (int t = tid; t < n; t += nt) {
      const double nx = gx[t] + (double)(t1[t] + nz * y[t]);
      gx[t] = nx;
      x[t] = (R)nx;
    }
    __syncthreads();
  }
}

class BDBase {
 public:
  virtual ~BDBase() {}
  virtual void step(int64_t n, uint32_t k0, cudaStream_t s) = 0;
  virtual void get(double* x, cudaStream_t s) = 0;
  virtual unsigned status(cudaStream_t s) = 0;
};

template <class R>
class BDT final : public BDBase {
 public:
  BDT(int reps, const BDK<R>& P, const double* x0) : reps_(reps), P_(P) {
    const size_t n = 3 * (size_t)P.N;
    cuda_check(cudaMalloc(&P_.x, reps * n * sizeof(double)), "BD positions");
    cuda_check(cudaMalloc(&P_.status, sizeof(unsigned)), "BD status");
    cuda_check(cudaMemcpy(P_.x, x0, reps * n * sizeof(double), cudaMemcpyHostToDevice), "upload BD positions");
    cuda_check(cudaMemset(P_.status, 0, sizeof(unsigned)), "BD status");
    kernel_ = k_bd_steps<R>;
    threads_ = kBDThreads;
    smem_ = (n * n + 8 * n + 32 + kBDMaxDegree + 1 + 2) * sizeof(R);
    if constexpr (sizeof(R) == 4) {  // the fewest beads per thread that hold a row in eight threads
      if (P.N <= 8) use_registers<1>();
      else if (P.N <= 16) use_registers<2>();
      else if (P.N <= 24) use_registers<3>();
      else if (P.N <= 32) use_registers<4>();
      else if (P.N <= 40) use_registers<5>();
      else if (P.N <= 48) use_registers<6>();
      else if (P.N <= 64) use_registers<8>();
    }
    if (smem_ > 48 * 1024)
      cuda_check(allow_all_shared((const void*)kernel_), "BD shared memory");
  }
  ~BDT() override {
    cudaFree(P_.x);
    cudaFree(P_.status);
  }
  void step(int64_t n, uint32_t k0, cudaStream_t s) override {
    const int chunk = 4096;  // steps per launch
    for (int64_t done = 0; done < n;) {
      const int m = (int)(n - done < chunk ? n - done : chunk);
      kernel_<<<reps_, threads_, smem_, s>>>(P_, k0 + (uint32_t)done, m);
      cuda_check(cudaGetLastError(), "BD kernel");
      done += m;
    }
  }
  void get(double* x, cudaStream_t s) override {
    cuda_check(cudaMemcpyAsync(x, P_.x, reps_ * 3 * (size_t)P_.N * sizeof(double), cudaMemcpyDeviceToHost, s),
               "download BD positions");
    cuda_check(cudaStreamSynchronize(s), "sync BD");
  }
  unsigned status(cudaStream_t s) override {
    unsigned st = 0;
    cuda_check(cudaMemcpyAsync(&st, P_.status, sizeof(unsigned), cudaMemcpyDeviceToHost, s), "BD status");
    cuda_check(cudaStreamSynchronize(s), "sync BD status");
    return st;
  }

 private:
  template <int B>
  void use_registers() {
    kernel_ = k_bd_steps_reg<B>;
    threads_ = (12 * P_.N + 31) / 32 * 32;
    smem_ = (size_t)BDReg<B>(P_.N, P_.degree + 1).total * sizeof(R);
  }
  int reps_;
  BDK<R> P_;
  void (*kernel_)(const BDK<R>, uint32_t, int) = nullptr;
  int threads_ = 0;
  size_t smem_ = 0;
};

int bd_fail(int code) { return code; }

}  // namespace
}  // namespace gblb

using namespace gblb;

struct lb_bd {
  std::unique_ptr<BDBase> b;
  int reps = 0, N = 0;
  int64_t step = 0;
  cudaStream_t stream = nullptr;
};

namespace {

template <class F>
int bd_guard(F&& f) {
  try {
    return f();
  } catch (const LbError& e) {
    return bd_fail(e.code);
  } catch (...) {
    return LB_ERR_CUDA;
  }
}

template <class R>
BDK<R> bd_params(int N, double kT, double zeta, double eta_s, double dt, double k_fene, double R0, double eps,
                 double sigma, int hi, int degree, int piters, uint64_t seed) {
  BDK<R> P;
  memset(&P, 0, sizeof(P));
  P.N = N;
  P.kT = (R)kT;
  P.zeta = (R)zeta;
  P.eta = (R)eta_s;
  P.radius = (R)(zeta / (6.0 * M_PI * eta_s));
  P.dt = (R)dt;
  P.kfene = (R)k_fene;
  P.R0sq = (R)(R0 * R0);
  P.eps = (R)eps;
  P.sig2 = (R)(sigma * sigma);
  P.rc2 = (R)(pow(2.0, 1.0 / 3.0) * sigma * sigma);
  P.hi = hi ? 1 : 0;
  P.degree = degree;
  P.piters = piters;
  P.k0 = (uint32_t)(seed & 0xffffffffu);
  return P;
}

}  // namespace

extern "C" {

int lb_bd_create(lb_bd** out, int replicas, int N, double kT, double zeta, double eta_s, double dt, double k_fene,
                 double R0, double eps, double sigma, int hi, int degree, int power_iters, uint64_t seed,
                 const double* x0, int precision) {
  if (!out || !x0 || replicas < 1 || replicas > 65535 || N < 1 || !(kT > 0) || !(zeta > 0) || !(eta_s > 0) ||
      !(dt > 0) || !(k_fene >= 0) || !(R0 > 0) || !(sigma > 0) || degree < 1 || degree > kBDMaxDegree ||
      power_iters < 1 || (precision != LB_FP64 && precision != LB_FP32))
    return LB_ERR_ARG;
  const int max_n = precision == LB_FP64 ? 52 : 74;  // the 3N x 3N matrix lives in shared memory
  if (N > max_n) return LB_ERR_ARG;
  return bd_guard([&] {
    std::unique_ptr<lb_bd> b(new lb_bd);
    b->reps = replicas;
    b->N = N;
    if (precision == LB_FP64)
      b->b.reset(new BDT<double>(replicas, bd_params<double>(N, kT, zeta, eta_s, dt, k_fene, R0, eps, sigma, hi,
                                                             degree, power_iters, seed),
                                 x0));
    else
      b->b.reset(new BDT<float>(replicas, bd_params<float>(N, kT, zeta, eta_s, dt, k_fene, R0, eps, sigma, hi,
                                                           degree, power_iters, seed),
                                x0));
    *out = b.release();
    return (int)LB_OK;
  });
}

int lb_bd_set_stream(lb_bd* b, void* stream) {
  if (!b) return LB_ERR_ARG;
  b->stream = (cudaStream_t)stream;
  return LB_OK;
}

int lb_bd_step(lb_bd* b, int64_t n) {
  if (!b || n < 0) return LB_ERR_ARG;
  return bd_guard([&] {
    b->b->step(n, (uint32_t)b->step, b->stream);
    b->step += n;
    return (int)LB_OK;
  });
}

int lb_bd_sync(lb_bd* b) {
  if (!b) return LB_ERR_ARG;
  return bd_guard([&] { return b->b->status(b->stream) ? (int)LB_ERR_FENE : (int)LB_OK; });
}

int lb_bd_get_beads(lb_bd* b, double* x, size_t cap) {
  if (!b || !x) return LB_ERR_ARG;
  if (cap < (size_t)b->reps * 3 * b->N) return LB_ERR_ARG;
  return bd_guard([&] {
    b->b->get(x, b->stream);
    return b->b->status(b->stream) ? (int)LB_ERR_FENE : (int)LB_OK;
  });
}

int64_t lb_bd_get_step(lb_bd* b) { return b ? b->step : -1; }

void lb_bd_destroy(lb_bd* b) { delete b; }

}  // extern "C"
