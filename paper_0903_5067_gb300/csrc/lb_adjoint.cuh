// Adjoint (reverse-mode derivative) of the coupled LB + chain step with the noise held
// fixed, for gradients of a chain observable with respect to the initial bead positions and
// the friction coefficient zeta.
//
// The forward step (see lb_device.cuh) is, per step k:
//   beads:  v_h = v + h F/2m;  x' = x + h v_h;  F_cons(x');  u_b = sum_c w_c(x') J_c/rho_c (a/h);
//           F_c = -zeta (v_h - u_b) + sqrt(2 kT zeta / h) g_b;  F' = F_cons + F_c;
//           v' = v_h + h F'/2m
//   fluid:  n_ps = pull-stream(n*);  n*' = collide(n_ps) + correction(rho, J, f(x', F_c))
// The adjoint runs the same chain of maps backwards: the fluid adjoint lambda(n*) goes
// through the transposed collision Jacobian (node-local) and the push-stream (the transpose
// of the pull); the chain adjoint through the transposed Jacobians of the integrator, the
// friction, the interpolation (including the gradient of the trilinear weights), the
// spreading and force correction, and the Hessian of FENE + WCA.  The bead side produces the
// derivative with respect to (rho, J) of the post-stream state at the <= 8N corner nodes,
// which a small kernel adds into the pushed fluid adjoint.
#pragma once
#include "lb_device.cuh"

namespace gblb {

// dcoef/d(r^2) of the pair force coefficient (force on b = coef * d, see pair_coef)
template <class R>
__device__ __forceinline__ R pair_coef_deriv(R r2, bool bonded, const ChainK<R>& C) {
  R dc = R(0);
  if (r2 < C.rc2) {
    const R s2 = C.sig2 / r2;
    const R s6 = s2 * s2 * s2;
    dc += R(24) * C.eps / (r2 * r2) * (R(-14) * s6 * s6 + R(4) * s6);
  }
  if (bonded && r2 < C.R0sq) {
    const R t = R(1) - r2 / C.R0sq;
    dc -= C.kfene / C.R0sq / (t * t);
  }
  return dc;
}

// xbar_b += sum_j [coef I + 2 coef' d d^T] (Fbar_b - Fbar_j): the chain-force Hessian applied
// to the force adjoint.  Positions in shared memory (hi, lo); by nt threads (whole warps; tid: this
// one's number among them), lanes per bead as in chain_forces_block; the result is added to out.
template <class R>
__device__ __forceinline__ void chain_force_vjp_block(const R* __restrict__ sh, const R* __restrict__ sl,
                                                      const R* __restrict__ fbar, const ChainK<R>& C,
                                                      R* __restrict__ out, const int tid, const int nt) {
  const int N = C.N;
  int lanes = 1;  // (more than N lanes would add zeros)
  while (lanes < 32 && lanes < N && lanes * 2 * N <= (int)blockDim.x) lanes *= 2;
  const int per = nt / lanes;
  const int lane = tid % lanes;
  for (int base = 0; base < N; base += per) {
    const int b = base + tid / lanes;
    R acc[3] = {R(0), R(0), R(0)};
    if (b < N) {
      for (int j = lane; j < N; j += lanes) {
        if (j == b) continue;
        R d[3], D[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          d[q] = pair_delta<R>(sh[3 * b + q], sl[3 * b + q], sh[3 * j + q], sl[3 * j + q], C.box, C.half_box);
          D[q] = fbar[3 * b + q] - fbar[3 * j + q];
        }
        const R r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
        const bool bonded = (j == b - 1) || (j == b + 1);
        const R c = pair_coef<R>(r2, bonded, C, C.status);
        const R cp = pair_coef_deriv<R>(r2, bonded, C);
        const R dD = d[0] * D[0] + d[1] * D[1] + d[2] * D[2];
#pragma unroll
        for (int q = 0; q < 3; ++q) acc[q] += c * D[q] + R(2) * cp * dD * d[q];
      }
    }
    for (int o = lanes / 2; o > 0; o /= 2) {
#pragma unroll
      for (int q = 0; q < 3; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o, lanes);
    }
    if (b < N && lane == 0) {
#pragma unroll
      for (int q = 0; q < 3; ++q) out[3 * b + q] += acc[q];
    }
  }
}

// Vector-Jacobian product of force_moments with respect to (rho, J, dJ).
template <class R>
__device__ __forceinline__ void force_moments_vjp(R rho, R jx, R jy, R jz, R dx, R dy, R dz, R gs, R gb,
                                                  const R dmb[10], R& rhob, R Jb[3], R dJb[3]) {
  const R ir = R(1) / rho;
  const R ux = (jx + R(0.5) * dx) * ir, uy = (jy + R(0.5) * dy) * ir, uz = (jz + R(0.5) * dz) * ir;
  const R cs = R(0.5) * (R(1) + gs);
  const R cdiag = (R(1) + gb) / R(3) - R(2) / R(3) * cs;
  const R Pxx = dmb[4] + R(2) * dmb[5];
  const R Pyy = dmb[4] - dmb[5] + dmb[6];
  const R Pzz = dmb[4] - dmb[5] - dmb[6];
  const R Pxy = dmb[7], Pyz = dmb[8], Pxz = dmb[9];
  const R udb = cdiag * (Pxx + Pyy + Pzz);
  // adjoint of U'
  const R Ux = R(2) * cs * dx * Pxx + cs * (dy * Pxy + dz * Pxz) + udb * dx;
  const R Uy = R(2) * cs * dy * Pyy + cs * (dx * Pxy + dz * Pyz) + udb * dy;
  const R Uz = R(2) * cs * dz * Pzz + cs * (dy * Pyz + dx * Pxz) + udb * dz;
  // adjoint of dJ: direct (modes 1..3), through the stress products, through U'
  dJb[0] = dmb[1] + R(2) * cs * ux * Pxx + cs * (uy * Pxy + uz * Pxz) + udb * ux + R(0.5) * Ux * ir;
  dJb[1] = dmb[2] + R(2) * cs * uy * Pyy + cs * (ux * Pxy + uz * Pyz) + udb * uy + R(0.5) * Uy * ir;
  dJb[2] = dmb[3] + R(2) * cs * uz * Pzz + cs * (uy * Pyz + ux * Pxz) + udb * uz + R(0.5) * Uz * ir;
  Jb[0] = Ux * ir;
  Jb[1] = Uy * ir;
  Jb[2] = Uz * ir;
  rhob = -(ux * Ux + uy * Uy + uz * Uz) * ir;
}

// a-bar_k = sum_i w_i e_k(c_i) nbar_i: adjoint of the scaled moments from the adjoint of
// the populations they produce (n_i = w_i sum_k e_k(c_i) a_k)
template <class R>
__device__ __forceinline__ void scaled_moment_adjoint(const R nb[Q], R ab[Q]) {
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    R acc = R(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const int c = basis(k, i) * w36(i);
      if (c != 0) acc += R(c) * nb[i];
    }
    ab[k] = acc * (R(1) / R(36));
  }
}

// ---------------------------------------------------------------------------------------
// fluid adjoint of one step: lambda(n*_k) from lambda(n*_{k+1}), every node
//   n_ps(r) = pull(n*_k) ; n*_{k+1}(r) = collide(n_ps(r))   (corrections handled sparsely)
//   nbar_ps(r) = J_collide(r)^T lambda_{k+1}(r);  lambda_k,i(r - e_i) = nbar_ps,i(r)   (push)
// ---------------------------------------------------------------------------------------
// Launched with programmatic stream serialization after the previous reverse step's bead
// adjoint: it waits for that grid (which has added its forced-node terms to lam_in) before
// reading, then releases the bead adjoint of its own step, which runs beside it (see
// k_adj_bead).
template <class S, class R, bool DEV, bool NOISE>
__global__ void __launch_bounds__(256) k_adj_lb(const S* __restrict__ state, const R* __restrict__ lam_in,
                                                 R* __restrict__ lam_out, const FluidK<R> P, const uint32_t step_arg) {
  grid_dependency_wait();
  allow_dependent_launch();
  const uint32_t step = launch_step(P, step_arg);
  const unsigned L = P.L;
  const unsigned x = blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned y = blockIdx.y * blockDim.y + threadIdx.y;
  const unsigned z = blockIdx.z;
  if (x >= L || y >= L) return;
  const unsigned node = x + L * (y + L * z);
  unsigned nb_idx[Q];  // node r - e_i: source of the pull, target of the push
  R n[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const unsigned sx = (x + L - (unsigned)(cx(i) + 0)) % L;
    const unsigned sy = (y + L - (unsigned)(cy(i) + 0)) % L;
    const unsigned sz = (z + L - (unsigned)(cz(i) + 0)) % L;
    nb_idx[i] = sx + L * (sy + L * sz);
    n[i] = ld<S, R>(state + (unsigned long long)i * P.plane + nb_idx[i]);
  }
  R m[10];
  moments_0_9<R>(n, m);
  const R rho = DEV ? P.rho0 + m[0] : m[0];
  const R jx = m[1], jy = m[2], jz = m[3];
  const R ir = R(1) / rho;
  R lb_[Q], ab[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) lb_[i] = lam_in[(unsigned long long)i * P.plane + node];
  scaled_moment_adjoint<R>(lb_, ab);
  // m-bar from the scaled-moment map a(m)
  R mb[10];
  mb[0] = ab[0];
  mb[1] = ab[1] * R(InvB<1>::v);
  mb[2] = ab[2] * R(InvB<2>::v);
  mb[3] = ab[3] * R(InvB<3>::v);
  R Eb[10];
#pragma unroll
  for (int k = 4; k < 10; ++k) {
    mb[k] = P.am[k] * ab[k];
    Eb[k] = P.ae[k] * ab[k];
  }
  const R E4 = (jx * jx + jy * jy + jz * jz) * ir, E5 = (R(2) * jx * jx - jy * jy - jz * jz) * ir;
  const R E6 = (jy * jy - jz * jz) * ir, E7 = jx * jy * ir, E8 = jy * jz * ir, E9 = jx * jz * ir;
  mb[0] -= (Eb[4] * E4 + Eb[5] * E5 + Eb[6] * E6 + Eb[7] * E7 + Eb[8] * E8 + Eb[9] * E9) * ir;
  mb[1] += (R(2) * jx * Eb[4] + R(4) * jx * Eb[5] + jy * Eb[7] + jz * Eb[9]) * ir;
  mb[2] += (R(2) * jy * Eb[4] - R(2) * jy * Eb[5] + R(2) * jy * Eb[6] + jx * Eb[7] + jz * Eb[8]) * ir;
  mb[3] += (R(2) * jz * Eb[4] - R(2) * jz * Eb[5] - R(2) * jz * Eb[6] + jy * Eb[8] + jx * Eb[9]) * ir;
  if (NOISE && rho > R(0)) {
    // a_k += ag_k sqrt(rho) g_k:  d/drho = ag_k g_k / (2 sqrt(rho))
    R acc = R(0);
    fluid_noise<R>(step, node, P.rk, P.ncalls > 1, NoiseScale<R>(R(1)),
                   [&](int j, R g) { acc += P.ag[4 + j] * g * ab[4 + j]; }, P.tab);
    mb[0] += acc * R(0.5) / sqrt(rho);
  }
  // nbar_ps,i = sum_k e_k(c_i) mb_k, pushed to r - e_i
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    R acc = R(0);
#pragma unroll
    for (int k = 0; k < 10; ++k) {
      const int c = basis(k, i);
      if (c != 0) acc += R(c) * mb[k];
    }
    lam_out[(unsigned long long)i * P.plane + nb_idx[i]] = acc;
  }
}

// What the chain part of the adjoint of a step needs of the forward step alone: for each step of a
// segment one region of global memory, written by k_adj_prep.
template <class R>
struct AdjPrep {
  R *vh, *ub, *g, *fc, *sx, *sl;  // 3N each: half-step velocity, fluid velocity, noise, coupling force,
                                  // drifted position (high, low)
  R* gw;       // 3 x 8N weight gradients (per unit length) of the corner entries
  R* w;        // 8N trilinear weights
  R* mom;      // 4 x 8N post-stream density and momentum at the entries' nodes
  R* uf;       // 3 x 8N force density on the u-th forced node
  int* order;  // 8N entries grouped by node, in entry order within a node
  int* first;  // 8N + 1: the u-th node's entries are order[first[u]] .. order[first[u + 1] - 1]
  int* slot;   // 8N: the entry's node u
  int* node;   // 8N: index of the u-th forced node
  int* nu;     // number of forced nodes
  __host__ __device__ int carve(unsigned char* base, int N) {  // returns its size, a multiple of 16
    int off = 0;
    auto take = [&](int bytes) {
      unsigned char* q = base + off;
      off += (bytes + 15) / 16 * 16;
      return q;
    };
    const int r = (int)sizeof(R), n3 = 3 * N, ne = 8 * N;
    vh = (R*)take(n3 * r);
    ub = (R*)take(n3 * r);
    g = (R*)take(n3 * r);
    fc = (R*)take(n3 * r);
    sx = (R*)take(n3 * r);
    sl = (R*)take(n3 * r);
    gw = (R*)take(3 * ne * r);
    w = (R*)take(ne * r);
    mom = (R*)take(4 * ne * r);
    uf = (R*)take(3 * ne * r);
    order = (int*)take(ne * 4);
    first = (int*)take((ne + 1) * 4);
    slot = (int*)take(ne * 4);
    node = (int*)take(ne * 4);
    nu = (int*)take(4);
    return off;
  }
};

// shared memory of k_adj_prep: positions, sort keys, leader slots
template <class R>
__host__ __device__ inline size_t adj_prep_smem(int N) {
  size_t M = 1;
  while (M < 8 * (size_t)N) M <<= 1;
  return 6 * (size_t)N * sizeof(R) + 32 + M * 8 + 8 * (size_t)N * 4 + 64;
}

// A checkpoint of the forward pass: the populations (16-byte words) and the bead arrays behind them
// (4-byte words) to checkpoint (*d_step - k0) / K of those that lie `stride` bytes apart from `to` on
__global__ static void k_adj_checkpoint(const int4* __restrict__ pops, size_t npops, const int* __restrict__ beads, int nbeads,
                                        unsigned char* __restrict__ to, size_t stride, const uint32_t* __restrict__ d_step,
                                        uint32_t k0, uint32_t K) {
  unsigned char* dst = to + (size_t)((*d_step - k0) / K) * stride;
  int4* p = reinterpret_cast<int4*>(dst);
  int* b = reinterpret_cast<int*>(dst + npops * 16);
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x, n = (size_t)gridDim.x * blockDim.x;
  for (size_t i = t; i < npops; i += n) p[i] = pops[i];
  for (size_t i = t; i < (size_t)nbeads; i += n) b[i] = beads[i];
}

// xbar of the last step: d/dx of sum (x - x0)^2 from the FP64 positions
template <class R>
__global__ void k_adj_seed(const double* __restrict__ x0, const double* __restrict__ x, int n, R* __restrict__ xbar) {
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x)
    xbar[t] = (R)(2.0 * (x[t] - x0[t]));
}

// The forward recomputation of the bead step for the steps step_arg + j, j = blockIdx.x, of a segment,
// a block per step: it depends on no other step and on no adjoint, so it is off the chain of
// reverse steps (of whose 15 us per step, N = 16, it took 5 as the first part of k_adj_bead).
// The state of step j lies j * state_stride bytes behind `state` and the arrays of C, its region
// j * prep_stride bytes behind `prep`.
template <class S, class R, bool DEV>
__global__ void __launch_bounds__(512) k_adj_prep(const S* __restrict__ state, const FluidK<R> P, const ChainK<R> C,
                                                   unsigned char* prep, int prep_stride, size_t state_stride,
                                                   const uint32_t step_arg) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int N = C.N, ne = 8 * N, tid = threadIdx.x, nt = blockDim.x, L = (int)P.L;
  const uint32_t step = launch_step(P, step_arg) + blockIdx.x;
  auto behind = [&](const void* q) {
    return reinterpret_cast<const unsigned char*>(q) + (size_t)blockIdx.x * state_stride;
  };
  const S* pop = reinterpret_cast<const S*>(behind(state));
  const R *cx_ = reinterpret_cast<const R*>(behind(C.x)), *cxl = reinterpret_cast<const R*>(behind(C.xl)),
          *cv = reinterpret_cast<const R*>(behind(C.v)), *cF = reinterpret_cast<const R*>(behind(C.F));
  AdjPrep<R> A;
  A.carve(prep + (size_t)blockIdx.x * prep_stride, N);
  R* sx = reinterpret_cast<R*>(smem);
  R* sl = sx + 3 * N;
  for (int t = tid; t < 3 * N; t += nt) {
    R vh, hi, lo;
    int im = 0;
    drift<R>(C, cv[t], cF[t], cx_[t], cxl[t], im, vh, hi, lo);
    A.vh[t] = vh;
    A.sx[t] = sx[t] = hi;
    A.sl[t] = sl[t] = lo;
  }
  __syncthreads();
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(
      (reinterpret_cast<uintptr_t>(smem + 6 * N * sizeof(R)) + 15) & ~(uintptr_t)15);
  int M = 1;
  while (M < ne) M <<= 1;
  for (int e = tid; e < M; e += nt) {
    if (e >= ne) {
      keys[e] = ~0ull;
      continue;
    }
    const int b = e >> 3, c = e & 7;
    const int d3[3] = {c & 1, (c >> 1) & 1, (c >> 2) & 1};
    R fr[3];
    int cl[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      R unused;
      const R xh = sx[3 * b + q];
      cl[q] = cell_of<R>(xh, C.a, L, unused);
      const R f = floor(xh / C.a);
      fr[q] = (fma(-f, C.a, xh) + sl[3 * b + q]) / C.a;
    }
    R ws[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) ws[q] = d3[q] ? fr[q] : R(1) - fr[q];
    // dw/dx_q = (+-1/a) * product of the other two factors
    A.gw[0 * ne + e] = (d3[0] ? R(1) : R(-1)) * ws[1] * ws[2] / C.a;
    A.gw[1 * ne + e] = (d3[1] ? R(1) : R(-1)) * ws[0] * ws[2] / C.a;
    A.gw[2 * ne + e] = (d3[2] ? R(1) : R(-1)) * ws[0] * ws[1] / C.a;
    const int qx = (cl[0] + d3[0]) % L, qy = (cl[1] + d3[1]) % L, qz = (cl[2] + d3[2]) % L;
    R mom[4];
    gather_node<S, R, DEV>(pop, P, qx, qy, qz, mom);
    A.w[e] = ws[0] * ws[1] * ws[2];
#pragma unroll
    for (int q = 0; q < 4; ++q) A.mom[q * ne + e] = mom[q];
    keys[e] = ((unsigned long long)(unsigned)(qx + L * (qy + L * qz)) << 32) | (unsigned)e;
  }
  __syncthreads();
  for (int b = tid; b < N; b += nt) {
    R ub[3] = {R(0), R(0), R(0)};
    for (int c = 0; c < 8; ++c) {
      const int e = 8 * b + c;
      const R w = A.w[e], ir = R(1) / A.mom[e];
      ub[0] += w * A.mom[ne + e] * ir;
      ub[1] += w * A.mom[2 * ne + e] * ir;
      ub[2] += w * A.mom[3 * ne + e] * ir;
    }
    R g[4] = {R(0), R(0), R(0), R(0)};
    if (C.amp != R(0)) gauss4<R>(step, (uint32_t)b, 0u, C.k0, C.k1, g);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int t = 3 * b + q;
      const R u = ub[q] * C.u_scale;
      A.ub[t] = u;
      A.g[t] = g[q];
      A.fc[t] = -C.zeta * (A.vh[t] - u) + C.amp * g[q];
    }
  }
  // entries ordered by node (and by entry within a node)
  if (ne <= nt) {
    // few entries: each thread places its key by its rank among all keys (distinct: the entry
    // index is in the low bits), two barriers instead of the bitonic network's log2(M)^2 / 2
    const unsigned long long mine = tid < ne ? keys[tid] : 0ull;
    int rank = 0;
    if (tid < ne)
      for (int j = 0; j < ne; ++j) rank += keys[j] < mine;
    __syncthreads();
    if (tid < ne) keys[rank] = mine;
    __syncthreads();
  } else {
    for (int k = 2; k <= M; k <<= 1) {
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int i = tid; i < M; i += nt) {
          const int ixj = i ^ j;
          if (ixj > i) {
            const unsigned long long ka = keys[i], kb = keys[ixj];
            const bool up = (i & k) == 0;
            if ((ka > kb) == up) {
              keys[i] = kb;
              keys[ixj] = ka;
            }
          }
        }
        __syncthreads();
      }
    }
  }
  int* lead = reinterpret_cast<int*>(keys + M);
  if (tid < 32) {
    int base = 0;
    for (int c0 = 0; c0 < ne; c0 += 32) {
      const int i = c0 + tid;
      int l = 0;
      if (i < ne) l = (i == 0) || ((keys[i] >> 32) != (keys[i - 1] >> 32));
      const unsigned mask = __ballot_sync(0xffffffffu, l);
      if (i < ne) lead[i] = l ? base + __popc(mask & ((1u << tid) - 1u)) : -1;
      base += __popc(mask);
    }
    if (tid == 0) {
      *A.nu = base;
      A.first[base] = ne;
    }
  }
  __syncthreads();
  for (int i = tid; i < ne; i += nt) {
    A.order[i] = (int)(keys[i] & 0xffffffffu);
    const int u = lead[i];
    if (u < 0) continue;
    const int node = (int)(keys[i] >> 32);
    R f[3] = {R(0), R(0), R(0)};
    for (int r = i; r < ne && (int)(keys[r] >> 32) == node; ++r) {
      const int e = (int)(keys[r] & 0xffffffffu);
      const int b = e >> 3;
      A.slot[e] = u;
      f[0] -= A.w[e] * A.fc[3 * b + 0] * C.inv_a3;
      f[1] -= A.w[e] * A.fc[3 * b + 1] * C.inv_a3;
      f[2] -= A.w[e] * A.fc[3 * b + 2] * C.inv_a3;
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) A.uf[q * ne + u] = f[q];
    A.first[u] = i;
    A.node[u] = node;
  }
}

// Chain part of the adjoint of one step, one thread block.
// In:  the step's AdjPrep region, lambda(n*_{k+1}) (`lam`), xbar/vbar/fbar of step k+1.
// Out: xbar/vbar/fbar of step k (in place), zbar (+= d/dzeta), and lambda(n*_k) (`lam_out`)
//      completed: lambda_k,i(r - e_i) += rho-bar(r) + c_i . J-bar(r) at the forced nodes r.
// Launched with programmatic stream serialization after k_adj_lb of the same step, which writes
// the rest of lambda(n*_k): everything up to that last addition runs beside it, and the
// addition waits for it.  Bound by the latency of its phases: 19 us alone before the forward
// recomputation moved to k_adj_prep (8 us for ten steps at once), 9.5 us now at N = 16 (copy of the
// region and the adjoints 1.5 us, per-node adjoints and Hessian side by side 1.8, per-bead and
// per-entry adjoints 1.2, integrator, sums and additions 1.6).  (Releasing the next step's k_adj_lb
// from here, before this grid ends, cost more than it gave: its waiting blocks hold the SMs that the
// recomputation beside the sweep needs, 3.39 against 3.28 ms per call at L = 32, T = 100.)
template <class R>
struct AdjK {
  R *xbar, *vbar, *fbar;  // 3N each, in/out across the reverse steps (global)
  double* zbar;           // accumulated d objective / d zeta (global)
  // scratch of one reverse step: carved from the kernel's dynamic shared memory, with the step's
  // AdjPrep region copied in front of it, when in_smem is set (small chains), else global memory
  R *fct, *vhb, *xpb, *hes;  // 3N each
  R* e_rb;      // 4 x 8N (rho-bar, J-bar) per entry
  R* u_fb;      // 3 x 8N: f-bar per unique node
  R* u_rb;      // 4 x 8N: forced-node (rho, J) adjoint per unique node
  R* u_sp;      // 4 x 8N: (rho-bar, J-bar) summed per unique forced node
  R* e_wb;      // 8N: weight adjoint per entry
  R* zb_b;      // N: zeta-bar per bead
  unsigned char* scratch;  // global scratch (in_smem not set)
  int in_smem;
  __host__ __device__ int carve(unsigned char* base, int N) {
    int off = 0;
    auto take = [&](int bytes) {
      unsigned char* q = base + off;
      off += (bytes + 15) / 16 * 16;
      return q;
    };
    const int r = (int)sizeof(R), n3 = 3 * N, ne = 8 * N;
    fct = (R*)take(n3 * r);
    vhb = (R*)take(n3 * r);
    xpb = (R*)take(n3 * r);
    hes = (R*)take(n3 * r);
    e_rb = (R*)take(4 * ne * r);
    u_fb = (R*)take(3 * ne * r);
    u_rb = (R*)take(4 * ne * r);
    u_sp = (R*)take(4 * ne * r);
    e_wb = (R*)take(ne * r);
    zb_b = (R*)take(N * r);
    return off;
  }
};

template <class R>
__global__ void __launch_bounds__(512) k_adj_bead(const R* __restrict__ lam, R* __restrict__ lam_out, const FluidK<R> P,
                                                   const ChainK<R> C, const AdjK<R> A0, unsigned char* prep,
                                                   const int prep_bytes) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int N = C.N, ne = 8 * N, tid = threadIdx.x, nt = blockDim.x, L = (int)P.L;
  AdjK<R> A = A0;
  AdjPrep<R> F;
  if (A0.in_smem) {
    F.carve(smem, N);
    A.carve(smem + prep_bytes, N);
  } else {
    F.carve(prep, N);
    A.carve(A0.scratch, N);
  }
  const R h = C.h;
  // d/dzeta so far, read now so that the update at the end is a plain store (no other grid
  // writes it while this one runs: the previous reverse step has completed)
  const double zbar_in = tid == nt - 32 ? *A.zbar : 0.0;
  for (int t = tid; t < 3 * N; t += nt) {
    // adjoint of the total force of step k+1 and of v_h (from v' = v_h + h F'/2m)
    const R vb = A.vbar[t];
    A.fct[t] = A.fbar[t] + h / (R(2) * C.m) * vb;
    A.vhb[t] = vb;
    A.xpb[t] = A.xbar[t];  // x' is the position output of this step
    A.hes[t] = R(0);
  }
  if (A0.in_smem) {
    const int4* from = reinterpret_cast<const int4*>(prep);
    int4* to = reinterpret_cast<int4*>(smem);
    for (int i = nt - 1 - tid; i < prep_bytes / 16; i += nt) to[i] = from[i];
  }
  __syncthreads();
  const int nu = *F.nu;
  // per unique node p: force-correction adjoint -> fbar(p), forced-node (rho, J) adjoint; on the
  // warps left over the chain forces: Hessian . F_cons-bar (F_cons-bar = F_total-bar)
  const int nodew = (nu + 31) / 32 * 32;
  const int h0 = nodew + 128 <= nt ? nodew : 0;  // the Hessian's first thread
  for (int u = tid; u < nu; u += nt) {
    const int node = F.node[u], e0 = F.order[F.first[u]];
    const R rho = F.mom[e0], jx = F.mom[ne + e0], jy = F.mom[2 * ne + e0], jz = F.mom[3 * ne + e0];
    R nb[Q], ab[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) nb[q] = lam[(unsigned long long)q * P.plane + (unsigned)node];
    scaled_moment_adjoint<R>(nb, ab);
    R dmb[10];
    dmb[0] = R(0);
    dmb[1] = ab[1] * R(InvB<1>::v);
    dmb[2] = ab[2] * R(InvB<2>::v);
    dmb[3] = ab[3] * R(InvB<3>::v);
    dmb[4] = ab[4] * R(InvB<4>::v);
    dmb[5] = ab[5] * R(InvB<5>::v);
    dmb[6] = ab[6] * R(InvB<6>::v);
    dmb[7] = ab[7] * R(InvB<7>::v);
    dmb[8] = ab[8] * R(InvB<8>::v);
    dmb[9] = ab[9] * R(InvB<9>::v);
    R rb, Jb[3], dJb[3];
    force_moments_vjp<R>(rho, jx, jy, jz, F.uf[u] * C.dJ_scale, F.uf[ne + u] * C.dJ_scale, F.uf[2 * ne + u] * C.dJ_scale,
                         P.gs, P.gb, dmb, rb, Jb, dJb);
    A.u_fb[u] = dJb[0] * C.dJ_scale;
    A.u_fb[ne + u] = dJb[1] * C.dJ_scale;
    A.u_fb[2 * ne + u] = dJb[2] * C.dJ_scale;
    A.u_rb[u] = rb;
    A.u_rb[ne + u] = Jb[0];
    A.u_rb[2 * ne + u] = Jb[1];
    A.u_rb[3 * ne + u] = Jb[2];
  }
  if (tid >= h0) chain_force_vjp_block<R>(F.sx, F.sl, A.fct, C, A.hes, tid - h0, nt - h0);
  __syncthreads();
  // ---- per bead and component: spreading, friction adjoints ----------------------------
  for (int t = tid; t < 3 * N; t += nt) {
    const int b = t / 3, q = t - 3 * b;
    R fcb = A.fct[t];
    for (int c = 0; c < 8; ++c) {
      const int e = 8 * b + c;
      fcb -= F.w[e] * C.inv_a3 * A.u_fb[q * ne + F.slot[e]];
    }
    // friction + noise: F_c = -zeta (v_h - u_b) + amp(zeta) g
    A.vhb[t] -= C.zeta * fcb;
    A.fct[t] = fcb;  // from here on the adjoint of F_c (the Hessian has used that of the total)
  }
  __syncthreads();
  // ---- per entry: interpolation u_b = sum_e w_e J_e / rho_e (a/h), weight adjoint ---------
  for (int e = tid; e < ne; e += nt) {
    const int b = e >> 3, u = F.slot[e];
    const R fc[3] = {F.fc[3 * b], F.fc[3 * b + 1], F.fc[3 * b + 2]};
    const R fbx = A.u_fb[u], fby = A.u_fb[ne + u], fbz = A.u_fb[2 * ne + u];
    // spreading: f(p) = -sum_e w_e F_c,b / a^3
    R wb = -C.inv_a3 * (fc[0] * fbx + fc[1] * fby + fc[2] * fbz);
    R Ub[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) Ub[q] = C.zeta * A.fct[3 * b + q];
    const R w = F.w[e], rho = F.mom[e], ir = R(1) / rho;
    const R J[3] = {F.mom[ne + e], F.mom[2 * ne + e], F.mom[3 * ne + e]};
    R ue[3], uJ = R(0);
#pragma unroll
    for (int q = 0; q < 3; ++q) ue[q] = J[q] * ir * C.u_scale;
    wb += ue[0] * Ub[0] + ue[1] * Ub[1] + ue[2] * Ub[2];
    R ueb[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      ueb[q] = w * Ub[q];
      uJ += J[q] * ueb[q];
    }
    A.e_rb[e] = -C.u_scale * uJ * ir * ir;
#pragma unroll
    for (int q = 0; q < 3; ++q) A.e_rb[(q + 1) * ne + e] = C.u_scale * ueb[q] * ir;
    A.e_wb[e] = wb;
  }
  __syncthreads();
  // ---- integrator: x' = x + h v_h ; v_h = v + h F / 2m ------------------------------------
  for (int t = nt - 1 - tid; t < 3 * N; t += nt) {
    const int b = t / 3, q = t - 3 * b;
    R xpb = R(0);
    for (int c = 0; c < 8; ++c) xpb += A.e_wb[8 * b + c] * F.gw[q * ne + 8 * b + c];  // trilinear weight gradient
    xpb = (A.xpb[t] + xpb) + A.hes[t];
    const R vhb = A.vhb[t] + h * xpb;
    A.xbar[t] = xpb;
    A.vbar[t] = vhb;
    A.fbar[t] = h / (R(2) * C.m) * vhb;
  }
  // ---- sparse (rho, J) adjoint per unique node, entries summed in entry order -----------
  for (int u = tid; u < nu; u += nt) {
    R v[4] = {A.u_rb[u], A.u_rb[ne + u], A.u_rb[2 * ne + u], A.u_rb[3 * ne + u]};
    for (int r = F.first[u]; r < F.first[u + 1]; ++r) {
      const int e = F.order[r];
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] += A.e_rb[q * ne + e];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) A.u_sp[q * ne + u] = v[q];
  }
  // ---- zeta-bar: per bead, then a fixed-order block sum ------------------------------------
  for (int b = tid; b < N; b += nt) {
    const R damp = C.zeta > R(0) ? C.amp / (R(2) * C.zeta) : R(0);
    R zb = R(0);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int t = 3 * b + q;
      zb += A.fct[t] * (-(F.vh[t] - F.ub[t]) + damp * F.g[t]);
    }
    A.zb_b[b] = zb;
  }
  __syncthreads();
  if (tid >= nt - 32) {  // the last warp: in a fixed tree
    double acc = 0.0;
    for (int b = tid & 31; b < N; b += 32) acc += (double)A.zb_b[b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (tid == nt - 32) *A.zbar = zbar_in + acc;
  }
  // ---- lambda_k,i(r - e_i) += rho-bar(r) + c_i . J-bar(r) at the forced nodes, once the
  //      adjoint LB kernel of this step has written lambda_k (each (i, r - e_i) target belongs
  //      to one forced node r, so the additions do not collide) --------------------------
  //      In chunks of kAddBatch targets per thread: all loads of a chunk, then its stores (one
  //      memory round trip per chunk instead of one per target); the first chunk's targets and
  //      terms are formed before the wait.
  const int total = Q * nu;
  constexpr int kAddBatch = 8;
  unsigned long long at[kAddBatch];
  R v[kAddBatch];
  auto form = [&](int k0) {
#pragma unroll
    for (int j = 0; j < kAddBatch; ++j) {
      const int k = k0 + j * nt;
      if (k >= total) break;
      const int i = k / nu, u = k - i * nu;
      const int node = F.node[u];
      const int x = node % L, y = (node / L) % L, z = node / (L * L);
      const int ex = unpack_component(pack_component(0), i), ey = unpack_component(pack_component(1), i),
                ez = unpack_component(pack_component(2), i);
      const int sx = (x - ex + L) % L, sy = (y - ey + L) % L, sz = (z - ez + L) % L;
      v[j] = A.u_sp[u] + R(ex) * A.u_sp[ne + u] + R(ey) * A.u_sp[2 * ne + u] + R(ez) * A.u_sp[3 * ne + u];
      at[j] = (unsigned long long)i * P.plane + (unsigned)(sx + L * (sy + L * sz));
    }
  };
  form(tid);
  grid_dependency_wait();
  for (int k0 = tid; k0 < total; k0 += kAddBatch * nt) {
    if (k0 != tid) form(k0);
    R old[kAddBatch];
#pragma unroll
    for (int j = 0; j < kAddBatch; ++j) {
      if (k0 + j * nt >= total) break;
      old[j] = lam_out[at[j]];
    }
#pragma unroll
    for (int j = 0; j < kAddBatch; ++j) {
      if (k0 + j * nt >= total) break;
      lam_out[at[j]] = old[j] + v[j];
    }
  }
}

// xbar += Hessian(F_cons)(x) . fbar at a given configuration (the initial force F_0 =
// F_cons(x_0) depends on x_0)
template <class R>
__global__ void __launch_bounds__(512) k_chain_force_vjp(const ChainK<R> C, const R* __restrict__ fbar,
                                                          R* __restrict__ xbar) {
  extern __shared__ __align__(16) unsigned char smem[];
  R* sx = reinterpret_cast<R*>(smem);
  R* sl = sx + 3 * C.N;
  for (int t = threadIdx.x; t < 3 * C.N; t += blockDim.x) {
    sx[t] = C.x[t];
    sl[t] = C.xl[t];
  }
  __syncthreads();
  chain_force_vjp_block<R>(sx, sl, fbar, C, xbar, threadIdx.x, blockDim.x);
}

}  // namespace gblb
