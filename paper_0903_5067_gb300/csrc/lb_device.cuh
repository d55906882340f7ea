// Device code of the fluctuating D3Q19 LB + bead-spring chain step.
//
// Storage: populations in structure-of-arrays planes pop[i][z][y][x] (plane stride
// `plane` elements), two buffers A/B.  FP32/BF16/FP16 contexts store the deviation
// n_i - w_i rho0 (DEV = true), the FP64 context the full n_i.  A step reads buffer A
// (post-collision populations of the previous step, "pull" storage) and writes B.
//
// One step = k_bead_step (one thread block, or a cluster of up to 8: velocity Verlet,
// FENE/WCA, interpolation, friction + noise, spreading -> population corrections at the nodes around
// the beads, in a field of the populations' layout, with a list of the nodes), k_lb_step (every
// node: pull-stream, moments, relaxation + noise, back-transform) and the force corrections, added to
// B by k_apply_pending or, kept pending, by the next step's kernels where they read.  The bead kernel
// and the LB kernel read only A, so they are independent; the correction is additive on the
// post-collision populations because the collision conserves the density and momentum it depends on.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "d3q19.cuh"
#include "philox.cuh"

namespace gblb {

enum : unsigned { ST_FENE = 1u, ST_NONFINITE = 2u, ST_TIMEOUT = 4u };

// ---------------------------------------------------------------------------------------
// storage <-> arithmetic conversions
// ---------------------------------------------------------------------------------------
template <class S, class R>
__device__ __forceinline__ R ld(const S* p) { return (R)(*p); }
template <>
__device__ __forceinline__ float ld<__nv_bfloat16, float>(const __nv_bfloat16* p) { return __bfloat162float(*p); }
template <>
__device__ __forceinline__ float ld<__half, float>(const __half* p) { return __half2float(*p); }

template <class S, class R>
__device__ __forceinline__ void st(S* p, R v) { *p = (S)v; }
template <>
__device__ __forceinline__ void st<__nv_bfloat16, float>(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
template <>
__device__ __forceinline__ void st<__half, float>(__half* p, float v) { *p = __float2half_rn(v); }

// two consecutive elements (the first at an even element offset, so 2 sizeof(S)-aligned) in
// one access: 8 bytes for FP32, 16 for FP64, 4 for the 16-bit formats
template <class S, class R>
__device__ __forceinline__ void ld2(const S* p, R& a, R& b);
template <>
__device__ __forceinline__ void ld2<float, float>(const float* p, float& a, float& b) {
  const float2 v = *reinterpret_cast<const float2*>(p);
  a = v.x;
  b = v.y;
}
template <>
__device__ __forceinline__ void ld2<double, double>(const double* p, double& a, double& b) {
  const double2 v = *reinterpret_cast<const double2*>(p);
  a = v.x;
  b = v.y;
}
template <>
__device__ __forceinline__ void ld2<__nv_bfloat16, float>(const __nv_bfloat16* p, float& a, float& b) {
  const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(p);
  a = __low2float(v);
  b = __high2float(v);
}
template <>
__device__ __forceinline__ void ld2<__half, float>(const __half* p, float& a, float& b) {
  const __half2 v = *reinterpret_cast<const __half2*>(p);
  a = __low2float(v);
  b = __high2float(v);
}
template <class S, class R>
__device__ __forceinline__ void st2(S* p, R a, R b);
template <>
__device__ __forceinline__ void st2<float, float>(float* p, float a, float b) {
  *reinterpret_cast<float2*>(p) = make_float2(a, b);
}
template <>
__device__ __forceinline__ void st2<double, double>(double* p, double a, double b) {
  *reinterpret_cast<double2*>(p) = make_double2(a, b);
}
template <>
__device__ __forceinline__ void st2<__nv_bfloat16, float>(__nv_bfloat16* p, float a, float b) {
  *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(a, b);
}
template <>
__device__ __forceinline__ void st2<__half, float>(__half* p, float a, float b) {
  *reinterpret_cast<__half2*>(p) = __floats2half2_rn(a, b);
}

// 1/rho for the LB kernel: the hardware reciprocal in single precision (1 ulp; the density is
// a normal number), correctly rounded division in double
template <class R>
__device__ __forceinline__ R lb_rcp(R x) { return R(1) / x; }
template <>
__device__ __forceinline__ float lb_rcp<float>(float x) { return approx_rcp(x); }

// ---------------------------------------------------------------------------------------
// kernel parameter blocks (passed by value)
// ---------------------------------------------------------------------------------------
template <class R>
struct FluidK {
  unsigned L;
  unsigned long long plane;  // elements between population planes
  R rho0;
  R gs, gb;        // relaxation eigenvalues: shear modes 5..9, bulk mode 4 (kinetic modes: 0)
  // the same relaxation and noise in terms of the scaled moments a_k = m*_k / b_k used by the
  // back-transform: a_k = am_k m_k + ae_k m_eq,k + ag_k sqrt(rho) g_k  (k = 4..18; ag_k b_k = sqrt(mu b_k
  // (1 - gamma_k^2)), 0 for a silent mode)
  R am[Q], ae[Q], ag[Q];
  // the same times w_2 = 1/36, the weight of the next-nearest velocities, which the forward
  // kernel's back-transform then needs no more multiplications for
  R wam[Q], wae[Q], wag[Q];
  uint32_t k0, k1; // Philox key of the fluid stream
  RoundKeys rk;    // its ten round keys
  int ncalls;      // Philox calls per node: 0 (noise off), 1 (stress modes only), 2 (all)
  int body_on;     // uniform body force
  R body_dJ[3];    // lattice momentum it adds per step and node: f h^2 / a
  unsigned long long* nonpos;  // counter of non-positive densities met by the noise
  int pdl;         // launch chaining of the LB kernel: bit 0 waits for the previous grid before
                   // reading, bit 1 waits for it before completing (see k_lb_step)
  unsigned row, mag_row, rows;  // k_lb_step: threads per row segment, its reciprocal, rows per block
  NoiseTab tab;    // double precision: the noise's radii and angles
  // null, or a device counter the step kernels add their step argument to (graph replays of a
  // fixed sequence of launches at other step numbers)
  const uint32_t* d_step;
};

// the step number of a launch: its argument, offset by the device counter when there is one
template <class R>
__device__ __forceinline__ uint32_t launch_step(const FluidK<R>& P, uint32_t step) {
  return P.d_step ? *P.d_step + step : step;
}

// *p = v on the stream (a device step counter before a graph replay)
template <class T>
__global__ void k_store_value(T* p, T v) { *p = v; }
template <class T>
__global__ void k_add_value(T* p, T v) { *p += v; }

template <class R>
struct ChainK {
  int N;
  R m, zeta, kfene, R0sq, eps, sig2, rc2;
  R h, a, box, half_box;
  // 1/(2m) and 1/a where they are exact (2m, a powers of two): the product is then the quotient,
  // without a division; else 0
  R inv_2m, inv_a;
  R amp;            // sqrt(2 kT zeta / h), 0 without bead noise
  uint32_t k0, k1;  // Philox key of the bead stream
  R ext[3];         // constant external force on each bead
  R u_scale;        // a / h (h: the LB step): lattice -> physical velocity
  R inv_a3;         // 1 / a^3
  R dJ_scale;       // h^2 / a: force density -> lattice momentum per LB step
  int nsub;         // MD steps per LB step (h above is the MD step h_LB / nsub)
  R spread;         // 1 / nsub: each MD step's reaction, averaged over the LB step
  R* fc_hist;       // nsub x 3N coupling forces of the MD substeps
  // bead state (global, 3N each, bead-major).  The bead kernel reads the state at the start
  // of a step from the *_in arrays (normally the same arrays; the adjoint's recomputation
  // reads one saved state and writes the next) and writes the end state to x .. Fc
  const R *x_in, *xl_in, *v_in, *F_in;
  const int* img_in;
  R* x;    // wrapped positions in [0, box): high part
  R* xl;   // low part: position = x + xl + img * box (compensated, ~2x the precision of R)
  int* img;  // periodic image counters
  R* v;
  R* F;    // total force of the last step (F_cons + F_c)
  R* Fc;   // coupling force of the last step
  // scratch (global)
  R* vh;       // 3N half-step velocities
  R* fcons;    // 3N conservative forces
  int* e_node;  // 8N corner nodes
  R* e_w;      // 8N trilinear weights
  R* e_mom;    // 4 x 8N: post-stream rho, Jx, Jy, Jz at the corner node
  int cap;     // 8N
  unsigned* status;
  // FP64 snapshot of the state after each step, written by the bead kernel of step k into
  // slot k mod 2 (3N unwrapped positions x + xl + img box, then 3N velocities), or null
  double* snap;
  double snap_box;  // L a in FP64
};

// Force corrections in flight between consecutive steps of a multi-step run.  The bead kernel
// of step k writes them into a dense correction field of the population layout [i][plane] that is
// zero except at pending nodes, and lists the nodes (some list entries may be empty: node < 0);
// it also marks, in a bit mask over the nodes (one 32-bit word per 32 consecutive
// linear indices), every node that pulls from a corrected node.  The LB kernel of step k+1
// adds the dense field to what it pulls at marked nodes, and the bead kernel of step k+1 to
// what it gathers.  Two slots alternate by step; a bead kernel first clears its slot's dense
// entries and mask words of the list from two steps before, and a flush clears what it
// applies.
template <class R>
struct PendK {
  int have_prev;          // 0: nothing pending (the stored populations are complete)
  const unsigned* prev_mask;  // nodes that pull from the previous step's corrected nodes
  const R* prev_dense;    // the previous step's corrections, dense
  int4* cur_pos;          // this step's list: {node, x, y, z}, node < 0: empty
  int* cur_count;
  R* cur_dense;           // this step's slot of the dense field
  unsigned* cur_mask;     // this step's slot of the mask (cleared of the old list)
  R* apply_to;            // null, or FP32/FP64 populations the old list's corrections, not yet applied
                          // to them, are added to where they are cleared
  int mark;               // 1: mark the pulling nodes of this step's list (deferred steps)
  unsigned long long plane;  // element stride between the 19 planes
  unsigned seg0;             // index of this box's first word in the mask arrays
};

constexpr int kSegShift = 5;  // mask words of 32 consecutive nodes

// ---------------------------------------------------------------------------------------
// moment algebra
// ---------------------------------------------------------------------------------------
// scaled moments a_k = m_k / b_k  ->  populations n_i = w_i sum_k e_k(c_i) a_k: the rest population
// and the pair (2p + 1, 2p + 2) of opposite ones, p a constant after unrolling
template <class R>
__device__ __forceinline__ R pop_of_modes(const R a[Q], int i) {
  R acc = R(0);
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    const int c = basis(k, i);
    if (c != 0) acc += R(c) * a[k];
  }
  return acc * (R(w36(i)) / R(36));
}
template <class R>
__device__ __forceinline__ void pair_of_modes(const R a[Q], const int p, R& n1, R& n2) {
  const int i = 2 * p + 1;
  R S = R(0), D = R(0);
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    const int c = basis(k, i);
    if (c == 0) continue;
    if (odd_mode(k))
      D += R(c) * a[k];
    else
      S += R(c) * a[k];
  }
  const R w = R(w36(i)) / R(36);
  n1 = w * (S + D);
  n2 = w * (S - D);
}
template <class R>
__device__ __forceinline__ void modes_to_pops(const R a[Q], R out[Q]) {
  out[0] = pop_of_modes<R>(a, 0);
#pragma unroll
  for (int p = 0; p < NPAIR; ++p) pair_of_modes<R>(a, p, out[2 * p + 1], out[2 * p + 2]);
}

template <int K>
struct InvB {
  static constexpr double v = 36.0 / (double)norm36(K);
};

// Moment increments (modes 1..9) of a force adding lattice momentum dJ at a node of
// density rho and pre-collision momentum J (second-order forcing reading):
//   dm_1..3 = dJ;  dPi = (1+g_s)/2 (U'dJ + dJU' - 2/3 1 U'.dJ) + (1+g_b)/3 1 U'.dJ,
//   U' = (J + dJ/2)/rho, mapped onto modes 4..9.
template <class R>
__device__ __forceinline__ void force_moments(R rho, R jx, R jy, R jz, R dx, R dy, R dz, R gs,
                                              R gb, R dm[10]) {
  const R ir = R(1) / rho;
  const R ux = (jx + R(0.5) * dx) * ir, uy = (jy + R(0.5) * dy) * ir, uz = (jz + R(0.5) * dz) * ir;
  const R ud = ux * dx + uy * dy + uz * dz;
  const R cs = R(0.5) * (R(1) + gs);
  const R diag = ((R(1) + gb) / R(3) - R(2) / R(3) * cs) * ud;
  const R pxx = R(2) * cs * ux * dx + diag;
  const R pyy = R(2) * cs * uy * dy + diag;
  const R pzz = R(2) * cs * uz * dz + diag;
  dm[0] = R(0);
  dm[1] = dx;
  dm[2] = dy;
  dm[3] = dz;
  dm[4] = pxx + pyy + pzz;
  dm[5] = R(2) * pxx - pyy - pzz;
  dm[6] = pyy - pzz;
  dm[7] = cs * (ux * dy + uy * dx);
  dm[8] = cs * (uy * dz + uz * dy);
  dm[9] = cs * (ux * dz + uz * dx);
}

// scaled moments of the moment increments dm(1) .. dm(9) (the others zero)
template <class R, class F>
__device__ __forceinline__ void scaled_increments(F&& dm, R a[Q]) {
  a[0] = R(0);
  a[1] = dm(1) * R(InvB<1>::v);
  a[2] = dm(2) * R(InvB<2>::v);
  a[3] = dm(3) * R(InvB<3>::v);
  a[4] = dm(4) * R(InvB<4>::v);
  a[5] = dm(5) * R(InvB<5>::v);
  a[6] = dm(6) * R(InvB<6>::v);
  a[7] = dm(7) * R(InvB<7>::v);
  a[8] = dm(8) * R(InvB<8>::v);
  a[9] = dm(9) * R(InvB<9>::v);
#pragma unroll
  for (int k = 10; k < Q; ++k) a[k] = R(0);
}

// ---------------------------------------------------------------------------------------
// explicit D3Q19 transforms in the ABI velocity order (pairs 2p+1, 2p+2 opposite):
// the same linear maps as the basis tables above, with the sums shared between modes and
// between populations written out, which the compiler cannot do itself without reassociating
// floating-point sums.
// ---------------------------------------------------------------------------------------
// moments 0..9 (density, momentum, stress modes) of 19 populations
template <class R>
__host__ __device__ __forceinline__ void moments_0_9(const R n[Q], R m[10]) {
  const R s0 = n[1] + n[2], d0 = n[1] - n[2];
  const R s1 = n[3] + n[4], d1 = n[3] - n[4];
  const R s2 = n[5] + n[6], d2 = n[5] - n[6];
  const R s3 = n[7] + n[8], d3 = n[7] - n[8];
  const R s4 = n[9] + n[10], d4 = n[9] - n[10];
  const R s5 = n[11] + n[12], d5 = n[11] - n[12];
  const R s6 = n[13] + n[14], d6 = n[13] - n[14];
  const R s7 = n[15] + n[16], d7 = n[15] - n[16];
  const R s8 = n[17] + n[18], d8 = n[17] - n[18];
  const R sxy = s3 + s4, sxz = s5 + s6, syz = s7 + s8;
  const R snn = sxy + sxz + syz;
  m[0] = n[0] + (s0 + s1 + s2) + snn;
  m[1] = d0 + d3 + d4 + d5 + d6;
  m[2] = d1 + d3 - d4 + d7 + d8;
  m[3] = d2 + d5 - d6 + d7 - d8;
  m[4] = snn - n[0];
  m[5] = R(2) * (s0 - syz) - s1 - s2 + sxy + sxz;
  m[6] = s1 - s2 + sxy - sxz;
  m[7] = s3 - s4;
  m[8] = s7 - s8;
  m[9] = s5 - s6;
}

// populations n_i = w_i sum_k e_k(c_i) a_k from scaled moments a_k = m_k / b_k
template <class R>
__host__ __device__ __forceinline__ void pops_from_scaled(const R a[Q], R n[Q]) {
  const R w0 = R(1) / R(3), w1 = R(1) / R(18), w2 = R(1) / R(36);
  n[0] = w0 * (a[0] - a[4] + a[16]);
  // nearest neighbours
  const R t = a[0] - a[5] - R(2) * a[16] + a[17];
  const R Sx = a[0] + R(2) * (a[5] - a[16] - a[17]);
  const R Sy = t + (a[6] - a[18]);
  const R Sz = t - (a[6] - a[18]);
  const R Dx = a[1] - R(2) * a[10], Dy = a[2] - R(2) * a[11], Dz = a[3] - R(2) * a[12];
  n[1] = w1 * (Sx + Dx);
  n[2] = w1 * (Sx - Dx);
  n[3] = w1 * (Sy + Dy);
  n[4] = w1 * (Sy - Dy);
  n[5] = w1 * (Sz + Dz);
  n[6] = w1 * (Sz - Dz);
  // next-nearest neighbours
  const R base = a[0] + a[4] + a[16];
  const R P = a[5] + a[17], Qv = a[6] + a[18];
  const R X = base + P + Qv, Y = base + P - Qv, Z = base - R(2) * P;
  const R A = a[1] + a[10], B = a[2] + a[11], Cc = a[3] + a[12];
  const R D3 = (A + B) + (a[13] - a[14]);
  const R D4 = (A - B) + (a[13] + a[14]);
  const R D5 = (A + Cc) - (a[13] - a[15]);
  const R D6 = (A - Cc) - (a[13] + a[15]);
  const R D7 = (B + Cc) + (a[14] - a[15]);
  const R D8 = (B - Cc) + (a[14] + a[15]);
  const R S3 = X + a[7], S4 = X - a[7];
  const R S5 = Y + a[9], S6 = Y - a[9];
  const R S7 = Z + a[8], S8 = Z - a[8];
  n[7] = w2 * (S3 + D3);
  n[8] = w2 * (S3 - D3);
  n[9] = w2 * (S4 + D4);
  n[10] = w2 * (S4 - D4);
  n[11] = w2 * (S5 + D5);
  n[12] = w2 * (S5 - D5);
  n[13] = w2 * (S6 + D6);
  n[14] = w2 * (S6 - D6);
  n[15] = w2 * (S7 + D7);
  n[16] = w2 * (S7 - D7);
  n[17] = w2 * (S8 + D8);
  n[18] = w2 * (S8 - D8);
}

// the same map from w_2-scaled moments a'_k = a_k / 36: n_0 = 12 (...), nearest-neighbour
// populations 2 (S' +- D'), next-nearest S' +- D'
template <class R>
__host__ __device__ __forceinline__ void pops_from_w2scaled(const R a[Q], R n[Q]) {
  n[0] = R(12) * (a[0] - a[4] + a[16]);
  const R t = a[0] - a[5] - R(2) * a[16] + a[17];
  const R Sx = a[0] + R(2) * (a[5] - a[16] - a[17]);
  const R Sy = t + (a[6] - a[18]);
  const R Sz = t - (a[6] - a[18]);
  const R Dx = a[1] - R(2) * a[10], Dy = a[2] - R(2) * a[11], Dz = a[3] - R(2) * a[12];
  n[1] = R(2) * (Sx + Dx);
  n[2] = R(2) * (Sx - Dx);
  n[3] = R(2) * (Sy + Dy);
  n[4] = R(2) * (Sy - Dy);
  n[5] = R(2) * (Sz + Dz);
  n[6] = R(2) * (Sz - Dz);
  const R base = a[0] + a[4] + a[16];
  const R P = a[5] + a[17], Qv = a[6] + a[18];
  const R X = base + P + Qv, Y = base + P - Qv, Z = base - R(2) * P;
  const R A = a[1] + a[10], B = a[2] + a[11], Cc = a[3] + a[12];
  const R D3 = (A + B) + (a[13] - a[14]);
  const R D4 = (A - B) + (a[13] + a[14]);
  const R D5 = (A + Cc) - (a[13] - a[15]);
  const R D6 = (A - Cc) - (a[13] + a[15]);
  const R D7 = (B + Cc) + (a[14] - a[15]);
  const R D8 = (B - Cc) + (a[14] + a[15]);
  const R S3 = X + a[7], S4 = X - a[7];
  const R S5 = Y + a[9], S6 = Y - a[9];
  const R S7 = Z + a[8], S8 = Z - a[8];
  n[7] = S3 + D3;
  n[8] = S3 - D3;
  n[9] = S4 + D4;
  n[10] = S4 - D4;
  n[11] = S5 + D5;
  n[12] = S5 - D5;
  n[13] = S6 + D6;
  n[14] = S6 - D6;
  n[15] = S7 + D7;
  n[16] = S7 - D7;
  n[17] = S8 + D8;
  n[18] = S8 - D8;
}

// ---------------------------------------------------------------------------------------
// LB kernel: pull-stream + collide for every node (Sec. II B, Eq. 3)
// ---------------------------------------------------------------------------------------
// Collide the 19 pulled populations n of one node (Sec. II B, Eq. 3) into its 19
// post-collision populations out (lb_collide_store: written to dst at element offset
// i * pl + node for population i).
template <class R, bool DEV, bool NOISE>
__device__ __forceinline__ void lb_collide(const R* n, R out[Q], const FluidK<R>& P, const RoundKeys& rk,
                                           unsigned long long* nonpos, const uint32_t step, const unsigned node) {
  // moments 0..9 (the kinetic modes relax to zero and are not needed)
  R m[10];
  moments_0_9<R>(n, m);
  const R rho = DEV ? P.rho0 + m[0] : m[0];
  const R jx = m[1], jy = m[2], jz = m[3];
  const R ir = lb_rcp<R>(rho);
  const R xx = jx * jx * ir, yy = jy * jy * ir, zz = jz * jz * ir;
  // post-collision moments, directly as w_2-scaled moments a'_k = m*_k / (36 b_k): relaxation
  // of the stress modes towards equilibrium (Eq. 4), kinetic modes to zero, plus the
  // fluctuating part sqrt(rho) phi_k g_k / (36 b_k)
  R a[Q];
  a[0] = m[0] * R(1.0 / 36.0);
  a[1] = jx * R(InvB<1>::v / 36.0);
  a[2] = jy * R(InvB<2>::v / 36.0);
  a[3] = jz * R(InvB<3>::v / 36.0);
  {
    const R e4 = xx + yy + zz, e5 = R(2) * xx - yy - zz, e6 = yy - zz;
    const R e7 = jx * jy * ir, e8 = jy * jz * ir, e9 = jx * jz * ir;
    a[4] = P.wam[4] * m[4] + P.wae[4] * e4;
    a[5] = P.wam[5] * m[5] + P.wae[5] * e5;
    a[6] = P.wam[6] * m[6] + P.wae[6] * e6;
    a[7] = P.wam[7] * m[7] + P.wae[7] * e7;
    a[8] = P.wam[8] * m[8] + P.wae[8] * e8;
    a[9] = P.wam[9] * m[9] + P.wae[9] * e9;
  }
#pragma unroll
  for (int k = 10; k < Q; ++k) a[k] = R(0);

  if (NOISE) {
    if (!(rho > R(0))) atomicAdd(nonpos, 1ull);
    fluid_noise<R>(step, node, rk, P.ncalls > 1, NoiseScale<R>(rho),
                   [&](int j, R g) { a[4 + j] += P.wag[4 + j] * g; }, P.tab);
  }

  if (P.body_on) {
    R dm[10];
    force_moments(rho, jx, jy, jz, P.body_dJ[0], P.body_dJ[1], P.body_dJ[2], P.gs, P.gb, dm);
    a[1] += dm[1] * R(InvB<1>::v / 36.0);
    a[2] += dm[2] * R(InvB<2>::v / 36.0);
    a[3] += dm[3] * R(InvB<3>::v / 36.0);
    a[4] += dm[4] * R(InvB<4>::v / 36.0);
    a[5] += dm[5] * R(InvB<5>::v / 36.0);
    a[6] += dm[6] * R(InvB<6>::v / 36.0);
    a[7] += dm[7] * R(InvB<7>::v / 36.0);
    a[8] += dm[8] * R(InvB<8>::v / 36.0);
    a[9] += dm[9] * R(InvB<9>::v / 36.0);
  }

  pops_from_w2scaled<R>(a, out);
}

// The two nodes of a thread as the two lanes of packed single-precision arithmetic
// (add.f32x2, mul.f32x2, fma.f32x2: one instruction for both nodes, each lane rounded as the
// scalar operation), so that the moment transforms above serve both nodes at once.
struct f2 {
  float2 v;
  __device__ __forceinline__ f2() {}
  __device__ __forceinline__ explicit f2(float s) : v(make_float2(s, s)) {}
  __device__ __forceinline__ f2(float a, float b) : v(make_float2(a, b)) {}
};
__device__ __forceinline__ f2 mk2(float2 v) {
  f2 r;
  r.v = v;
  return r;
}
__device__ __forceinline__ f2 operator+(f2 a, f2 b) { return mk2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ f2 operator-(f2 a, f2 b) { return mk2(__fadd2_rn(a.v, make_float2(-b.v.x, -b.v.y))); }
__device__ __forceinline__ f2 operator*(f2 a, f2 b) { return mk2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { return mk2(__ffma2_rn(a.v, b.v, c.v)); }

// Box-Muller pairs of the noise words w0 (node) and w1 (node + 1): lane by lane the
// arithmetic of fluid_pair<float>, the special-function operations per lane, the rest packed.
template <bool SECOND>
__device__ __forceinline__ void fluid_pair2(uint32_t w0, uint32_t w1, f2 cl, f2& g, f2& h) {
  const f2 u0 = f2(fluid_radius_1p(w0), fluid_radius_1p(w1)) - f2(0x1.fffff8p-1f);  // (k_r + 1/2) 2^-21
  const f2 t = f2(1.0f) - u0;
  const f2 ser = t * fma2(t, fma2(t, f2(-0.480898347f), f2(-0.721347520f)), f2(-1.44269504f));
  const f2 l2(t.v.x < 1.0e-3f ? ser.v.x : approx_lg2(u0.v.x), t.v.y < 1.0e-3f ? ser.v.y : approx_lg2(u0.v.y));
  const f2 x = cl * l2;
  const f2 r = x * f2(approx_rsqrt(x.v.x), approx_rsqrt(x.v.y));
  const f2 d = f2(fluid_angle_1p(w0), fluid_angle_1p(w1)) - f2(1.5f);  // k_a 2^-11 - 1/2, exact
  const f2 th = fma2(f2(6.28318530717958647692f), d, f2(1.53398078788564123e-3f));
  g = r * f2(approx_cos(th.v.x), approx_cos(th.v.y));
  if (SECOND) h = r * f2(approx_sin(th.v.x), approx_sin(th.v.y));
}
template <int PR, bool SECOND = true, class Emit>
__device__ __forceinline__ void fluid_pair2_emit(uint32_t w0, uint32_t w1, f2 cl, Emit& emit) {
  f2 g, h;
  fluid_pair2<SECOND>(w0, w1, cl, g, h);
  emit(2 * PR, g);
  if (SECOND) emit(2 * PR + 1, h);
}
// fluid_noise for the nodes (node, node + 1) at once: emit(j, (g_j of node, g_j of node + 1))
template <class Emit>
__device__ __forceinline__ void fluid_noise2(uint32_t step, uint32_t node, const RoundKeys& rk, bool kinetic, f2 cl,
                                             Emit emit) {
  U4 a = philox4x32_10_rk(U4{step, node, 0u, 0u}, rk);
  U4 b = philox4x32_10_rk(U4{step, node + 1u, 0u, 0u}, rk);
  fluid_pair2_emit<0>(a.x, b.x, cl, emit);
  fluid_pair2_emit<1>(a.y, b.y, cl, emit);
  fluid_pair2_emit<2>(a.z, b.z, cl, emit);
  if (!kinetic) return;
  fluid_pair2_emit<3>(a.w, b.w, cl, emit);
  a = philox4x32_10_rk(U4{step, node, 1u, 0u}, rk);
  b = philox4x32_10_rk(U4{step, node + 1u, 1u, 0u}, rk);
  fluid_pair2_emit<4>(a.x, b.x, cl, emit);
  fluid_pair2_emit<5>(a.y, b.y, cl, emit);
  fluid_pair2_emit<6>(a.z, b.z, cl, emit);
  fluid_pair2_emit<7, false>(a.w, b.w, cl, emit);
}

// lb_collide for the two nodes of a thread (node, node + 1), lane by lane the same update:
// moments, relaxation and back-transform in packed arithmetic; the noise packed too
// (PACKED_NOISE: both nodes' Philox words turned into Gaussians together, fluid_noise2) or
// node by node.  Measured at L = 128: the packed noise cuts the warp instructions per 32 nodes
// from 541 to 483 and the 16-bit-storage step from 49.5 to 46.1 us, but holds two Philox
// states at once and slows the FP32-storage kernel (53.0 to 54.1 us), which waits on memory
// more than on issue slots; so FP32 storage takes the noise node by node.
template <bool DEV, bool NOISE, bool PACKED_NOISE>
__device__ __forceinline__ void lb_collide_pair(const f2 n[Q], f2 out[Q], const FluidK<float>& P,
                                                const RoundKeys& rk, unsigned long long* nonpos,
                                                const uint32_t step, const unsigned node) {
  f2 m[10];
  moments_0_9<f2>(n, m);
  const f2 rho = DEV ? f2(P.rho0) + m[0] : m[0];
  const f2 jx = m[1], jy = m[2], jz = m[3];
  const f2 ir(lb_rcp<float>(rho.v.x), lb_rcp<float>(rho.v.y));
  const f2 xx = jx * jx * ir, yy = jy * jy * ir, zz = jz * jz * ir;
  f2 a[Q];
  a[0] = m[0] * f2((float)(1.0 / 36.0));
  a[1] = jx * f2((float)(InvB<1>::v / 36.0));
  a[2] = jy * f2((float)(InvB<2>::v / 36.0));
  a[3] = jz * f2((float)(InvB<3>::v / 36.0));
  {
    const f2 e4 = xx + yy + zz, e5 = f2(2.0f) * xx - yy - zz, e6 = yy - zz;
    const f2 e7 = jx * jy * ir, e8 = jy * jz * ir, e9 = jx * jz * ir;
    a[4] = fma2(f2(P.wam[4]), m[4], f2(P.wae[4]) * e4);
    a[5] = fma2(f2(P.wam[5]), m[5], f2(P.wae[5]) * e5);
    a[6] = fma2(f2(P.wam[6]), m[6], f2(P.wae[6]) * e6);
    a[7] = fma2(f2(P.wam[7]), m[7], f2(P.wae[7]) * e7);
    a[8] = fma2(f2(P.wam[8]), m[8], f2(P.wae[8]) * e8);
    a[9] = fma2(f2(P.wam[9]), m[9], f2(P.wae[9]) * e9);
  }
#pragma unroll
  for (int k = 10; k < Q; ++k) a[k] = f2(0.0f);

  if (NOISE) {
    if (!(rho.v.x > 0.0f) || !(rho.v.y > 0.0f))
      atomicAdd(nonpos, (unsigned long long)(!(rho.v.x > 0.0f)) + (unsigned long long)(!(rho.v.y > 0.0f)));
    if constexpr (PACKED_NOISE) {
      // NoiseScale<float> of each lane: -2 ln(2) rho, a non-positive rho as 1e-30
      const f2 cl = f2(-1.38629436112f) * f2(rho.v.x > 0.0f ? rho.v.x : 1.0e-30f, rho.v.y > 0.0f ? rho.v.y : 1.0e-30f);
      fluid_noise2(step, node, rk, P.ncalls > 1, cl,
                   [&](int j, f2 g) { a[4 + j] = fma2(f2(P.wag[4 + j]), g, a[4 + j]); });
    } else {
      fluid_noise<float>(step, node, rk, P.ncalls > 1, NoiseScale<float>(rho.v.x),
                         [&](int j, float g) { a[4 + j].v.x = fmaf(P.wag[4 + j], g, a[4 + j].v.x); }, P.tab);
      fluid_noise<float>(step, node + 1, rk, P.ncalls > 1, NoiseScale<float>(rho.v.y),
                         [&](int j, float g) { a[4 + j].v.y = fmaf(P.wag[4 + j], g, a[4 + j].v.y); }, P.tab);
    }
  }

  if (P.body_on) {
    float d0[10], d1[10];
    force_moments(rho.v.x, jx.v.x, jy.v.x, jz.v.x, P.body_dJ[0], P.body_dJ[1], P.body_dJ[2], P.gs, P.gb, d0);
    force_moments(rho.v.y, jx.v.y, jy.v.y, jz.v.y, P.body_dJ[0], P.body_dJ[1], P.body_dJ[2], P.gs, P.gb, d1);
    a[1] = fma2(f2(d0[1], d1[1]), f2((float)(InvB<1>::v / 36.0)), a[1]);
    a[2] = fma2(f2(d0[2], d1[2]), f2((float)(InvB<2>::v / 36.0)), a[2]);
    a[3] = fma2(f2(d0[3], d1[3]), f2((float)(InvB<3>::v / 36.0)), a[3]);
    a[4] = fma2(f2(d0[4], d1[4]), f2((float)(InvB<4>::v / 36.0)), a[4]);
    a[5] = fma2(f2(d0[5], d1[5]), f2((float)(InvB<5>::v / 36.0)), a[5]);
    a[6] = fma2(f2(d0[6], d1[6]), f2((float)(InvB<6>::v / 36.0)), a[6]);
    a[7] = fma2(f2(d0[7], d1[7]), f2((float)(InvB<7>::v / 36.0)), a[7]);
    a[8] = fma2(f2(d0[8], d1[8]), f2((float)(InvB<8>::v / 36.0)), a[8]);
    a[9] = fma2(f2(d0[9], d1[9]), f2((float)(InvB<9>::v / 36.0)), a[9]);
  }

  pops_from_w2scaled<f2>(a, out);
}

template <class S, class R, bool DEV, bool NOISE, class I>
__device__ __forceinline__ void lb_collide_store(const R* n, S* __restrict__ dst, const FluidK<R>& P, const I pl,
                                                 const RoundKeys& rk, unsigned long long* nonpos,
                                                 const uint32_t step, const unsigned node) {
  R out[Q];
  lb_collide<R, DEV, NOISE>(n, out, P, rk, nonpos, step, node);
#pragma unroll
  for (int i = 0; i < Q; ++i) st<S, R>(dst + ((I)i * pl + (I)node), out[i]);
}

// The 19 populations node (x, y, z) pulls from its neighbours in src (periodic): n_i(r) =
// src_i(r - c_i) (Sec. II B, Eq. 3, streaming).
template <class S, class R, class I>
__device__ __forceinline__ void lb_pull(const S* __restrict__ src, const unsigned L, const I pl, const unsigned x,
                                        const unsigned y, const unsigned z, R n[Q]) {
  const unsigned xm = x ? x - 1 : L - 1, xp = (x + 1 < L) ? x + 1 : 0;
  const unsigned ym = y ? y - 1 : L - 1, yp = (y + 1 < L) ? y + 1 : 0;
  const unsigned zm = z ? z - 1 : L - 1, zp = (z + 1 < L) ? z + 1 : 0;
  const unsigned LL = L * L;
  // row offsets of the source rows: [dy+1][dz+1] for a pull from y - dy, z - dz
  const unsigned ry[3] = {yp * L, y * L, ym * L};
  const unsigned rz[3] = {zp * LL, z * LL, zm * LL};
  const unsigned sxs[3] = {xp, x, xm};
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const unsigned idx = sxs[cx(i) + 1] + ry[cy(i) + 1] + rz[cz(i) + 1];
    n[i] = ld<S, R>(src + ((I)i * pl + (I)idx));
  }
}

// Shared memory of one warp that adds the previous step's corrections: coordinates and 19 values
// of up to 32 marked nodes.
template <class R>
struct WarpStage {
  static constexpr unsigned kNodes = 32;
  static constexpr unsigned kBytes = kNodes * (sizeof(uint2) + Q * sizeof(R));
  uint2* at;  // x | y << 16, z
  R* v;       // v[19 slot + i]
  __device__ __forceinline__ WarpStage(unsigned char* smem, unsigned warp)
      : at(reinterpret_cast<uint2*>(smem + warp * kBytes)), v(reinterpret_cast<R*>(at + kNodes)) {}
};

// Slots of a thread's marked nodes in the pass that begins at slot `base` (2^31 and more: not in it).
template <bool PAIR>
struct MarkedSlots {
  unsigned s0, s1, total, below;
  __device__ __forceinline__ MarkedSlots(unsigned mw, unsigned part, unsigned base) {
    const unsigned b0 = __ballot_sync(part, mw & 1u), b1 = PAIR ? __ballot_sync(part, mw & 2u) : 0u;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(below));
    total = __popc(b0) + __popc(b1);
    s0 = (mw & 1u) ? __popc(b0 & below) - base : ~0u;
    s1 = PAIR && (mw & 2u) ? __popc(b0) + __popc(b1 & below) - base : ~0u;
  }
};

// Stage the corrections at the 19 pull sources of the warp's marked nodes of slots base ... base +
// kNodes - 1 (the first nodes' slots, then, with PAIR, the second ones', in the order of the lanes).
// The coordinates are listed in shared memory and the 19 sources of all of them dealt out to the
// lanes of `part`.
template <class R, bool PAIR>
__device__ __forceinline__ void stage_marked(const R* __restrict__ corr, unsigned long long plane, unsigned L,
                                          unsigned node, unsigned mw, unsigned part, unsigned base,
                                          unsigned char* smem) {
  static_assert(sizeof(R) == 4 || sizeof(R) == 8, "cp.async copies 4 or 8 bytes");
  constexpr unsigned long long PX = pack_component(0), PY = pack_component(1), PZ = pack_component(2);
  constexpr unsigned kNodes = WarpStage<R>::kNodes;
  const WarpStage<R> W(smem, (threadIdx.x + blockDim.x * threadIdx.y) / 32);
  const MarkedSlots<PAIR> m(mw, part, base);
  const unsigned row = node / L, x = node - row * L, z = row / L, y = row - z * L;
  if (m.s0 < kNodes) W.at[m.s0] = make_uint2(x | y << 16, z);
  if (PAIR && m.s1 < kNodes) W.at[m.s1] = make_uint2((x + 1) | y << 16, z);
  __syncwarp(part);
  const unsigned items = Q * (m.total - base < kNodes ? m.total - base : kNodes);
#pragma unroll 1
  for (unsigned k = __popc(part & m.below); k < items; k += __popc(part)) {
    const unsigned slot = k / Q, i = k - slot * Q;
    const uint2 c = W.at[slot];
    int sx = (int)(c.x & 0xFFFFu) - unpack_component(PX, i), sy = (int)(c.x >> 16) - unpack_component(PY, i),
        sz = (int)c.y - unpack_component(PZ, i);
    sx = sx < 0 ? sx + (int)L : (sx >= (int)L ? sx - (int)L : sx);
    sy = sy < 0 ? sy + (int)L : (sy >= (int)L ? sy - (int)L : sy);
    sz = sz < 0 ? sz + (int)L : (sz >= (int)L ? sz - (int)L : sz);
    const R* from = corr + ((unsigned long long)i * plane + ((unsigned)sx + L * ((unsigned)sy + L * (unsigned)sz)));
    const unsigned to = (unsigned)__cvta_generic_to_shared(W.v + k);
    if (sizeof(R) == 4)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(to), "l"(from) : "memory");
    else
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(to), "l"(from) : "memory");
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncwarp(part);
}

// The same as a call, for the FP32 kernels: they hold 19 or 38 populations across it in as many
// registers as they have, and what has to make room is then saved around the call, on this rare
// path.  (Inlined, the spills were on every warp's path: 53.0 against 50.2 us per step at L = 128.
// Kernels that had spilled before gained by the call: 43.9 to 42.5 us in BF16 at L = 128, 131.7 to
// 127.2 us for 64 replicas of L = 16 ... 64.  The FP64 kernels have the registers: 18.9 us with the
// call against 18.2 at L = 24.)
template <bool PAIR>
__device__ __noinline__ void stage_marked_call(const float* __restrict__ corr, unsigned long long plane, unsigned L,
                                               unsigned node, unsigned mw, unsigned part, unsigned base,
                                               unsigned char* smem) {
  stage_marked<float, PAIR>(corr, plane, L, node, mw, part, base, smem);
}

// Add the previous step's corrections at the pull sources of the warp's marked nodes to what they
// pulled: bit 0 of mw marks the thread's node, with PAIR bit 1 its second one, `node` + 1.  Called by
// all lanes of `part`.  A warp with m marked nodes runs 19 m / 32 rounds of index arithmetic
// (stage_marked) and waits for one flight of asynchronous copies (cp.async).  A bead marks about 4
// nodes of a row, and a kernel whose blocks are all resident ends with its slowest warp: with
// every marked thread staging its own nodes one after the other, 19 rounds and one flight each,
// the step at L = 64, N = 64 (FP32) took 11.4 us, of which 3.2 went with the corrections left out;
// then 8.6 (7.4 without a chain); 7.8 with blocks of 128 threads (7.15).  INLINE: not as a call in
// single precision either (persistent blocks, in whose loop over tiles the call made the main path
// spill: 64 replicas of L = 32 on one block of 128 threads per SM 185 us per step, inlined 175).
template <class R, bool PAIR, bool INLINE = false>
__device__ __forceinline__ void add_corrections(const R* __restrict__ corr, unsigned long long plane, unsigned L,
                                                unsigned node, unsigned mw, unsigned part, unsigned char* smem,
                                                R* n0, R* n1) {
  if (!__any_sync(part, mw & (PAIR ? 3u : 1u))) return;
  constexpr unsigned kNodes = WarpStage<R>::kNodes;
#pragma unroll 1
  for (unsigned base = 0;; base += kNodes) {
    if constexpr (sizeof(R) == 4 && !INLINE)
      stage_marked_call<PAIR>(corr, plane, L, node, mw, part, base, smem);
    else
      stage_marked<R, PAIR>(corr, plane, L, node, mw, part, base, smem);
    const WarpStage<R> W(smem, (threadIdx.x + blockDim.x * threadIdx.y) / 32);
    const MarkedSlots<PAIR> m(mw, part, base);
    if (m.s0 < kNodes) {
#pragma unroll
      for (int i = 0; i < Q; ++i) n0[i] += W.v[Q * m.s0 + i];
    }
    if (PAIR && m.s1 < kNodes) {
#pragma unroll
      for (int i = 0; i < Q; ++i) n1[i] += W.v[Q * m.s1 + i];
    }
    __syncwarp(part);  // all have read before the next pass or tile writes
    if (!PAIR || m.total <= base + kNodes) break;
  }
}

// One node: pull-stream + collide (Sec. II B, Eq. 3).  Every thread loads its 19 populations and
// its mark word together; a node marked by the previous deferred step then adds that step's
// corrections at its pull sources to what it pulled (add_corrections: `part` are the warp's lanes
// that have a node), and one copy of the collision follows.  (Branching on the mark
// before the loads put an L2 round trip in front of every warp's loads, 1.4 us per launch at
// L = 128 with no node marked; with two inlined copies of the update, a warp holding marked and
// unmarked nodes ran both: 67.8 against 64.0 us with 1.5 % of the nodes marked.)
// CORR = false (a box without a chain): no correction code at all (the dead correction path
// alone cost 0.5 us per chained launch at L = 128).
template <class S, class R, bool DEV, bool NOISE, class I, bool CORR>
__device__ __forceinline__ void lb_node(const S* __restrict__ src, S* __restrict__ dst, const FluidK<R>& P,
                                        const PendK<R>& Pd, const uint32_t step, unsigned x, unsigned y, unsigned z,
                                        unsigned char* smem, unsigned part) {
  const unsigned L = P.L;
  const unsigned node = x + L * (y + L * z);
  const unsigned mw = CORR && Pd.have_prev ? Pd.prev_mask[Pd.seg0 + (node >> kSegShift)] >> (node & 31u) : 0u;
  const I pl = (I)P.plane;
  R n[Q];
  lb_pull<S, R, I>(src, L, pl, x, y, z, n);
  if (CORR) add_corrections<R, false>(Pd.prev_dense, Pd.plane, L, node, mw, part, smem, n, n);
  lb_collide_store<S, R, DEV, NOISE, I>(n, dst, P, pl, P.rk, P.nonpos, step, node);
}

// Collide the pulled populations n0, n1 of the nodes (node, node + 1) and store the pairs
// (single precision: packed arithmetic for both nodes, lb_collide_pair; the noise packed
// too for 16-bit storage).
template <class S, class R, bool DEV, bool NOISE, class I>
__device__ __forceinline__ void lb_collide2_store(const R n0[Q], const R n1[Q], S* __restrict__ dst,
                                                  const FluidK<R>& P, const I pl, const RoundKeys& rk,
                                                  unsigned long long* nonpos, const uint32_t step,
                                                  const unsigned node) {
  if constexpr (sizeof(R) == 4) {
    f2 n[Q], o[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) n[i] = f2(n0[i], n1[i]);
    lb_collide_pair<DEV, NOISE, sizeof(S) == 2>(n, o, P, rk, nonpos, step, node);
#pragma unroll
    for (int i = 0; i < Q; ++i) st2<S, R>(dst + ((I)i * pl + (I)node), o[i].v.x, o[i].v.y);
  } else {
    R o0[Q], o1[Q];
    lb_collide<R, DEV, NOISE>(n0, o0, P, rk, nonpos, step, node);
    lb_collide<R, DEV, NOISE>(n1, o1, P, rk, nonpos, step, node + 1);
#pragma unroll
    for (int i = 0; i < Q; ++i) st2<S, R>(dst + ((I)i * pl + (I)node), o0[i], o1[i]);
  }
}

// The populations the two nodes (x0, y, z) and (x0 + 1, y, z), x0 even, pull from their
// neighbours (periodic; Sec. II B, Eq. 3): n0 for x0, n1 for x0 + 1.  The planes with c_x = 0
// read both nodes' sources with one two-element access (x0 even and L even keep it aligned);
// the planes with c_x = +-1 read their two sources x0 - c_x, x0 + 1 - c_x one by one.
template <class S, class R, class I>
__device__ __forceinline__ void lb_pull2(const S* __restrict__ src, const unsigned L, const I pl, const unsigned x0,
                                         const unsigned y, const unsigned z, R n0[Q], R n1[Q]) {
  const unsigned xm = x0 ? x0 - 1 : L - 1, xp = x0 + 1, xpp = (x0 + 2 < L) ? x0 + 2 : 0;
  const unsigned ym = y ? y - 1 : L - 1, yp = (y + 1 < L) ? y + 1 : 0;
  const unsigned zm = z ? z - 1 : L - 1, zp = (z + 1 < L) ? z + 1 : 0;
  const unsigned LL = L * L;
  const unsigned ry[3] = {yp * L, y * L, ym * L};
  const unsigned rz[3] = {zp * LL, z * LL, zm * LL};
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const I row = (I)i * pl + (I)(ry[cy(i) + 1] + rz[cz(i) + 1]);
    if (cx(i) == 0) {
      ld2<S, R>(src + (row + (I)x0), n0[i], n1[i]);
    } else if (cx(i) == 1) {  // sources x0 - 1, x0
      n0[i] = ld<S, R>(src + (row + (I)xm));
      n1[i] = ld<S, R>(src + (row + (I)x0));
    } else {  // sources x0 + 1, x0 + 2
      n0[i] = ld<S, R>(src + (row + (I)xp));
      n1[i] = ld<S, R>(src + (row + (I)xpp));
    }
  }
}

// Two nodes (x0, y, z) and (x0 + 1, y, z), x0 even, L even: the same update as lb_node, node by
// node, with the 19 post-collision pairs written by two-element stores.
template <class S, class R, bool DEV, bool NOISE, class I, bool CORR>
__device__ __forceinline__ void lb_nodes2(const S* __restrict__ src, S* __restrict__ dst, const FluidK<R>& P,
                                          const PendK<R>& Pd, const uint32_t step, unsigned x0, unsigned y,
                                          unsigned z, unsigned char* smem, unsigned part) {
  const unsigned L = P.L;
  const unsigned node = x0 + L * (y + L * z);
  const unsigned mw = CORR && Pd.have_prev ? Pd.prev_mask[Pd.seg0 + (node >> kSegShift)] >> (node & 31u) : 0u;
  const I pl = (I)P.plane;
  R n0[Q], n1[Q];
  lb_pull2<S, R, I>(src, L, pl, x0, y, z, n0, n1);
  if (CORR) add_corrections<R, true>(Pd.prev_dense, Pd.plane, L, node, mw, part, smem, n0, n1);
  lb_collide2_store<S, R, DEV, NOISE, I>(n0, n1, dst, P, pl, P.rk, P.nonpos, step, node);
}

// Programmatic dependent launch (a grid launched with programmatic stream serialization may
// start before the previous grid in the stream has completed): `wait` blocks until that
// previous grid has completed and its writes are visible; `release` lets the next grid start.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void allow_dependent_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// LB kernel: 3D grid of (x-row segments) x (groups of y rows) x z planes (a block's threads take
// P.rows row segments of P.row threads, one after the other: lb_row_shape), plus (when it follows the
// bead kernel of its step) one more plane of blocks that only wait.  Every grid releases the
// next one at once.  Launched after the previous LB kernel (no chain): it waits for that grid
// before reading (P.pdl bit 0), so that only the launch latency and block scheduling overlap.
// Launched after the bead kernel of the same step: it reads nothing that kernel writes and
// runs beside it; the blocks of plane z = L, scheduled last, wait for it (bit 1), so that the
// grid completes only after the bead kernel and whatever comes next may take this grid's
// completion for both.  (A wait at the end of every block raised the register count.)
// Resident blocks of 256 threads per SM that the single-precision LB kernels are compiled
// for: 6 (40 registers) with one node per thread, 4 (64 registers) with two, so that 48 and 32
// warps keep 48 and 64 node updates' loads in flight per SM quarter; the FP64 kernel is
// bound by FP64 arithmetic and compiled without a bound.
template <class R, bool PAIR>
struct LbMinBlocks {
  static constexpr int value = sizeof(R) == 4 ? (PAIR ? 4 : 6) : 1;
};

// n / d for n < 2^24 and 2 <= d <= 256 by one multiply-high with m = ceil(2^32 / d): with
// e = m d - 2^32 < d, n m / 2^32 = n / d + n e / (d 2^32) and n e < 2^32 keeps the error below
// the distance of n / d to the next integer (checked exhaustively for every d and n in range).
__host__ __device__ __forceinline__ unsigned magic_of(unsigned d) {
  return (unsigned)((0x100000000ull + d - 1) / d);
}
__device__ __forceinline__ unsigned div_magic(unsigned n, unsigned m) { return __umulhi(n, m); }

// PAIR: two nodes per thread along x (lb_nodes2, L even), else one (lb_node).
template <class S, class R, bool DEV, bool NOISE, class I, bool CORR, bool PAIR>
__global__ void __launch_bounds__(256, LbMinBlocks<R, PAIR>::value) k_lb_step(const S* __restrict__ src, S* __restrict__ dst,
                                                  const FluidK<R> P, const PendK<R> Pd, const uint32_t step) {
  extern __shared__ __align__(16) unsigned char lsm[];
  if (blockIdx.z >= P.L) {  // a waiting block
    allow_dependent_launch();
    if (P.pdl & 2) grid_dependency_wait();
    return;
  }
  if (P.pdl & 1) grid_dependency_wait();
  allow_dependent_launch();
  const uint32_t k = launch_step(P, step);
  const unsigned ty = div_magic(threadIdx.x, P.mag_row);
  const unsigned xt = blockIdx.x * P.row + (threadIdx.x - ty * P.row), y = blockIdx.y * P.rows + ty;
  const bool in = ty < P.rows && (PAIR ? 2 * xt : xt) < P.L && y < P.L;
  const unsigned part = CORR ? __ballot_sync(~0u, in) : 0u;
  if (!in) return;
  if constexpr (PAIR)
    lb_nodes2<S, R, DEV, NOISE, I, CORR>(src, dst, P, Pd, k, 2 * xt, y, blockIdx.z, lsm, part);
  else
    lb_node<S, R, DEV, NOISE, I, CORR>(src, dst, P, Pd, k, xt, y, blockIdx.z, lsm, part);
}

// The same launch over consecutive nodes (4 <= L <= 256), one block of threads after the other, with
// one more block that waits, for the FP64 kernel.  That kernel is bound by the FP64 pipe (2
// multiply-adds per clock and SM), which an instruction holds for 16 clocks whatever its lanes do:
// no lane may idle, and a small box must reach every SM.  With the noise's radii and angles read
// from tables, L = 72: 163 us per step (580 with a logarithm and a square root per pair; 2.3
// GLUPS); L = 16, alone under ncu: 46 us (32 blocks of 256 threads with half the lanes idle) to
// the bead kernel's shadow.
template <class S, class R, bool DEV, bool NOISE, bool CORR>
__global__ void __launch_bounds__(256) k_lb_linear(const S* __restrict__ src, S* __restrict__ dst, const FluidK<R> P,
                                                   const PendK<R> Pd, const uint32_t step, const unsigned nnodes,
                                                   const unsigned mag_L) {
  extern __shared__ __align__(16) unsigned char lsm[];
  const unsigned node = blockIdx.x * blockDim.x + threadIdx.x;
  if (P.pdl & 1) grid_dependency_wait();
  allow_dependent_launch();
  if ((P.pdl & 2) && blockIdx.x == gridDim.x - 1) {  // the waiting block
    grid_dependency_wait();
    return;
  }
  const unsigned part = CORR ? __ballot_sync(~0u, node < nnodes) : 0u;
  if (node >= nnodes) return;
  const uint32_t k = launch_step(P, step);
  const unsigned row = div_magic(node, mag_L), x = node - row * P.L;
  const unsigned z = div_magic(row, mag_L), y = row - z * P.L;
  lb_node<S, R, DEV, NOISE, unsigned, CORR>(src, dst, P, Pd, k, x, y, z, lsm, part);
}

// ---------------------------------------------------------------------------------------
// bead / coupling kernel (one thread block or one cluster)
// ---------------------------------------------------------------------------------------
// cell of a coordinate: floor(x/a) mod L into [0, L); frac = x/a - floor(x/a)
template <class R>
__device__ __forceinline__ int cell_of(R x, R a, int L, R& frac) {
  const R s = x / a;
  const R f = floor(s);
  frac = s - f;
  long long c = (long long)f;
  long long r = c % L;
  if (r < 0) r += L;
  return (int)r;
}

// Pair vector r_b - r_j under the minimum image convention from compensated positions
// (hi in [0, box), lo): the coordinate above box/2 is moved down by the box, which is exact
// (Sterbenz), so the difference of two nearby beads carries no rounding from their distance to
// the origin.
template <class R>
__device__ __forceinline__ R pair_delta(R hb, R lb, R hj, R lj, R box, R half_box) {
  const R dh = hb - hj;
  if (dh > half_box)
    hb -= box;
  else if (dh < -half_box)
    hj -= box;
  return (hb - hj) + (lb - lj);
}

// FENE (bonded) + WCA force coefficient: force on b = coef * d
template <class R>
__device__ __forceinline__ R pair_coef(R r2, bool bonded, const ChainK<R>& C, unsigned* status) {
  R coef = R(0);
  if (r2 < C.rc2) {
    const R s2 = C.sig2 / r2;
    const R s6 = s2 * s2 * s2;
    coef += R(24) * C.eps / r2 * (R(2) * s6 * s6 - s6);
  }
  if (bonded) {
    if (r2 >= C.R0sq) {
      atomicOr(status, ST_FENE);
    } else {
      coef -= C.kfene / (R(1) - r2 / C.R0sq);
    }
  }
  return coef;
}

// Conservative force (FENE + WCA) on bead b from the positions of all beads staged in shared
// memory; `lanes` neighbouring threads (lane: this one's) split the partners and combine in a
// fixed shuffle tree.  Whole warps call it together (beads past the end: b = N).
template <class R>
__device__ __forceinline__ void bead_force(const R* __restrict__ sh, const R* __restrict__ sl, const ChainK<R>& C,
                                           const int b, const int lane, const int lanes, R f[3]) {
  const int N = C.N;
  f[0] = f[1] = f[2] = R(0);
  if (b < N) {
    for (int j = lane; j < N; j += lanes) {
      if (j == b) continue;
      const bool bonded = (j == b - 1) || (j == b + 1);
      R d[3];
#pragma unroll
      for (int q = 0; q < 3; ++q)
        d[q] = pair_delta<R>(sh[3 * b + q], sl[3 * b + q], sh[3 * j + q], sl[3 * j + q], C.box, C.half_box);
      const R r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
      const R coef = pair_coef<R>(r2, bonded, C, C.status);
      f[0] += coef * d[0];
      f[1] += coef * d[1];
      f[2] += coef * d[2];
    }
  }
  for (int o = lanes / 2; o > 0; o /= 2) {
#pragma unroll
    for (int q = 0; q < 3; ++q) f[q] += __shfl_xor_sync(0xffffffffu, f[q], o, lanes);
  }
}

// Conservative forces (FENE + WCA + external) on every bead by a block; as many threads per bead
// as fit
template <class R>
__device__ __forceinline__ void chain_forces_block(const R* __restrict__ sh, const R* __restrict__ sl,
                                                   const ChainK<R>& C, R* __restrict__ out) {
  const int N = C.N, nt = blockDim.x * blockDim.y, tid = threadIdx.x + blockDim.x * threadIdx.y;
  int lanes = 1;
  while (lanes < 32 && lanes * 2 * N <= nt) lanes *= 2;
  const int lane = tid % lanes;
  for (int base = 0; base < N; base += nt / lanes) {
    const int b = base + tid / lanes;
    R f[3];
    bead_force<R>(sh, sl, C, b, lane, lanes, f);
    if (b < N && lane == 0) {
#pragma unroll
      for (int q = 0; q < 3; ++q) out[3 * b + q] = f[q] + C.ext[q];
    }
  }
}

// Bitonic sort (ascending) of M keys in shared memory, M a power of two >= 32, by a block of
// nt threads (a multiple of 32).  Compare-exchange distances j >= 32 go through shared memory
// with a barrier each; the distances j < 32 of every stage run in registers, each warp
// holding a contiguous chunk of 32 keys and exchanging through shuffles.
__device__ __forceinline__ void bitonic_sort_block(unsigned long long* keys, int M, int tid, int nt) {
  for (int k = 2; k <= M; k <<= 1) {
    for (int j = k >> 1; j >= 32; j >>= 1) {
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
    for (int i = tid; i < M; i += nt) {  // whole warps: M and nt are multiples of 32
      unsigned long long v = keys[i];
      const bool up = (i & k) == 0;
      for (int j = (k >> 1) < 16 ? (k >> 1) : 16; j > 0; j >>= 1) {
        const unsigned lo = __shfl_xor_sync(0xffffffffu, (unsigned)v, j);
        const unsigned hi = __shfl_xor_sync(0xffffffffu, (unsigned)(v >> 32), j);
        const unsigned long long o = ((unsigned long long)hi << 32) | lo;
        // the lower element of the pair keeps the minimum in an ascending run
        const bool take_min = ((i & j) == 0) == up;
        v = take_min ? (o < v ? o : v) : (o > v ? o : v);
      }
      keys[i] = v;
    }
    __syncthreads();
  }
}

// post-stream populations at node (qx,qy,qz): rho and lattice momentum; with the dense field
// of the previous step's corrections (corr != nullptr) added to the pulled populations
template <class S, class R, bool DEV>
__device__ __forceinline__ void gather_node_c(const S* __restrict__ pop, const FluidK<R>& P, int qx, int qy,
                                              int qz, R mom[4], const R* __restrict__ corr) {
  const int L = (int)P.L;
  unsigned idx[Q];
  R v[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    int sx = qx - cx(i), sy = qy - cy(i), sz = qz - cz(i);
    sx = sx < 0 ? sx + L : (sx >= L ? sx - L : sx);
    sy = sy < 0 ? sy + L : (sy >= L ? sy - L : sy);
    sz = sz < 0 ? sz + L : (sz >= L ? sz - L : sz);
    idx[i] = (unsigned)sx + (unsigned)L * ((unsigned)sy + (unsigned)L * (unsigned)sz);
    v[i] = ld<S, R>(pop + (unsigned long long)i * P.plane + idx[i]);
  }
  if (corr) {
#pragma unroll
    for (int i = 0; i < Q; ++i) v[i] += corr[(unsigned long long)i * P.plane + idx[i]];
  }
  R rho = R(0), jx = R(0), jy = R(0), jz = R(0);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    rho += v[i];
    if (cx(i)) jx += R(cx(i)) * v[i];
    if (cy(i)) jy += R(cy(i)) * v[i];
    if (cz(i)) jz += R(cz(i)) * v[i];
  }
  mom[0] = DEV ? P.rho0 + rho : rho;
  mom[1] = jx;
  mom[2] = jy;
  mom[3] = jz;
}

// post-stream populations at node (qx,qy,qz): rho and lattice momentum
template <class S, class R, bool DEV>
__device__ __forceinline__ void gather_node(const S* __restrict__ pop, const FluidK<R>& P, int qx, int qy,
                                            int qz, R mom[4]) {
  const int L = (int)P.L;
  R rho = R(0), jx = R(0), jy = R(0), jz = R(0);
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    int sx = qx - cx(i), sy = qy - cy(i), sz = qz - cz(i);
    sx = sx < 0 ? sx + L : (sx >= L ? sx - L : sx);
    sy = sy < 0 ? sy + L : (sy >= L ? sy - L : sy);
    sz = sz < 0 ? sz + L : (sz >= L ? sz - L : sz);
    const unsigned idx = (unsigned)sx + (unsigned)L * ((unsigned)sy + (unsigned)L * (unsigned)sz);
    const R v = ld<S, R>(pop + (unsigned long long)i * P.plane + idx);
    rho += v;
    if (cx(i)) jx += R(cx(i)) * v;
    if (cy(i)) jy += R(cy(i)) * v;
    if (cz(i)) jz += R(cz(i)) * v;
  }
  mom[0] = DEV ? P.rho0 + rho : rho;
  mom[1] = jx;
  mom[2] = jy;
  mom[3] = jz;
}

// Mark the nodes of one row (dy, dz) that pull from node (px, py, pz), periodic: the three x
// neighbours, or only px on a diagonal row; one atomic per word (the three bits lie in one word
// unless they straddle two or wrap).
__device__ __forceinline__ void mark_row(unsigned* mask, unsigned seg0, int L, int px, int py, int pz, int dy, int dz) {
  int y = py + dy, z = pz + dz;
  y = y < 0 ? L - 1 : (y >= L ? 0 : y);
  z = z < 0 ? L - 1 : (z >= L ? 0 : z);
  const int row = L * (y + L * z);
  const unsigned c = (unsigned)(row + px);
  unsigned bits = 1u << (c & 31u);
  if (dy == 0 || dz == 0) {
    const unsigned l = (unsigned)(row + (px ? px - 1 : L - 1)), r = (unsigned)(row + (px + 1 < L ? px + 1 : 0));
    if ((l >> kSegShift) == (c >> kSegShift)) bits |= 1u << (l & 31u);
    else atomicOr(mask + (seg0 + (l >> kSegShift)), 1u << (l & 31u));
    if ((r >> kSegShift) == (c >> kSegShift)) bits |= 1u << (r & 31u);
    else atomicOr(mask + (seg0 + (r >> kSegShift)), 1u << (r & 31u));
  }
  atomicOr(mask + (seg0 + (c >> kSegShift)), bits);
}

// Clear the mask words of the nodes that pull from node (px, py, pz) (whole words: in its slot
// a word holds marks of one list only)
__device__ __forceinline__ void clear_marks(unsigned* mask, unsigned seg0, int L, int px, int py, int pz) {
  const int xm = px ? px - 1 : L - 1, xp = px + 1 < L ? px + 1 : 0;
  const int ys[3] = {py ? py - 1 : L - 1, py, py + 1 < L ? py + 1 : 0};
  const int zs[3] = {pz ? pz - 1 : L - 1, pz, pz + 1 < L ? pz + 1 : 0};
#pragma unroll
  for (int j = 0; j < 9; ++j) {
    const int row = L * (ys[j % 3] + L * zs[j / 3]);
    const unsigned c = (unsigned)(row + px) >> kSegShift;
    mask[seg0 + c] = 0u;
    if (j % 3 == 1 || j / 3 == 1) {
      const unsigned l = (unsigned)(row + xm) >> kSegShift, r = (unsigned)(row + xp) >> kSegShift;
      if (l != c) mask[seg0 + l] = 0u;
      if (r != c) mask[seg0 + r] = 0u;
    }
  }
}

// Moment increments 1..9 of the force density f on a node of the given post-stream density and
// momentum (the coupling of Sec. II B, spread back to the fluid)
template <class R>
__device__ __forceinline__ void coupling_moments(const FluidK<R>& P, const ChainK<R>& C, const R f[3], R rho, R jx,
                                                 R jy, R jz, R dm[10]) {
  R dJ[3] = {f[0] * C.dJ_scale, f[1] * C.dJ_scale, f[2] * C.dJ_scale};
  if (P.body_on) {
    // the LB kernel applies the body-force correction on every node; here add the
    // difference between the correction for the total force and the body-only one
    R dmb[10];
    force_moments(rho, jx, jy, jz, P.body_dJ[0], P.body_dJ[1], P.body_dJ[2], P.gs, P.gb, dmb);
    force_moments(rho, jx, jy, jz, dJ[0] + P.body_dJ[0], dJ[1] + P.body_dJ[1], dJ[2] + P.body_dJ[2],
                  P.gs, P.gb, dm);
#pragma unroll
    for (int k = 0; k < 10; ++k) dm[k] -= dmb[k];
  } else {
    force_moments(rho, jx, jy, jz, dJ[0], dJ[1], dJ[2], P.gs, P.gb, dm);
  }
}

// The pending correction of one node by one thread: population corrections written to the dense
// field, the node listed at index u, and the nodes pulling from it marked.
template <class R>
__device__ __forceinline__ void node_correction(const FluidK<R>& P, const ChainK<R>& C, const PendK<R>& Pd, int L,
                                                int u, int node, const R f[3], R rho, R jx, R jy, R jz) {
  R dm[10], a[Q], dn[Q];
  coupling_moments<R>(P, C, f, rho, jx, jy, jz, dm);
  scaled_increments<R>([&](int k) { return dm[k]; }, a);
  modes_to_pops(a, dn);
  const int pz = node / (L * L), py = (node / L) % L, px = node % L;
  Pd.cur_pos[u] = make_int4(node, px, py, pz);
#pragma unroll
  for (int q = 0; q < Q; ++q) Pd.cur_dense[(unsigned long long)q * Pd.plane + (unsigned)node] = dn[q];
  if (Pd.mark) {
    // (unrolled: as a loop the marks of 1000 nodes took 108 us by a block in FP64, where they take a few;
    // 880 -> 730 us per step for 16 replicas of L = 24, N = 200; FP32 L = 32, N = 16 6.7 -> 6.3)
#pragma unroll
    for (int j = 0; j < 9; ++j) mark_row(Pd.cur_mask, Pd.seg0, L, px, py, pz, j % 3 - 1, j / 3 - 1);
  }
}

// Empty the list entry u (of this slot's list from two steps before, or already applied): its
// node's corrections (added to apply_to where given) and the marks of the nodes pulling from it back
// to zero
template <class R>
__device__ __forceinline__ void clear_correction(const PendK<R>& Pd, int L, int u) {
  const int4 p = Pd.cur_pos[u];
  if (p.x < 0) return;
  R* d = Pd.cur_dense + (unsigned)p.x;
  if (Pd.apply_to) {
    R* n = Pd.apply_to + (unsigned)p.x;
    R c[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) c[i] = n[(unsigned long long)i * Pd.plane] + d[(unsigned long long)i * Pd.plane];
#pragma unroll
    for (int i = 0; i < Q; ++i) n[(unsigned long long)i * Pd.plane] = c[i];
  }
#pragma unroll
  for (int i = 0; i < Q; ++i) d[(unsigned long long)i * Pd.plane] = R(0);
  if (Pd.cur_mask) clear_marks(Pd.cur_mask, Pd.seg0, L, p.y, p.z, p.w);
}

// v into the same shared-memory location of block `rank` of the cluster
template <class T>
__device__ __forceinline__ void cluster_store(T* p, int rank, T v) {
  static_assert(sizeof(T) == 4 || sizeof(T) == 8, "4- or 8-byte values");
  unsigned d;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  if constexpr (sizeof(T) == 4)
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(d), "r"(__float_as_uint(v)) : "memory");
  else
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(d), "l"(__double_as_longlong(v)) : "memory");
}

// The two halves of a barrier over the thread blocks of a cluster; release and acquire order every memory
// access before it (shared, distributed shared and global) before every access after it.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
// an arrival that orders no memory access (a release waits for the thread's writes in flight)
__device__ __forceinline__ void cluster_arrive_relaxed() {
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// f / (2 m) and x / a, by the exact reciprocal where there is one
template <class R>
__device__ __forceinline__ R over_2m(R f, const ChainK<R>& C) {
  return C.inv_2m != R(0) ? f * C.inv_2m : f / (R(2) * C.m);
}
template <class R>
__device__ __forceinline__ R over_a(R x, const ChainK<R>& C) {
  return C.inv_a != R(0) ? x * C.inv_a : x / C.a;
}

// First half kick and drift of one coordinate: v_half = v + h F/2m, x' = x + h v_half, in
// compensated (hi, lo) arithmetic, then wrapped into [0, box) with the image counter
template <class R>
__device__ __forceinline__ void drift(const ChainK<R>& C, R v, R F, R xh, R xl, int& im, R& vh, R& hi, R& lo) {
  vh = v + over_2m(C.h * F, C);
  const R dx = C.h * vh;
  hi = xh + dx;
  const R bp = hi - xh;
  lo = xl + ((xh - (hi - bp)) + (dx - bp));
  {
    const R s2 = hi + lo;
    lo = lo - (s2 - hi);
    hi = s2;
  }
  if (hi < R(0)) {
    const R s2 = C.box + hi;
    lo += hi - (s2 - C.box);
    hi = s2;
    --im;
  }
  if (hi >= C.box) {
    hi -= C.box;
    ++im;
  }
}

// Entries (corners of beads over all substeps) up to which the bead step compares beads with one
// another (bead_step_block); beyond, it sorts the entries (bead_step_sorted).
constexpr int kGroupMax = 1024;

// Shared memory of bead_step_block for N beads and nsub substeps of which a block has at most nb
// beads.  A bead and substep is counted as "place" sub N + b, its corner c as entry 8 place + c.
template <class R>
struct BeadSmem {
  R *x, *l, *vh;      // 3N each: drifted positions (high, low) and half-step velocities
  R *fr;              // 3N: position inside the cell
  R *v, *F;           // 2 x 3N each (nsub > 1): end of a substep, by its parity
  R *fc;              // 3N nsub: coupling forces
  R *w;               // 8 N nsub: trilinear weights of every entry
  R *mom;             // 5 x own: density, momentum and 1/density at the block's corner nodes
  R *fcons;           // 3 nb: conservative forces
  R *g;               // 3 nb nsub: noise
  int *node;          // own: the block's corner nodes
  int *img;           // 3N
  int *cell;          // 3N nsub
  int *near;          // nb nsub x N nsub: of each of the block's places the ones whose cells touch its
                      // cell: place | corners shared << 8 | (shift of the corner number + 8) << 16
  int *nnear;         // nb nsub: their number
  // lays the arrays out from base on; returns their size
  __host__ __device__ __forceinline__ int carve(unsigned char* base, int N, int nsub, int nb) {
    int off = 0;
    auto take = [&](int bytes) {  // (no test of base: the compiler must see that these are shared)
      unsigned char* p = base + off;
      off += (bytes + 15) / 16 * 16;
      return p;
    };
    const int r = (int)sizeof(R), n3 = 3 * N, own = 8 * nb * nsub;
    x = (R*)take(n3 * r);
    l = (R*)take(n3 * r);
    vh = (R*)take(n3 * r);
    fr = (R*)take(n3 * r);
    v = (R*)take(nsub > 1 ? 2 * n3 * r : 0);
    F = (R*)take(nsub > 1 ? 2 * n3 * r : 0);
    fc = (R*)take(n3 * nsub * r);
    w = (R*)take(8 * N * nsub * r);
    mom = (R*)take(5 * own * r);
    fcons = (R*)take(3 * nb * r);
    g = (R*)take(3 * nb * nsub * r);
    node = (int*)take(own * 4);
    img = (int*)take(n3 * 4);
    cell = (int*)take(n3 * nsub * 4);
    near = (int*)take(nb * nsub * N * nsub * 4);
    nnear = (int*)take(nb * nsub * 4);
    return off;
  }
};

// trilinear weight of corner c (bit q: the far side along q) at position fr inside the cell
template <class R>
__device__ __forceinline__ R corner_weight(const R* fr, int c) {
  const R x = c & 1 ? fr[0] : R(1) - fr[0], y = c & 2 ? fr[1] : R(1) - fr[1], z = c & 4 ? fr[2] : R(1) - fr[2];
  return x * y * z;
}

// One coupled bead step for one chain: velocity Verlet, FENE/WCA, interpolation of the
// post-stream flow at the 8 corners, friction + Langevin force, and the deterministic
// spreading of the reaction into per-node population corrections.  Run by the G blocks of a
// cluster (G = 1: one block; any size, a multiple of 32; rank: this block's).
//
// The step is a chain of dependent phases and bound by their latency, so what a phase hands
// to the next stays in shared memory (through global memory each hand-over costs an L2 round
// trip) and phases that do not depend on one another run on different warps:
//   0  noise of the block's beads, before the wait for the previous grid;
//   1  drift of every bead in every block (cheaper than an exchange); the threads left over
//      clear the slot's old list meanwhile;
//   2  the first warps gather density and momentum at the corner nodes of the block's beads (38
//      loads each, in flight together), the others compute the weights and conservative forces;
//   3  friction and second half kick of the block's beads; the coupling forces go to every block
//      of the cluster (distributed shared memory); while they travel, the beads whose cells touch
//      those of the block's beads;
//   4  each node is corrected by the block that owns its first entry: the forces of all its
//      entries, summed in entry order, need nothing from other blocks but the forces.
// Comparing the cells of all beads (a corner is shared by beads of touching cells only) replaces
// grouping the corners by a hash table with two scans on block 0 and two cluster barriers.
// Kernel alone under ncu, before and after: N = 32 with two substeps 25 -> 11 us, N = 64 19 -> 11,
// N = 16 14 -> 9 (FP32), N = 8 in FP64 50 -> 26.  Inside (clock stamps, N = 16): noise 0.6 us
// (before the wait), drift 0.6, gathers and forces 1.2, friction 0.4, barrier 0.6, corrections 2.2
// (some 0.3 less since their marks are unrolled):
// single warps issuing dependent instructions, no longer memory.  (Spreading gathers and
// corrections over all warps by population, which multiplies their index arithmetic, came out
// slower: 7.1 against 6.9 us per step at L = 32, N = 16; 31 against 26 for 64 replicas of L = 15.)
template <class S, class R, bool DEV, bool PDL>
__device__ __forceinline__ void bead_step_block(const S* __restrict__ pop, const FluidK<R>& P, const ChainK<R>& C,
                                                const PendK<R>& Pd, const uint32_t step, unsigned char* smem,
                                                const int rank, const int G) {
  const int N = C.N, nsub = C.nsub;
  const int tid = threadIdx.x + blockDim.x * threadIdx.y, nt = blockDim.x * blockDim.y;
  const int lane = tid & 31, warp = tid >> 5, nwarp = nt >> 5;
  const int L = (int)P.L;
  const R h = C.h;
  const int b0 = rank * N / G, nb = (rank + 1) * N / G - b0;  // this block's beads
  const int nc = 8 * nb;                                      // and their corners in one substep
  const int own = nc * nsub, np = N * nsub;                   // entries of the block, places
  BeadSmem<R> M;
  M.carve(smem, N, nsub, (N + G - 1) / G);
  // the chain's number of the block's place i (sub nb + b)
  auto place = [&](int i) {
    if (nsub == 1) return b0 + i;
    const int sub = i / nb;
    return sub * N + b0 + i - sub * nb;
  };
  // 0. noise
  for (int i = tid; i < nb * nsub; i += nt) {
    const int sub = i / nb, b = b0 + i - sub * nb;
    R g[4] = {R(0), R(0), R(0), R(0)};
    if (C.amp != R(0)) gauss4<R>(step * (uint32_t)nsub + (uint32_t)sub, (uint32_t)b, 0u, C.k0, C.k1, g);
    M.g[3 * i] = g[0];
    M.g[3 * i + 1] = g[1];
    M.g[3 * i + 2] = g[2];
  }
  if (PDL) {
    grid_dependency_wait();
    allow_dependent_launch();
  }
  // clear this slot's old list; the list's entries are numbered alike every step, so that a block
  // clears those it rewrites in phase 4.  Other blocks write new corrections (possibly at the
  // same nodes) only after the second cluster barrier.
  bool wrote = false;  // whether the warp has written what other blocks read or write after it
  {
    const int nd = 3 * N, c0 = nd < nt ? nd : 0;
    if (tid >= c0 && *Pd.cur_count > 0)
      for (int i = tid - c0; i < own; i += nt - c0) {
        clear_correction<R>(Pd, L, 8 * place(i >> 3) + (i & 7));
        wrote = true;
      }
  }
  const R* corr = Pd.have_prev ? Pd.prev_dense : nullptr;
  // MD substeps against the frozen post-stream fluid (one for LB step = MD step)
  for (int sub = 0; sub < nsub; ++sub) {
    const int poff = sub * 3 * N, ooff = sub * nc;
    const bool last = sub + 1 == nsub;
    // 1. drift of every bead, cells
    const R* const pv = M.v + ((sub - 1) & 1) * 3 * N;
    const R* const pF = M.F + ((sub - 1) & 1) * 3 * N;
    for (int t = tid; t < 3 * N; t += nt) {
      R vh, hi, lo;
      int im;
      if (sub == 0) {
        im = C.img_in[t];
        drift<R>(C, C.v_in[t], C.F_in[t], C.x_in[t], C.xl_in[t], im, vh, hi, lo);
      } else {  // from the state the previous substep left here
        im = M.img[t];
        drift<R>(C, pv[t], pF[t], M.x[t], M.l[t], im, vh, hi, lo);
      }
      M.x[t] = hi;
      M.l[t] = lo;
      M.vh[t] = vh;
      M.img[t] = im;
      // cell = floor(x/a) mod L; the position inside it from the exact remainder x - floor(x/a) a
      const R f = floor(over_a(hi, C));
      int c = (int)f;
      if ((unsigned)c >= (unsigned)L) {  // x/a rounded up to L, or not finite
        R unused;
        c = cell_of<R>(hi, C.a, L, unused);
      }
      M.cell[poff + t] = c;
      M.fr[t] = over_a(fma(-f, C.a, hi) + lo, C);
    }
    __syncthreads();
    // every block has started and read the state, once all have arrived: waited for before the
    // first remote store and the first write of the state.  The last warp's arrival is a release
    // (with the block's barrier before it for the reads of all its warps); it has the time: 10.05 us
    // per step at L = 25, N = 32, two substeps, as with none, 10.33 with the first warp's, which gathers.
    if (G > 1 && sub == 0) {
      if (warp == nwarp - 1) cluster_arrive();
      else cluster_arrive_relaxed();
    }
    // 2. post-stream density and momentum at the corner nodes of the block's beads ...
    const int gw = (nc + 31) >> 5;            // warps that gather
    const int g0 = gw < nwarp ? 32 * gw : 0;  // the other threads (all, when none is left over)
    for (int i = tid; i < nc; i += nt) {
      const int* cl = M.cell + poff + 3 * (b0 + (i >> 3));
      int q[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        q[j] = cl[j] + ((i >> j) & 1);
        if (q[j] >= L) q[j] -= L;
      }
      R mom[4];
      gather_node_c<S, R, DEV>(pop, P, q[0], q[1], q[2], mom, corr);
      const int o = ooff + i;
      M.node[o] = q[0] + L * (q[1] + L * q[2]);
#pragma unroll
      for (int j = 0; j < 4; ++j) M.mom[j * own + o] = mom[j];
      M.mom[4 * own + o] = R(1) / mom[0];
    }
    //    ... and on the other warps every corner's weight and the conservative forces at x': FENE on
    //    bonds, WCA on all pairs, minimum image; the lanes of a bead split the partners and combine
    //    in a fixed shuffle tree
    if (tid >= g0) {
      const int t1 = tid - g0, n1 = nt - g0;
      for (int i = n1 - 1 - t1; i < 8 * N; i += n1) M.w[sub * 8 * N + i] = corner_weight(M.fr + 3 * (i >> 3), i & 7);
      int lanes = 32;
      while (lanes > 4 && nb * lanes > 2 * n1) lanes /= 2;
      const int fl = t1 % lanes;
      for (int base = 0; base < nb; base += n1 / lanes) {
        const int i = base + t1 / lanes;
        R f[3];
        bead_force<R>(M.x, M.l, C, i < nb ? b0 + i : N, fl, lanes, f);
        if (i < nb && fl < 3) M.fcons[3 * i + fl] = (fl == 0 ? f[0] : (fl == 1 ? f[1] : f[2])) + C.ext[fl];
      }
    }
    if (G > 1 && sub == 0) cluster_wait();
    __syncthreads();
    // 3. friction + Langevin force, second half kick
    auto write_state = [&](int t, R vn, R Ft, R fc) {
      C.x[t] = M.x[t];
      C.xl[t] = M.l[t];
      C.img[t] = M.img[t];
      C.v[t] = vn;
      C.F[t] = Ft;
      C.Fc[t] = fc;
    };
    R vn = R(0), Ft = R(0), fc = R(0);  // of coordinate 3 b0 + mine
    int mine = -1;
    for (int i = tid; i < 3 * nb; i += nt) {
      if (mine >= 0 && last) write_state(3 * b0 + mine, vn, Ft, fc);
      mine = i;
      const int bl = i / 3, q = i - 3 * bl, t = 3 * b0 + i;
      R ub = R(0);
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const int o = ooff + 8 * bl + c;
        ub += M.w[8 * (sub * N + b0 + bl) + c] * M.mom[(q + 1) * own + o] * M.mom[4 * own + o];
      }
      const R vh = M.vh[t];
      fc = -C.zeta * (vh - ub * C.u_scale) + C.amp * M.g[3 * (sub * nb + bl) + q];
      Ft = M.fcons[i] + fc;
      vn = vh + over_2m(h * Ft, C);
      R* const dst[3] = {M.fc + sub * 3 * N + t, M.v + (sub & 1) * 3 * N + t, M.F + (sub & 1) * 3 * N + t};
      if (G == 1) {
        *dst[0] = fc;
        if (!last) {
          *dst[1] = vn;
          *dst[2] = Ft;
        }
      } else {
        wrote = true;
        for (int r = 0; r < G; ++r) {
          cluster_store(dst[0], r, fc);
          if (!last) {
            cluster_store(dst[1], r, vn);
            cluster_store(dst[2], r, Ft);
          }
        }
      }
    }
    if (G > 1) {  // forces sent, old lists cleared (and, before the block's barrier, a substep's start read)
      if (__any_sync(0xffffffffu, wrote)) cluster_arrive();
      else cluster_arrive_relaxed();
    }
    if (!last) {
      if (G > 1)
        cluster_wait();
      else
        __syncthreads();
    } else if (mine >= 0) {  // the end state (every block has read the state: first cluster barrier)
      write_state(3 * b0 + mine, vn, Ft, fc);
    }
  }  // substeps

  // The places whose cells touch the cell of each of the block's places, a warp per place: with the
  // cells d apart (each component -1, 0 or 1), corner c of the one is corner c - d of the other
  // where both lie in {0, 1}^3.
  for (int i = nwarp - 1 - warp; i < nb * nsub; i += nwarp) {
    const int* mine = M.cell + 3 * place(i);
    int n = 0;
    for (int j0 = 0; j0 < np; j0 += 32) {
      const int j = j0 + lane;
      int shared = 0, shift = 0;
      if (j < np) {
        shared = 0xff;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          int d = M.cell[3 * j + q] - mine[q];
          d = d > 1 ? d - L : (d < -1 ? d + L : d);
          const int far = q == 0 ? 0xaa : (q == 1 ? 0xcc : 0xf0);  // corners with bit q set
          shared &= d == 0 ? 0xff : (d == 1 ? far : (d == -1 ? 0xff ^ far : 0));
          shift += d << q;
        }
      }
      const unsigned hit = __ballot_sync(0xffffffffu, shared != 0);
      if (shared) M.near[i * np + n + __popc(hit & ((1u << lane) - 1u))] = j | shared << 8 | (shift + 8) << 16;
      n += __popc(hit);
    }
    if (lane == 0) M.nnear[i] = n;
  }
  if (G > 1) cluster_wait();
  __syncthreads();
  // 4. deterministic spreading: the first entry of each node sums the node's contributions in
  //    entry order and turns the node force into population corrections (the last threads, whose
  //    warps are free)
  for (int o = nt - 1 - tid; o < own; o += nt) {
    const int i = o >> 3, c = o & 7, e = 8 * place(i) + c, node = M.node[o];
    C.e_node[e] = node;
    const int* near = M.near + i * np;
    const int n = M.nnear[i];
    R f[3] = {R(0), R(0), R(0)};
    bool first = false;
    for (int k = 0; k < n; ++k) {
      const int code = near[k];
      if (!((code >> (8 + c)) & 1)) continue;
      const int j = code & 0xff, cj = c - ((code >> 16) - 8);
      if (!first) {
        if (8 * j + cj != e) break;  // an earlier entry has the node
        first = true;
      }
      const R w = M.w[8 * j + cj] * C.spread;
      const R* fc = M.fc + 3 * j;
      f[0] -= w * fc[0] * C.inv_a3;
      f[1] -= w * fc[1] * C.inv_a3;
      f[2] -= w * fc[2] * C.inv_a3;
    }
    if (first)
      node_correction<R>(P, C, Pd, L, e, node, f, M.mom[o], M.mom[own + o], M.mom[2 * own + o], M.mom[3 * own + o]);
    else
      Pd.cur_pos[e] = make_int4(-1, 0, 0, 0);
  }
  // the end state once more, as the bead read-back forms it
  if (C.snap) {
    double* sn = C.snap + (size_t)(step & 1u) * 6 * N;
    for (int i = tid; i < 3 * nb; i += nt) {
      const int t = 3 * b0 + i;
      sn[t] = __dadd_rn(__dadd_rn((double)M.x[t], (double)M.l[t]), __dmul_rn((double)M.img[t], C.snap_box));
      sn[3 * N + t] = (double)C.v[t];
    }
  }
  if (rank == 0 && tid == 0) *Pd.cur_count = 8 * np;
}

// The same step by one block for more than kGroupMax entries: the entries are ordered by node by a
// bitonic sort of (node, entry) keys, and hand-overs go through global memory.  `smem` holds the
// positions (6N R), later the sort keys, leader slots and chunk counts.
template <class S, class R, bool DEV>
__device__ __forceinline__ void bead_step_sorted(const S* __restrict__ pop, const FluidK<R>& P, const ChainK<R>& C,
                                                 const PendK<R>& Pd, const uint32_t step, unsigned char* smem) {
  const int N = C.N;
  const int tid = threadIdx.x + blockDim.x * threadIdx.y, nt = blockDim.x * blockDim.y;
  const int L = (int)P.L;
  const R h = C.h;
  R* sx = reinterpret_cast<R*>(smem);
  R* sl = sx + 3 * N;
  // clear this slot's old list; the threads the first drift leaves idle do it while the others
  // drift (with no thread idle, every thread first)
  {
    const int nd = 3 * N, c0 = nd < nt ? nd : 0;
    if (tid >= c0) {
      const int old = *Pd.cur_count;
      for (int u = tid - c0; u < old; u += nt - c0) clear_correction<R>(Pd, L, u);
    }
  }
  const R* corr = Pd.have_prev ? Pd.prev_dense : nullptr;

  // MD substeps against the frozen post-stream fluid (one for LB step = MD step)
  for (int sub = 0; sub < C.nsub; ++sub) {
  const int eoff = sub * 8 * N;
  // 1. first half kick and drift
  const bool first = sub == 0;  // later substeps continue from the written state
  const R* const vin = first ? C.v_in : C.v;
  const R* const Fin = first ? C.F_in : C.F;
  const R* const xin = first ? C.x_in : C.x;
  const R* const xlin = first ? C.xl_in : C.xl;
  const int* const imgin = first ? C.img_in : C.img;
  for (int t = tid; t < 3 * N; t += nt) {
    R vh, hi, lo;
    int im = imgin[t];
    drift<R>(C, vin[t], Fin[t], xin[t], xlin[t], im, vh, hi, lo);
    C.vh[t] = vh;
    C.x[t] = hi;
    C.xl[t] = lo;
    C.img[t] = im;
    sx[t] = hi;
    sl[t] = lo;
  }
  __syncthreads();

  // 2. conservative forces at x': FENE on bonds, WCA on all pairs, minimum image
  chain_forces_block<R>(sx, sl, C, C.fcons);

  // 3. corners: cell, trilinear weight, post-stream rho and J at the node
  for (int e0 = tid; e0 < 8 * N; e0 += nt) {
    const int b = e0 >> 3, c = e0 & 7, e = eoff + e0;
    const int dx = c & 1, dy = (c >> 1) & 1, dz = (c >> 2) & 1;
    R fr[3];
    int cl[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      R unused;
      const R xh = sx[3 * b + q];
      cl[q] = cell_of<R>(xh, C.a, L, unused);
      // fractional position inside the cell from the exact remainder xh - floor(xh/a) a
      const R f = floor(xh / C.a);
      fr[q] = (fma(-f, C.a, xh) + sl[3 * b + q]) / C.a;
    }
    const int qx = (cl[0] + dx) % L, qy = (cl[1] + dy) % L, qz = (cl[2] + dz) % L;
    const R w = (dx ? fr[0] : R(1) - fr[0]) * (dy ? fr[1] : R(1) - fr[1]) * (dz ? fr[2] : R(1) - fr[2]);
    R mom[4];
    gather_node_c<S, R, DEV>(pop, P, qx, qy, qz, mom, corr);
    C.e_node[e] = qx + L * (qy + L * qz);
    C.e_w[e] = w;
#pragma unroll
    for (int q = 0; q < 4; ++q) C.e_mom[q * C.cap + e] = mom[q];
  }
  __syncthreads();

  // 4. friction + Langevin force, second half kick
  for (int b = tid; b < N; b += nt) {
    R ub[3] = {R(0), R(0), R(0)};
    for (int c = 0; c < 8; ++c) {
      const int e = eoff + 8 * b + c;
      const R w = C.e_w[e];
      const R ir = R(1) / C.e_mom[e];
      ub[0] += w * C.e_mom[1 * C.cap + e] * ir;
      ub[1] += w * C.e_mom[2 * C.cap + e] * ir;
      ub[2] += w * C.e_mom[3 * C.cap + e] * ir;
    }
    R g[4] = {R(0), R(0), R(0), R(0)};
    if (C.amp != R(0)) gauss4<R>(step * (uint32_t)C.nsub + (uint32_t)sub, (uint32_t)b, 0u, C.k0, C.k1, g);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int t = 3 * b + q;
      const R vh = C.vh[t];
      const R fc = -C.zeta * (vh - ub[q] * C.u_scale) + C.amp * g[q];
      const R Ft = C.fcons[t] + fc;
      C.Fc[t] = fc;
      C.fc_hist[sub * 3 * N + t] = fc;
      C.F[t] = Ft;
      const R vn = vh + over_2m(h * Ft, C);
      C.v[t] = vn;
      if (C.snap && sub == C.nsub - 1) {  // the step's end state, as the bead read-back forms it
        double* sn = C.snap + (size_t)(step & 1u) * 6 * N;
        const int im = C.img[t];
        sn[t] = __dadd_rn(__dadd_rn((double)sx[t], (double)sl[t]), __dmul_rn((double)im, C.snap_box));
        sn[3 * N + t] = (double)vn;
      }
    }
  }
  __syncthreads();
  }  // substeps

  // 5. deterministic spreading: order the corner entries by node, sum each node's contributions in
  //    entry order, then turn the node force into population corrections
  const int ne = 8 * N * C.nsub;
  const int lane = tid & 31, warp = tid >> 5, nwarp = nt >> 5;
  int M = 32;  // at least one warp-wide chunk; padding keys sort to the end
  while (M < ne) M <<= 1;
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(smem);
  for (int i = tid; i < M; i += nt)
    keys[i] = (i < ne) ? (((unsigned long long)(unsigned)C.e_node[i] << 32) | (unsigned)i) : ~0ull;
  __syncthreads();
  bitonic_sort_block(keys, M, tid, nt);
  // leaders: first entry of each node run, numbered in order (chunks of 32 entries: each
  // warp counts the leaders of its chunks, warp 0 scans the chunk counts)
  int* slot = reinterpret_cast<int*>(keys + M);
  int* cbase = slot + ne;
  const int nchunk = (ne + 31) >> 5;
  for (int c = warp; c < nchunk; c += nwarp) {
    const int i = (c << 5) + lane;
    const int lead = i < ne && ((i == 0) || ((keys[i] >> 32) != (keys[i - 1] >> 32)));
    const unsigned mask = __ballot_sync(0xffffffffu, lead);
    if (lane == 0) cbase[c] = __popc(mask);
  }
  __syncthreads();
  if (warp == 0) {
    int base = 0;
    for (int c0 = 0; c0 < nchunk; c0 += 32) {
      const int c = c0 + lane;
      const int v = c < nchunk ? cbase[c] : 0;
      int incl = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      if (c < nchunk) cbase[c] = base + incl - v;
      base += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) *Pd.cur_count = base;
  }
  __syncthreads();
  for (int c = warp; c < nchunk; c += nwarp) {
    const int i = (c << 5) + lane;
    const int lead = i < ne && ((i == 0) || ((keys[i] >> 32) != (keys[i - 1] >> 32)));
    const unsigned mask = __ballot_sync(0xffffffffu, lead);
    if (i < ne) slot[i] = lead ? cbase[c] + __popc(mask & ((1u << lane) - 1u)) : -1;
  }
  __syncthreads();
  for (int i = tid; i < ne; i += nt) {
    const int u = slot[i];
    if (u < 0) continue;
    const int node = (int)(keys[i] >> 32);
    int cnt = 1;
    while (i + cnt < ne && (int)(keys[i + cnt] >> 32) == node) ++cnt;
    const int e0 = (int)(keys[i] & 0xffffffffu);
    R f[3] = {R(0), R(0), R(0)};
    for (int r = i; r < i + cnt; ++r) {
      const int e = (int)(keys[r] & 0xffffffffu);
      const R w = C.e_w[e] * C.spread;
      const int sub = e / (8 * N), b = (e - sub * 8 * N) >> 3;
      const R* fch = C.fc_hist + sub * 3 * N;
      f[0] -= w * fch[3 * b + 0] * C.inv_a3;
      f[1] -= w * fch[3 * b + 1] * C.inv_a3;
      f[2] -= w * fch[3 * b + 2] * C.inv_a3;
    }
    node_correction<R>(P, C, Pd, L, u, node, f, C.e_mom[e0], C.e_mom[C.cap + e0], C.e_mom[2 * C.cap + e0],
                       C.e_mom[3 * C.cap + e0]);
  }
}

// The bead step as its own grid (one cluster of G blocks; SORTED: one block).  Launched with
// programmatic stream serialization after the previous step's LB kernel (which completes only
// after the previous bead kernel), it waits for that grid before reading; then it releases the LB
// kernel of the same step, which reads neither its outputs nor anything it writes and runs
// alongside.
template <class S, class R, bool DEV, bool SORTED>
__global__ void __launch_bounds__(512) k_bead_step(const S* __restrict__ pop, const FluidK<R> P,
                                                    const ChainK<R> C, const PendK<R> Pd, const uint32_t step) {
  extern __shared__ __align__(16) unsigned char smem[];
  if constexpr (SORTED) {
    grid_dependency_wait();
    allow_dependent_launch();
    bead_step_sorted<S, R, DEV>(pop, P, C, Pd, launch_step(P, step), smem);
  } else {
    unsigned rank, G;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(G));
    bead_step_block<S, R, DEV, true>(pop, P, C, Pd, launch_step(P, step), smem, (int)rank, (int)G);
  }
}

// B[i][node] += the dense field's corrections at every listed node (each appears once in the list),
// and those entries and the list's mask words (mask may be null) back to zero; one thread per
// (list entry, population): blockIdx.y is the population
template <class S, class R>
__global__ void __launch_bounds__(256) k_apply_pending(S* __restrict__ pop, const FluidK<R> P,
                                                        const int4* __restrict__ p_pos,
                                                        const int* __restrict__ p_count,
                                                        R* __restrict__ dense, unsigned* __restrict__ mask,
                                                        unsigned seg0) {
  const int u = blockIdx.x * blockDim.x + threadIdx.x;
  if (u >= *p_count) return;
  const int i = blockIdx.y;
  const int4 p = p_pos[u];
  if (p.x < 0) return;
  const unsigned long long off = (unsigned long long)i * P.plane + (unsigned)p.x;
  st<S, R>(pop + off, ld<S, R>(pop + off) + dense[off]);
  dense[off] = R(0);
  if (mask && i == 0) clear_marks(mask, seg0, (int)P.L, p.y, p.z, p.w);
}

// one trajectory frame: unwrapped positions x + xl + img * box in FP64, in the order (and
// without contraction) of the host read-back
template <class R>
__global__ void k_record_frame(const R* __restrict__ x, const R* __restrict__ xl, const int* __restrict__ img,
                               int n3, double box, double* __restrict__ dst) {
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n3; t += gridDim.x * blockDim.x)
    dst[t] = __dadd_rn(__dadd_rn((double)x[t], (double)xl[t]), __dmul_rn((double)img[t], box));
}

// bead read-back: out[0..n3) unwrapped positions as k_record_frame forms them, out[n3..2 n3)
// velocities, FP64; the device status word to status_out (may be null)
template <class R>
__global__ void k_bead_readback(const R* __restrict__ x, const R* __restrict__ xl, const int* __restrict__ img,
                                const R* __restrict__ v, int n3, double box, double* __restrict__ out,
                                const unsigned* __restrict__ status, unsigned* __restrict__ status_out) {
  if (status_out && blockIdx.x == 0 && threadIdx.x == 0) *status_out = *status;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n3; t += gridDim.x * blockDim.x) {
    out[t] = __dadd_rn(__dadd_rn((double)x[t], (double)xl[t]), __dmul_rn((double)img[t], box));
    out[n3 + t] = (double)v[t];
  }
}

// ---------------------------------------------------------------------------------------
// initial state, conversions, reductions
// ---------------------------------------------------------------------------------------
template <class S, class R, bool DEV>
__global__ void k_init_rest(S* __restrict__ pop, unsigned long long nnodes, unsigned long long plane, R rho0) {
  const unsigned long long t = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
  if (t >= nnodes) return;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const R v = DEV ? R(0) : rho0 * (R(w36(i)) / R(36));
    st<S, R>(pop + (unsigned long long)i * plane + t, v);
  }
}

// one population plane: full FP64 values <-> storage
// planes p0 .. p0 + gridDim.y - 1 of the stored populations as full FP64 populations:
// dst[(i - p0) n + t] = n_i(t) (+ w_i rho0 for deviation storage); dst may be page-locked host
// memory the device addresses directly
template <class S, class R, bool DEV>
__global__ void __launch_bounds__(256) k_planes_to_f64(double* __restrict__ dst, const S* __restrict__ src,
                                                       unsigned long long n, unsigned long long plane, int p0,
                                                       double rho0) {
  const int i = p0 + (int)blockIdx.y;
  const double wr = DEV ? rho0 * (double)w36(i) / 36.0 : 0.0;
  const S* s = src + (unsigned long long)i * plane;
  double* d = dst + (unsigned long long)blockIdx.y * n;
  for (unsigned long long t = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; t < n;
       t += (unsigned long long)gridDim.x * blockDim.x)
  {
    const double v = (double)ld<S, R>(s + t);
    d[t] = DEV ? v + wr : v;
  }
}
// the inverse: planes p0 .. p0 + gridDim.y - 1 of the stored populations from FP64 src
template <class S, class R, bool DEV>
__global__ void __launch_bounds__(256) k_planes_from_f64(S* __restrict__ dst, const double* __restrict__ src,
                                                         unsigned long long n, unsigned long long plane, int p0,
                                                         double rho0) {
  const int i = p0 + (int)blockIdx.y;
  const double wr = DEV ? rho0 * (double)w36(i) / 36.0 : 0.0;
  S* d = dst + (unsigned long long)i * plane;
  const double* s = src + (unsigned long long)blockIdx.y * n;
  for (unsigned long long t = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; t < n;
       t += (unsigned long long)gridDim.x * blockDim.x)
    st<S, R>(d + t, (R)(DEV ? s[t] - wr : s[t]));
}

// per-block FP64 partial sums of (sum n, Jx, Jy, Jz) of the stored populations
template <class S, class R, bool DEV>
__global__ void __launch_bounds__(256) k_fluid_partials(const S* __restrict__ pop, unsigned long long nnodes,
                                                         unsigned long long plane, double* __restrict__ part) {
  const unsigned long long t = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
  double v[4] = {0, 0, 0, 0};
  if (t < nnodes) {
    R r = R(0), jx = R(0), jy = R(0), jz = R(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const R n = ld<S, R>(pop + (unsigned long long)i * plane + t);
      r += n;
      if (cx(i)) jx += R(cx(i)) * n;
      if (cy(i)) jy += R(cy(i)) * n;
      if (cz(i)) jz += R(cz(i)) * n;
    }
    v[0] = (double)r;
    v[1] = (double)jx;
    v[2] = (double)jy;
    v[3] = (double)jz;
  }
  __shared__ double sh[4][8];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    double a = v[q];
    for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    if ((threadIdx.x & 31) == 0) sh[q][threadIdx.x >> 5] = a;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double a = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) a += sh[threadIdx.x][w];
    part[4ull * blockIdx.x + threadIdx.x] = a;
  }
}

// observables: fluid sums from the partials, bead quantities from the chain state (FP64)
template <class R>
struct ObsK {
  const double* part;
  int nparts;
  double mass_rest;   // rho0 L^3 for deviation storage (0 for full storage)
  double a3, u_scale;  // a^3, a/h
  int N;
  const R* x;
  const R* xl;
  const int* img;
  const R* v;
  const R* Fc;
  double box, m, h;
  const double* xref;  // 3N reference positions
  double* acc;         // [samples, sum Rg2, sum Re2]
  const unsigned long long* nonpos;
  double* out;         // LB_NOBS values
  long long step;
  int accumulate;      // 1: add this sample to the accumulators
};

template <class R>
__global__ void __launch_bounds__(256) k_observables(const ObsK<R> O) {
  __shared__ double sh[16][8];
  const int tid = threadIdx.x;
  // fluid: fixed-order reduction of the partials
  double f[4] = {0, 0, 0, 0};
  for (int p = tid; p < O.nparts; p += blockDim.x)
    for (int q = 0; q < 4; ++q) f[q] += O.part[4ll * p + q];
  // beads
  double cm[3] = {0, 0, 0}, mv[3] = {0, 0, 0}, fc[3] = {0, 0, 0}, v2 = 0;
  for (int b = tid; b < O.N; b += blockDim.x) {
    for (int q = 0; q < 3; ++q) {
      const double xu = (double)O.x[3 * b + q] + (double)O.xl[3 * b + q] + (double)O.img[3 * b + q] * O.box;
      cm[q] += xu;
      const double vv = (double)O.v[3 * b + q];
      mv[q] += O.m * vv;
      v2 += vv * vv;
      fc[q] += (double)O.Fc[3 * b + q];
    }
  }
  double vals[14] = {f[0], f[1], f[2], f[3], cm[0], cm[1], cm[2], mv[0], mv[1], mv[2], fc[0], fc[1], fc[2], v2};
  for (int q = 0; q < 14; ++q) {
    double a = vals[q];
    for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    if ((tid & 31) == 0) sh[q][tid >> 5] = a;
  }
  __syncthreads();
  __shared__ double tot[14];
  if (tid < 14) {
    double a = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) a += sh[tid][w];
    tot[tid] = a;
  }
  __syncthreads();
  // second pass: R_g^2 about the centre of mass, R_e^2, MSDs
  const int N = O.N;
  double rg = 0;
  for (int b = tid; b < N; b += blockDim.x) {
    for (int q = 0; q < 3; ++q) {
      const double xu = (double)O.x[3 * b + q] + (double)O.xl[3 * b + q] + (double)O.img[3 * b + q] * O.box;
      const double d = xu - tot[4 + q] / N;
      rg += d * d;
    }
  }
  for (int o = 16; o > 0; o >>= 1) rg += __shfl_down_sync(0xffffffffu, rg, o);
  __syncthreads();
  if ((tid & 31) == 0) sh[15][tid >> 5] = rg;
  __syncthreads();
  if (tid == 0) {
    double rgt = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) rgt += sh[15][w];
    double* o = O.out;
    o[0] = (double)O.step;
    o[1] = (O.mass_rest + tot[0]) * O.a3;
    const double s = O.u_scale * O.a3;
    o[5] = tot[1] * s;
    o[6] = tot[2] * s;
    o[7] = tot[3] * s;
    o[2] = o[5] + tot[7] + 0.5 * O.h * tot[10];
    o[3] = o[6] + tot[8] + 0.5 * O.h * tot[11];
    o[4] = o[7] + tot[9] + 0.5 * O.h * tot[12];
    double Rg2 = 0, Re2 = 0, g1 = 0, g3 = 0;
    if (N > 0) {
      Rg2 = rgt / N;
      double cmr[3] = {0, 0, 0};
      for (int b = 0; b < N; ++b)
        for (int q = 0; q < 3; ++q) cmr[q] += O.xref[3 * b + q];
      const int i0 = (N - 1) / 2, i1 = N / 2;
      for (int q = 0; q < 3; ++q) {
        const double xe = (double)O.x[3 * (N - 1) + q] + (double)O.xl[3 * (N - 1) + q] + (double)O.img[3 * (N - 1) + q] * O.box;
        const double xs = (double)O.x[q] + (double)O.xl[q] + (double)O.img[q] * O.box;
        Re2 += (xe - xs) * (xe - xs);
        const double a0 = (double)O.x[3 * i0 + q] + (double)O.xl[3 * i0 + q] + (double)O.img[3 * i0 + q] * O.box - O.xref[3 * i0 + q];
        const double a1 = (double)O.x[3 * i1 + q] + (double)O.xl[3 * i1 + q] + (double)O.img[3 * i1 + q] * O.box - O.xref[3 * i1 + q];
        g1 += 0.5 * (a0 * a0 + a1 * a1);
        const double dc = (tot[4 + q] - cmr[q]) / N;
        g3 += dc * dc;
      }
      o[10] = tot[4] / N;
      o[11] = tot[5] / N;
      o[12] = tot[6] / N;
      o[15] = O.m * tot[13] / (3.0 * N);
    } else {
      o[10] = o[11] = o[12] = 0;
      o[15] = 0;
    }
    o[8] = Rg2;
    o[9] = Re2;
    o[13] = g1;
    o[14] = g3;
    o[16] = (double)*O.nonpos;
    if (O.accumulate) {
      O.acc[0] += 1.0;
      O.acc[1] += Rg2;
      O.acc[2] += Re2;
    }
    o[17] = O.acc[0];
    o[18] = O.acc[0] > 0 ? O.acc[1] / O.acc[0] : 0.0;
    o[19] = O.acc[0] > 0 ? O.acc[2] / O.acc[0] : 0.0;
  }
}

}  // namespace gblb

namespace gblb {

// Forces of the initial configuration: F = F_cons(x0) (+ external), F_c = 0.
template <class R>
__global__ void __launch_bounds__(512) k_chain_init_forces(const ChainK<R> C) {
  extern __shared__ __align__(16) unsigned char smem[];
  R* sx = reinterpret_cast<R*>(smem);
  R* sl = sx + 3 * C.N;
  for (int t = threadIdx.x; t < 3 * C.N; t += blockDim.x) {
    sx[t] = C.x[t];
    sl[t] = C.xl[t];
  }
  __syncthreads();
  chain_forces_block<R>(sx, sl, C, C.F);
  __syncthreads();
  for (int t = threadIdx.x; t < 3 * C.N; t += blockDim.x) C.Fc[t] = R(0);
}

}  // namespace gblb
