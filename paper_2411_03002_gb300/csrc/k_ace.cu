// Linear atomic cluster expansion (Eq. energy_ace, linear part) for the atoms of
// the precise work queue, and its hand-written adjoint (forces).
//
// Basis (project-defined; the paper specifies ACE only by reference):
//   g_k(r)  = T_k(2r/rc - 1) f_cut(r/rc), k = 0..7          (f_cut of Appendix B)
//   R_nl(r) = sum_k W[l][n][k] g_k(r),    n = 0..7, l = 0..4
//   A_nlm   = (1/N0) sum_j R_nl(r_ij) Y_lm(r_ij/|r_ij|)     (real orthonormal Y_lm)
//   B: nu=1 A_n00; nu=2 sum_m A_n1lm A_n2lm; nu=3 sum_m G A A A (real Gaunt G)
//   E_i = sum_v c_v B_iv
// Because R is linear in g, A = W . G with G_klm = sum_j g_k Y_lm, and the force
// needs only u_klm = (1/N0) sum_n W[l][n][k] dE/dA_nlm per atom:
//   dE_i/dr_ij = sum_lm [ (sum_k u_klm g'_k) Y_lm r^ + (sum_k u_klm g_k) grad Y_lm ].
// Three kernels per evaluation, communicating through per-queue-position scratch:
//   k_ace_basis    one warp per precise atom (persistent CTAs, atomic work counter):
//                  row entries inside r_c compacted; G = g^T Y over 32-neighbour
//                  shared tiles; A = (1/N0) W . G; nu = 1, 2 energy and gradient;
//   k_ace_nu3      (k_ace_nu3.cu) the nu = 3 energy and gradient as straight-line code over
//                  the merged monomials generated from the basis (ace_nu3.inc);
//   k_ace_adjoint  8 or 32 lanes per precise atom: u = W^T dE/dA / N0; each lane evaluates
//                  the pair force of one neighbour at a time from u (pair_force) and
//                  scatters -w_i p_ij to neighbour j; +w_i sum p goes to i.
#include <complex>
#include <algorithm>
#include <cstring>
#include <cmath>

#include "ace_args.cuh"

namespace ap {

// ------------------------------------------------------------------ device code
namespace {

constexpr int kCols = 36;            // 32 neighbour slots + 4 pad (16-byte rows, conflict-free)
constexpr int kRows = 33;            // 8 radial + 25 angular rows
// Tensor-core staging of one 32-neighbour batch (FP32 path), per k-step of 8 neighbours:
// the Y^T operand fragments [m-tile 2][lane 32][4] + 16 pad floats, and the g operand
// fragments [lane 32][2] + 8 pad floats.  The pads put the four k-steps of one store
// on different banks.
constexpr int kTyStep = 2 * 128 + 16;
constexpr int kTgStep = 64 + 8;
template <typename R>
constexpr int kTileWords = sizeof(R) == 4 ? 4 * kTyStep + 4 * kTgStep : kRows * kCols;
// Warps per CTA and the minimum resident CTAs per SM
// the compiler budgets registers for; compile-time tuning parameters.
#ifndef AP_ACE_WARPS
#define AP_ACE_WARPS 6
#endif
#ifndef AP_ACE_MINB
#define AP_ACE_MINB 4   // FP32 only: four 6-warp CTAs per SM (shared memory and <= 85 registers)
#endif
template <typename R>
constexpr int kWarps = sizeof(R) == 4 ? AP_ACE_WARPS : 4;

__device__ inline float rsqrt_(float v) { return rsqrtf(v); }
__device__ inline double rsqrt_(double v) { return rsqrt(v); }

template <typename R>
__device__ inline typename V<R>::R4 ld4(const R* p) {
  return *reinterpret_cast<const typename V<R>::R4*>(p);
}

__device__ inline int l_of(int lm) { return lm >= 16 ? 4 : lm >= 9 ? 3 : lm >= 4 ? 2 : lm >= 1 ? 1 : 0; }

// Radial functions g_k = T_k(c) f_cut, c = 2 r/rc - 1, for r < rc.
template <typename R>
__device__ inline void radial(R r, R inv_rc, int mode, R g[8]) {
  R x = r * inv_rc;
  R t = mode == 1 ? R(2) * x - R(1) : x;
  R t2 = t * t;
  R poly = R(1) - R(1.875) * t + R(1.25) * t2 * t - R(0.375) * t2 * t2 * t;
  R fc = mode == 1 ? R(0.5) * poly : poly;
  R c = R(2) * x - R(1);
  R T0 = R(1), T1 = c;
  g[0] = fc;
  g[1] = c * fc;
#pragma unroll
  for (int k = 2; k < 8; ++k) {
    R T2 = R(2) * c * T1 - T0;
    g[k] = T2 * fc;
    T0 = T1;
    T1 = T2;
  }
}

// Real harmonics in the factored form Y_lm = N_lm Pi_lm(z) {A_m | B_m}(x, y) of a unit vector:
// A_m + i B_m = (x + i y)^m (A for m >= 0, B for m < 0) and Pi_lm the monic polynomial
// proportional to d^m P_l/dz^m.  kNorm[l^2 + l + m] = N_lm = sqrt((2l + 1)/(4 pi) (l - m)!/(l + m)!)
// (sqrt 2 if m > 0) (2l)!/(2^l l! (l - m)!).  The adjoint keeps its u rows in the order of
// evaluation, by m, cosine before sine, l ascending: kSlot[l^2 + l + m].
__constant__ double kNorm[25] = {
    0.28209479177387814, 0.48860251190291998, 0.48860251190291992, 0.48860251190291998, 0.54627421529603959,
    1.0925484305920792,  0.94617469575756008, 1.0925484305920792,  0.54627421529603959, 0.59004358992664363,
    1.4453057213202771,  2.2852289973223292,  1.865881662950577,   2.2852289973223292,  1.4453057213202771,
    0.59004358992664363, 0.62583573544917637, 1.7701307697799304,  3.3116114351514598,  4.6833258049010249,
    3.7024941420321507,  4.6833258049010249,  3.3116114351514598,  1.7701307697799304,  0.62583573544917637};
__constant__ unsigned char kSlot[25] = {0,  9,  1,  5,  16, 10, 2,  6,  13, 21, 17, 11, 3,
                                        7,  14, 19, 24, 22, 18, 12, 4,  8,  15, 20, 23};

// Y_lm / N_lm of a unit vector (x, y, z), index lm = l^2 + l + m: 32 operations, the norms being
// left to the sums over the neighbours (k_ace_basis FP64 1.31 -> 1.17 ms for 12,700 atoms, FP32
// 0.89 -> 0.87 ms for 255,840; about 70 operations with the norms in every value).
template <typename R>
__device__ inline void sh_values(R x, R y, R z, R Y[25]) {
  const R w = z * z;
  const R A2 = fma(x, x, -y * y), B2 = R(2) * x * y;
  const R A3 = fma(x, A2, -y * B2), B3 = fma(x, B2, y * A2);
  const R p31 = w - R(0.2), p41 = z * (w - R(3.0 / 7.0)), p42 = w - R(1.0 / 7.0);
  Y[0] = R(1);
  Y[1] = y;
  Y[2] = z;
  Y[3] = x;
  Y[4] = B2;
  Y[5] = z * y;
  Y[6] = w - R(1.0 / 3.0);
  Y[7] = z * x;
  Y[8] = A2;
  Y[9] = B3;
  Y[10] = z * B2;
  Y[11] = p31 * y;
  Y[12] = z * (w - R(0.6));
  Y[13] = p31 * x;
  Y[14] = z * A2;
  Y[15] = A3;
  Y[16] = fma(x, B3, y * A3);
  Y[17] = z * B3;
  Y[18] = p42 * B2;
  Y[19] = p41 * y;
  Y[20] = fma(w, w - R(6.0 / 7.0), R(3.0 / 35.0));
  Y[21] = p41 * x;
  Y[22] = p42 * A2;
  Y[23] = z * A3;
  Y[24] = fma(x, A3, -y * B3);
}

template <typename R>
__device__ inline void pair_disp(const SysInfo& S, const typename V<R>::S4& si, const typename V<R>::S4& sj,
                                 const int* off, size_t e, R d[3]) {
  int k0, k1, k2;
  if (off) {
    int p = off[e];
    k0 = off_x(p);
    k1 = off_y(p);
    k2 = off_z(p);
  } else {
    int wi = V<R>::code(si), wj = V<R>::code(sj);
    k0 = wrap_off(cell_x(wj) - cell_x(wi), S.nc[0], S.periodic[0]);
    k1 = wrap_off(cell_y(wj) - cell_y(wi), S.nc[1], S.periodic[1]);
    k2 = wrap_off(cell_z(wj) - cell_z(wi), S.nc[2], S.periodic[2]);
  }
  if constexpr (sizeof(R) == 4) {
    d[0] = (R)k0 * S.hf[0] + (sj.x - si.x);
    d[1] = (R)k1 * S.hf[1] + (sj.y - si.y);
    d[2] = (R)k2 * S.hf[2] + (sj.z - si.z);
  } else {
    d[0] = (R)k0 * S.h[0] + (sj.x - si.x);
    d[1] = (R)k1 * S.h[1] + (sj.y - si.y);
    d[2] = (R)k2 * S.h[2] + (sj.z - si.z);
  }
}

// Fixed-point force accumulation (ace_deterministic): contributions rounded to multiples
// of 2^-36 eV/A, summed with exact, order-independent 64-bit integer atomics.
__device__ inline unsigned long long to_fix(double v) { return (unsigned long long)llrint(v * kFixScale); }

template <typename R>
__device__ inline void add_force(float4* facc32, double* facc64, unsigned long long* fix, int j, R sx, R sy, R sz) {
  if (fix) {
    atomicAdd(&fix[3 * j + 0], to_fix((double)sx));
    atomicAdd(&fix[3 * j + 1], to_fix((double)sy));
    atomicAdd(&fix[3 * j + 2], to_fix((double)sz));
    return;
  }
  if constexpr (sizeof(R) == 4) {
    atomicAdd(&facc32[j], make_float4(sx, sy, sz, 0.f));
  } else {
    atomicAdd(&facc64[3 * j + 0], sx);
    atomicAdd(&facc64[3 * j + 1], sy);
    atomicAdd(&facc64[3 * j + 2], sz);
  }
}

// Force of one pair, p = dE_i/dr_ij, from the atom's coefficients U[slot][k] = N_lm u_klm:
//   E = f_cut(r) sum_lm P_lm(c) Pi_lm {A_m | B_m},  P_lm = sum_k U_k T_k(c),  Q_lm = dP_lm/dc.
// The sums over l are taken first, per m and for cosine and sine: C = sum_l P Pi, Cq = sum_l Q Pi,
// D = sum_l P dPi/dz.  Then V = sum C A, Vq = sum Cq A, and the gradient t of the (not
// homogeneous) extension needs x and y parts once per m instead of once per (l, m), with
// d(A_m + i B_m) = m (A_{m-1} + i B_{m-1}) d(x + i y).  Only its tangential part t - (t.u) u
// counts:  p = (f_cut' V + 2 f_cut/rc Vq) u + f_cut/r (t - (t.u) u).
// About 490 FP operations a pair; contracting g and g' with u and adding Y and grad Y per
// (l, m) took about 800.  These operations are what the kernel is bound by, in FP32 (issue)
// and above all in FP64 (one warp instruction per 16 cycles and SM).  Kernel times before and
// after, with the lane rule below: FP64 2.63 -> 1.47 ms (12,700 atoms), FP32 1.28 -> 0.89 ms
// (255,840 atoms).
template <typename R>
__device__ inline void pair_force(const R* __restrict__ U, R x, R y, R z, R r, R ir, R inv_rc, int mode, R& px, R& py,
                                  R& pz) {
  const R rr = r * inv_rc;
  const R c = fma(R(2), rr, R(-1)), c2 = c + c;
  R T[8], D[8];   // T_k and dT_k/dc
  T[1] = c;
  T[2] = fma(c2, c, R(-1));
  D[2] = c2 + c2;
  D[1] = R(1);
#pragma unroll
  for (int k = 3; k < 8; ++k) {
    T[k] = fma(c2, T[k - 1], -T[k - 2]);
    D[k] = fma(c2, D[k - 1], fma(R(2), T[k - 1], -D[k - 2]));
  }
  auto pq = [&](int slot, R& P, R& Q) {
    const auto ua = ld4<R>(U + slot * 8);
    const auto ub = ld4<R>(U + slot * 8 + 4);
    P = fma(ua.y, T[1], ua.x);
    P = fma(ua.z, T[2], P);
    P = fma(ua.w, T[3], P);
    P = fma(ub.x, T[4], P);
    P = fma(ub.y, T[5], P);
    P = fma(ub.z, T[6], P);
    P = fma(ub.w, T[7], P);
    Q = fma(ua.z, D[2], ua.y);
    Q = fma(ua.w, D[3], Q);
    Q = fma(ub.x, D[4], Q);
    Q = fma(ub.y, D[5], Q);
    Q = fma(ub.z, D[6], Q);
    Q = fma(ub.w, D[7], Q);
  };
  const R w = z * z, z2 = z + z;
  R V, Vq, tx, ty, tz, P, Q;
  {   // m = 0
    const R q2 = w - R(1.0 / 3.0), q3 = z * (w - R(0.6)), q4 = fma(w, w - R(6.0 / 7.0), R(3.0 / 35.0));
    pq(0, V, Vq);
    pq(1, P, Q);
    V = fma(P, z, V);
    Vq = fma(Q, z, Vq);
    tz = P;
    pq(2, P, Q);
    V = fma(P, q2, V);
    Vq = fma(Q, q2, Vq);
    tz = fma(P, z2, tz);
    pq(3, P, Q);
    V = fma(P, q3, V);
    Vq = fma(Q, q3, Vq);
    tz = fma(P, fma(R(3), w, R(-0.6)), tz);
    pq(4, P, Q);
    V = fma(P, q4, V);
    Vq = fma(Q, q4, Vq);
    tz = fma(P, z * fma(R(4), w, R(-12.0 / 7.0)), tz);
  }
  R C, Cq, E;   // per m and parity: sum_l P Pi, sum_l Q Pi, sum_l P dPi/dz
  {             // m = 1
    const R p3 = w - R(0.2), p4 = z * (w - R(3.0 / 7.0)), d4 = fma(R(3), w, R(-3.0 / 7.0));
    auto sum1 = [&](int s) {
      pq(s, C, Cq);
      pq(s + 1, P, Q);
      C = fma(P, z, C);
      Cq = fma(Q, z, Cq);
      E = P;
      pq(s + 2, P, Q);
      C = fma(P, p3, C);
      Cq = fma(Q, p3, Cq);
      E = fma(P, z2, E);
      pq(s + 3, P, Q);
      C = fma(P, p4, C);
      Cq = fma(Q, p4, Cq);
      E = fma(P, d4, E);
    };
    sum1(5);
    V = fma(C, x, V);
    Vq = fma(Cq, x, Vq);
    tx = C;
    tz = fma(E, x, tz);
    sum1(9);
    V = fma(C, y, V);
    Vq = fma(Cq, y, Vq);
    ty = C;
    tz = fma(E, y, tz);
  }
  // A_m, B_m and the next lower ones times m (the x and y derivatives)
  auto cosine = [&](R A, R mA, R mB) {
    V = fma(C, A, V);
    Vq = fma(Cq, A, Vq);
    tx = fma(C, mA, tx);
    ty = fma(-C, mB, ty);
  };
  auto sine = [&](R B, R mA, R mB) {
    V = fma(C, B, V);
    Vq = fma(Cq, B, Vq);
    tx = fma(C, mB, tx);
    ty = fma(C, mA, ty);
  };
  const R A2 = fma(x, x, -y * y), B2 = R(2) * x * y;
  {   // m = 2
    const R p4 = w - R(1.0 / 7.0);
    auto sum2 = [&](int s) {
      pq(s, C, Cq);
      pq(s + 1, P, Q);
      C = fma(P, z, C);
      Cq = fma(Q, z, Cq);
      E = P;
      pq(s + 2, P, Q);
      C = fma(P, p4, C);
      Cq = fma(Q, p4, Cq);
      E = fma(P, z2, E);
    };
    const R mA = x + x, mB = y + y;
    sum2(13);
    cosine(A2, mA, mB);
    tz = fma(E, A2, tz);
    sum2(16);
    sine(B2, mA, mB);
    tz = fma(E, B2, tz);
  }
  const R A3 = fma(x, A2, -y * B2), B3 = fma(x, B2, y * A2);
  {   // m = 3
    const R mA = R(3) * A2, mB = R(3) * B2;
    pq(19, C, Cq);
    pq(20, P, Q);
    C = fma(P, z, C);
    Cq = fma(Q, z, Cq);
    cosine(A3, mA, mB);
    tz = fma(P, A3, tz);
    pq(21, C, Cq);
    pq(22, P, Q);
    C = fma(P, z, C);
    Cq = fma(Q, z, Cq);
    sine(B3, mA, mB);
    tz = fma(P, B3, tz);
  }
  {   // m = 4
    const R mA = R(4) * A3, mB = R(4) * B3;
    pq(23, C, Cq);
    cosine(fma(x, A3, -y * B3), mA, mB);
    pq(24, C, Cq);
    sine(fma(x, B3, y * A3), mA, mB);
  }
  const R t = mode == 1 ? c : rr;   // the f_cut argument (mode 1: 2 r/rc - 1)
  const R t2 = t * t;
  R fc = R(1) - R(1.875) * t + R(1.25) * t2 * t - R(0.375) * t2 * t2 * t;
  if (mode == 1) fc *= R(0.5);
  const R dfc = (R(-1.875) + R(3.75) * t2 - R(1.875) * t2 * t2) * inv_rc;
  const R ft = fc * ir;
  const R tu = fma(tx, x, fma(ty, y, tz * z));
  const R a = fma(dfc, V, fma(R(2) * fc * inv_rc, Vq, -ft * tu));
  px = fma(a, x, ft * tx);
  py = fma(a, y, ft * ty);
  pz = fma(a, z, ft * tz);
}

template <typename T>
__device__ inline T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <typename T, int L>
__device__ inline T lane_sum(T v) {   // over groups of L lanes
#pragma unroll
  for (int o = L / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The warp's next work item: items below `first` were dealt out statically.
__device__ inline int next_item(int* counter, int step, int first) {
  int q = 0;
  if ((threadIdx.x & 31) == 0) q = atomicAdd(counter, step);
  return first + __shfl_sync(0xffffffffu, q, 0);
}

// ---- 3xTF32 on warp-level tensor cores (FP32 path).  An FP32 value x is carried as
// hi + lo: hi = x rounded to the 10-bit TF32 significand (ties away from zero), lo =
// x - hi (exact in FP32); the tensor core reads the leading TF32 bits of lo.  A
// product of two such pairs drops lo * lo', which leaves about the error of an FP32
// product (relative 2^-21 per term).
__device__ inline void tf32_split(float x, uint32_t& h, uint32_t& l) {
  h = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
  l = __float_as_uint(x - __uint_as_float(h));
}

// D += A B on one m16n8k8 tile (A 16x8 row-major, B 8x8 column-major, TF32 inputs, FP32
// accumulation).  Fragments of lane (g = lane / 4, t = lane % 4):
//   a = A[g][t], A[g+8][t], A[g][t+4], A[g+8][t+4];  b = B[t][g], B[t+4][g];
//   d = D[g][2t], D[g][2t+1], D[g+8][2t], D[g+8][2t+1].
__device__ inline void mma_tf32(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// D += (Ah + Al)(Bh + Bl) without Al Bl, the small products first.
__device__ inline void mma3(float (&d)[4], const uint32_t (&ah)[4], const uint32_t (&al)[4], uint32_t bh0,
                            uint32_t bh1, uint32_t bl0, uint32_t bl1) {
  mma_tf32(d, al, bh0, bh1);
  mma_tf32(d, ah, bl0, bl1);
  mma_tf32(d, ah, bh0, bh1);
}

// out[lm][n] = sum_k in[lm][k] F[l(lm)][n][k] for the 25 (l, m) rows (two m-tiles, rows
// 25..31 zero) and an 8 x 8 factor per l (F in shared memory, F[(l * 8 + n) * 8 + k]).
// `in` is held as m16n8k8 accumulator fragments (rows lm = 16 mt + g, + 8; columns
// k = 2t, 2t + 1), and so is `out`: the accumulator feeds the next product directly,
// with the contraction index relabelled (operand column t <-> k = 2t, t + 4 <-> 2t + 1,
// and B's rows the same way).  Rows of one m-tile carry several l, so tile 0 takes one
// product per l = 0..3 and every lane keeps the rows of its own l; tile 1 is l = 4.
__device__ inline void lm_mix(const float (&in)[2][4], const float* __restrict__ F, int g, int t,
                              float (&out)[2][4]) {
  uint32_t ah[2][4], al[2][4];
#pragma unroll
  for (int mt = 0; mt < 2; ++mt) {
    tf32_split(in[mt][0], ah[mt][0], al[mt][0]);
    tf32_split(in[mt][2], ah[mt][1], al[mt][1]);
    tf32_split(in[mt][1], ah[mt][2], al[mt][2]);
    tf32_split(in[mt][3], ah[mt][3], al[mt][3]);
  }
  const int l0 = g == 0 ? 0 : g < 4 ? 1 : 2;   // l of row g
  const int l1 = g == 0 ? 2 : 3;               // l of row g + 8
#pragma unroll
  for (int l = 0; l < 5; ++l) {
    const float2 f = *reinterpret_cast<const float2*>(&F[l * 64 + g * 8 + 2 * t]);
    uint32_t bh0, bl0, bh1, bl1;
    tf32_split(f.x, bh0, bl0);
    tf32_split(f.y, bh1, bl1);
    float d[4] = {0.f, 0.f, 0.f, 0.f};
    if (l < 4) {
      mma3(d, ah[0], al[0], bh0, bh1, bl0, bl1);
      if (l == l0) {
        out[0][0] = d[0];
        out[0][1] = d[1];
      }
      if (l == l1) {
        out[0][2] = d[2];
        out[0][3] = d[3];
      }
    } else {
      mma3(d, ah[1], al[1], bh0, bh1, bl0, bl1);
#pragma unroll
      for (int e = 0; e < 4; ++e) out[1][e] = d[e];
    }
  }
}

constexpr int kListCap = 192;   // in-range records per precise atom cached in shared memory (FCC bulk: 134)
#ifndef AP_ACE3_WARPS
#define AP_ACE3_WARPS 6
#endif
#ifndef AP_ACE3_MINB
#define AP_ACE3_MINB 4
#endif
template <typename R>
constexpr int kWarps3 = sizeof(R) == 4 ? AP_ACE3_WARPS : 4;   // warps per CTA of the adjoint kernel

// Kernel 1, one warp per precise atom (persistent CTAs, atomic work counter):
//   pass 0   row entries inside r_c compacted (displacement and j) into shared memory,
//            their row positions kept for kernel 3;
//   stage A  lanes evaluate g and Y for 32 neighbours into a shared tile, then
//            contract G = g^T Y; A = (1/N0) W . G;
//   nu = 1, 2: E12 and dE12/dA (symmetric 8x8 matrix-vector products per (l, m)).
// FP32: the three contractions run on the tensor cores (warp-level m16n8k8 TF32 MMAs
// with the 3xTF32 split, FP32 accumulation), G and A staying in accumulator fragments.
// FP64: SIMT loops, G with 4-wide vector loads along the neighbour axis.
template <typename R>
__global__ void __launch_bounds__(kWarps<R> * 32, sizeof(R) == 4 ? AP_ACE_MINB : 1) k_ace_basis(AceArgs<R> a) {
  // Shared memory: W [320] | M2 [320] | C1 [8] | M2b [320] | C1b [8] | C1l [8] | C1bl [8] | per warp: list
  // [kListCap][4] | tile [kTileWords] (FP32: operand fragments of one batch; FP64: the
  // g/Y tile [kRows][kCols], which A and the G scratch alias after stage A).
  extern __shared__ __align__(128) unsigned char smem_raw[];
  R* Ws = reinterpret_cast<R*>(smem_raw);
  R* M2 = Ws + 320;
  R* C1 = M2 + 320;
  R* M2b = C1 + 8;
  R* C1b = M2b + 320;
  R* C1l = C1b + 8;    // what FP32 rounds off C1 and C1b (0 in FP64)
  R* C1bl = C1l + 8;
  R* wbase = C1bl + 8;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  R* list = wbase + warp * (4 * kListCap + kTileWords<R>);
  R* tile = list + 4 * kListCap;
  for (int t = threadIdx.x; t < 320; t += blockDim.x) {
    Ws[t] = a.W[t];
    M2[t] = a.M2[t];
    M2b[t] = a.M2b[t];
  }
  if (threadIdx.x < 8) {
    C1[threadIdx.x] = a.C1[threadIdx.x];
    C1b[threadIdx.x] = a.C1b[threadIdx.x];
    C1l[threadIdx.x] = a.C1l[threadIdx.x];
    C1bl[threadIdx.x] = a.C1l[8 + threadIdx.x];
  }
  __syncthreads();
  const int m = *a.count;
  const int kq = lane & 7, grp = lane >> 3;
  const unsigned lt_mask = (1u << lane) - 1u;
  unsigned long long cnt_pairs = 0, cnt_atoms = 0, cnt_mma = 0;   // profiling counts of this warp
  const int q_first = warp * gridDim.x + blockIdx.x, q_all = kWarps<R> * gridDim.x;
  // norms N_lm of this lane's G entries: FP32 rows lm = lane / 4 + 8 u, FP64 lm = grp + 4 t
  R norm[sizeof(R) == 4 ? 4 : 7];
#pragma unroll
  for (int u = 0; u < (sizeof(R) == 4 ? 4 : 7); ++u) {
    const int lm = sizeof(R) == 4 ? (lane >> 2) + 8 * u : grp + 4 * u;
    norm[u] = lm < 25 ? (R)kNorm[lm] : R(0);
  }
  for (int q = q_first; q < m; q = next_item(a.counter, 1, q_all)) {
    const int i = a.queue[q];
    const SysInfo& S = a.sys[a.atom_sys ? a.atom_sys[i] : 0];
    const auto si = a.sh[i];
    const int c = a.cnt[q];
    const size_t row = (size_t)q * a.cap;

    // ---------------- pass 0: compact the row entries inside ace_rc.  The dependent loads
    // (row entry, then its shadow) run ahead of their use: the entry two batches ahead,
    // the shadow one batch ahead.
    int nin = 0;
    int j_a = lane < c ? a.nbr[row + lane] : 0;
    auto s_a = lane < c ? a.sh[j_a] : si;
    int j_b = lane + 32 < c ? a.nbr[row + lane + 32] : 0;
    for (int base = 0; base < c; base += 32) {
      const int slot = base + lane;
      const int j = j_a;
      const auto sj = s_a;
      j_a = j_b;
      if (slot + 32 < c) s_a = a.sh[j_a];
      j_b = slot + 64 < c ? a.nbr[row + slot + 64] : 0;
      bool in = false;
      R d[3] = {R(0), R(0), R(0)};
      if (slot < c) {
        pair_disp<R>(S, si, sj, a.off, row + slot, d);
        in = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] < a.rc2;
      }
      const unsigned mask = __ballot_sync(0xffffffffu, in);
      const int pos = nin + __popc(mask & lt_mask);   // < c <= rec
      if (in) {
        const auto rec = make_r4(d[0], d[1], d[2], pack_j(j, R(0)));
        a.list4[(size_t)q * a.rec + pos] = rec;
        if (pos < kListCap) *reinterpret_cast<typename V<R>::R4*>(&list[4 * pos]) = rec;
      }
      nin += __popc(mask);
    }
    if (lane == 0) a.nin[q] = nin;
    __syncwarp();   // also orders this warp's record stores before the reads of stage A

    // ---------------- stage A: G_klm = sum_j g_k Y_lm over the compacted neighbours,
    // then A = (1/N0) W . G and nu = 1, 2: E12 and dE12/dA
    R e = R(0), e_lo = R(0);   // the nu = 1, 2 energy, and what FP32 rounds off its C1
    if constexpr (sizeof(R) == 4) {
      // Tensor cores, 3xTF32: per k-step of 8 neighbours, D[lm][k] += Y^T[lm][j] g[j][k]
      // for two m-tiles of 16 (l, m) rows.  Each lane evaluates g and Y of one neighbour
      // and stores them as operand fragments; the accumulators end as G in fragment form.
      const int g8 = lane >> 2, t4 = lane & 3;
      float* ty = tile;
      float* tg = tile + 4 * kTyStep;
      float acc[2][4];
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[mt][u] = 0.f;
      // this lane's neighbour slot c of k-step ks: Y pairs (rows r, r + 8) go to the
      // fragment of lane (r % 8) * 4 + c % 4, elements 2 (c / 4) and 2 (c / 4) + 1; g_k
      // to lane k * 4 + c % 4, element c / 4
      const int pks = lane >> 3, pc = lane & 7;
      float* yb = ty + pks * kTyStep + (pc & 3) * 4 + (pc >> 2) * 2;
      float* gb = tg + pks * kTgStep + (pc & 3) * 2 + (pc >> 2);
      for (int base = 0; base < nin; base += 32) {
        const int slot = base + lane;
        float g[8], Y[25];
        if (slot < nin) {
          const auto en = slot < kListCap ? ld4<R>(&list[4 * slot]) : a.list4[(size_t)q * a.rec + slot];
          float r2 = en.x * en.x + en.y * en.y + en.z * en.z;
          float ir = rsqrt_(r2);
          radial<float>(r2 * ir, a.inv_rc, a.mode, g);
          sh_values<float>(en.x * ir, en.y * ir, en.z * ir, Y);
        } else {
#pragma unroll
          for (int k = 0; k < 8; ++k) g[k] = 0.f;
#pragma unroll
          for (int k = 0; k < 25; ++k) Y[k] = 0.f;
        }
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          *reinterpret_cast<float2*>(yb + r * 16) = make_float2(Y[r], Y[r + 8]);
          *reinterpret_cast<float2*>(yb + 128 + r * 16) = make_float2(Y[16 + r], r == 0 ? Y[24] : 0.f);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) gb[k * 8] = g[k];
        __syncwarp();
        const int nks = (min(32, nin - base) + 7) >> 3;
        for (int ks = 0; ks < nks; ++ks) {
          const float4 y0 = *reinterpret_cast<const float4*>(ty + ks * kTyStep + lane * 4);
          const float4 y1 = *reinterpret_cast<const float4*>(ty + ks * kTyStep + 128 + lane * 4);
          const float2 gg = *reinterpret_cast<const float2*>(tg + ks * kTgStep + lane * 2);
          uint32_t yh0[4], yl0[4], yh1[4], yl1[4], gh0, gl0, gh1, gl1;
          tf32_split(y0.x, yh0[0], yl0[0]);
          tf32_split(y0.y, yh0[1], yl0[1]);
          tf32_split(y0.z, yh0[2], yl0[2]);
          tf32_split(y0.w, yh0[3], yl0[3]);
          tf32_split(y1.x, yh1[0], yl1[0]);
          tf32_split(y1.y, yh1[1], yl1[1]);
          tf32_split(y1.z, yh1[2], yl1[2]);
          tf32_split(y1.w, yh1[3], yl1[3]);
          tf32_split(gg.x, gh0, gl0);
          tf32_split(gg.y, gh1, gl1);
          // each k-step's products from zero, summed into acc with round-to-nearest FP32
          // adds: the tensor core's own accumulation does not round to nearest, and 48
          // chained MMAs would bias G
          float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
          mma3(d0, yh0, yl0, gh0, gh1, gl0, gl1);
          mma3(d1, yh1, yl1, gh0, gh1, gl0, gl1);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            acc[0][u] += d0[u];
            acc[1][u] += d1[u];
          }
        }
        __syncwarp();
      }
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[mt][u] *= norm[2 * mt + (u >> 1)];
      // acc = G^T as fragments (rows lm, columns k); A = W G, then S = M2 A per l
      float am[2][4], sm[2][4];
      lm_mix(acc, Ws, g8, t4, am);
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int u = 0; u < 4; ++u) am[mt][u] *= a.inv_n0;
#pragma unroll
      for (int u = 0; u < 4; ++u) {   // the nu = 3 inputs: n <= 2, lm < 16 (tile 0)
        const int lm = g8 + 8 * (u >> 1), n = 2 * t4 + (u & 1);
        if (n < 3) a.a48[(size_t)q * 48 + n * 16 + lm] = am[0][u];
      }
      lm_mix(am, M2, g8, t4, sm);
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int lm = 16 * mt + g8 + 8 * (u >> 1), n = 2 * t4 + (u & 1);
          if (lm < 25) {
            const float lin = lm == 0 ? C1[n] : 0.f;
            e += am[mt][u] * (0.5f * sm[mt][u] + lin);
            // C1 to twice FP32's precision, in a sum of its own (e would round it off): its rounding
            // shifts every energy the same way, by half of the mean error of bulk atoms (E of
            // 255,840 atoms against FP64: mean 5.6e-6 -> 2.8e-6 eV, rms 2.84e-5 -> 2.80e-5 eV)
            if (lm == 0) e_lo += am[mt][u] * C1l[n];
            a.dA[(size_t)q * 200 + n * 25 + lm] = sm[mt][u] + lin;
          }
        }
      if (a.fs_on) {   // the same products with the phi^(2) coefficients
        lm_mix(am, M2b, g8, t4, sm);
        float eb = 0.f, eb_lo = 0.f;
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int lm = 16 * mt + g8 + 8 * (u >> 1), n = 2 * t4 + (u & 1);
            if (lm < 25) {
              const float lin = lm == 0 ? C1b[n] : 0.f;
              eb += am[mt][u] * (0.5f * sm[mt][u] + lin);
              if (lm == 0) eb_lo += am[mt][u] * C1bl[n];
              a.dAb[(size_t)q * 200 + n * 25 + lm] = sm[mt][u] + lin;
            }
          }
        const double Eb = warp_sum<double>((double)eb + (double)eb_lo);
        if (lane == 0) a.e12b[q] = Eb;
      }
    } else {
      // FP64: SIMT, G = g^T Y with 4-wide vector loads along the neighbour axis
      R* A = tile;
      R* Gs = tile + 600;
      R acc[7];
#pragma unroll
      for (int t = 0; t < 7; ++t) acc[t] = R(0);
      for (int base = 0; base < nin; base += 32) {
        const int slot = base + lane;
        R g[8], Y[25];
        if (slot < nin) {
          const auto en = slot < kListCap ? ld4<R>(&list[4 * slot]) : a.list4[(size_t)q * a.rec + slot];
          R r2 = en.x * en.x + en.y * en.y + en.z * en.z;
          R ir = rsqrt_(r2);
          radial<R>(r2 * ir, a.inv_rc, a.mode, g);
          sh_values<R>(en.x * ir, en.y * ir, en.z * ir, Y);
        } else {
#pragma unroll
          for (int k = 0; k < 8; ++k) g[k] = R(0);
#pragma unroll
          for (int k = 0; k < 25; ++k) Y[k] = R(0);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) tile[k * kCols + lane] = g[k];
#pragma unroll
        for (int k = 0; k < 25; ++k) tile[(8 + k) * kCols + lane] = Y[k];
        __syncwarp();
        const int nv = min(32, nin - base);
        for (int s4 = 0; s4 < (nv + 3) / 4; ++s4) {
          auto g4 = ld4<R>(&tile[kq * kCols + 4 * s4]);
#pragma unroll
          for (int t = 0; t < 7; ++t) {
            const int lm = grp + 4 * t;
            if (lm < 25) {
              auto y4 = ld4<R>(&tile[(8 + lm) * kCols + 4 * s4]);
              acc[t] += g4.x * y4.x + g4.y * y4.y + g4.z * y4.z + g4.w * y4.w;
            }
          }
        }
        __syncwarp();
      }
#pragma unroll
      for (int t = 0; t < 7; ++t) {
        const int lm = grp + 4 * t;
        if (lm < 25) Gs[kq * 25 + lm] = acc[t] * norm[t];
      }
      __syncwarp();
      for (int o = lane; o < 200; o += 32) {
        const int n = o / 25, lm = o - 25 * n, l = l_of(lm);
        const R* w = &Ws[(l * 8 + n) * 8];
        R s = R(0);
#pragma unroll
        for (int k = 0; k < 8; ++k) s += w[k] * Gs[k * 25 + lm];
        A[o] = s * a.inv_n0;
      }
      __syncwarp();
      for (int v = lane; v < 48; v += 32) a.a48[(size_t)q * 48 + v] = A[(v >> 4) * 25 + (v & 15)];
      for (int o = lane; o < 200; o += 32) {
        const int n = o / 25, lm = o - 25 * n, l = l_of(lm);
        const R* mrow = &M2[l * 64 + n * 8];
        R s = R(0);
#pragma unroll
        for (int n2 = 0; n2 < 8; ++n2) s += mrow[n2] * A[n2 * 25 + lm];
        const R lin = lm == 0 ? C1[n] : R(0);
        e += A[o] * (R(0.5) * s + lin);
        a.dA[(size_t)q * 200 + o] = s + lin;
      }
      if (a.fs_on) {   // the same products with the phi^(2) coefficients
        R eb = R(0);
        for (int o = lane; o < 200; o += 32) {
          const int n = o / 25, lm = o - 25 * n, l = l_of(lm);
          const R* mrow = &M2b[l * 64 + n * 8];
          R sb = R(0);
#pragma unroll
          for (int n2 = 0; n2 < 8; ++n2) sb += mrow[n2] * A[n2 * 25 + lm];
          const R lin = lm == 0 ? C1b[n] : R(0);
          eb += A[o] * (R(0.5) * sb + lin);
          a.dAb[(size_t)q * 200 + o] = sb + lin;
        }
        const double Eb = warp_sum<double>((double)eb);
        if (lane == 0) a.e12b[q] = Eb;
      }
    }
    const double E = warp_sum<double>((double)e + (double)e_lo);
    if (lane == 0) a.e12[q] = E;
    cnt_pairs += nin;
    cnt_atoms += 1;
    // tensor-core tiles: 6 per k-step of 8 neighbours, 15 per lm_mix
    if (sizeof(R) == 4) cnt_mma += 6 * ((nin + 7) / 8) + (a.fs_on ? 45 : 30);
    __syncwarp();
  }
  if (lane == 0 && cnt_atoms > 0) {   // the warp's counts, added once
    atomicAdd(&a.stats->ace_pairs, cnt_pairs);
    atomicAdd(&a.stats->ace_atoms, cnt_atoms);
    if (sizeof(R) == 4) atomicAdd(&a.stats->ace_mma, cnt_mma);
  }
}

// Energies alone: E_i = E12 + E3 (+ F), one thread per precise atom.
template <typename R, bool FS>
__global__ void k_ace_energy(AceArgs<R> a) {
  const int m = *a.count;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < m; q += gridDim.x * blockDim.x)
    a.e_prec[a.queue[q]] = a.e12[q] + a.e3[q] + (FS ? a.fs[2 * (size_t)q] : 0.0);
}

// Kernel 3, L lanes per precise atom: E_i = E12 + E3 -> e_prec, then
// u_klm = (1/N0) sum_n W[l][n][k] dE/dA_nlm (times N_lm, in the order of pair_force), and the
// pair forces: each lane takes every L-th record of its atom, scatters -w_i p_ij to neighbour
// j, and +w_i sum_j p_ij goes to i.  Persistent warps: every warp starts at its own position
// (block-major, so short queues spread over all SMs) and continues by an atomic work counter.
// L = 8 fills 98 % of the lanes with the about 134 neighbours of a bulk atom, L = 32 84 % of
// 5 turns, but short queues need the warps (adjoint_lanes has the figures).
template <typename R, bool FS, int L>
__global__ void __launch_bounds__(kWarps3<R> * 32, sizeof(R) == 4 ? AP_ACE3_MINB : 1) k_ace_adjoint(AceArgs<R> a) {
  constexpr int NA = 32 / L;   // atoms per warp
  // Shared memory: W [320] | per warp: dA [NA][200] | U [NA][200]
  extern __shared__ __align__(128) unsigned char smem_raw[];
  R* Ws = reinterpret_cast<R*>(smem_raw);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  R* dA = Ws + 320 + warp * (400 * NA);
  R* U = dA + 200 * NA;
  for (int t = threadIdx.x; t < 320; t += blockDim.x) Ws[t] = a.W[t];
  __syncthreads();
  const int m = *a.count;
  const int g = lane / L, sub = lane & (L - 1);
  const int q_first = NA * (warp * gridDim.x + blockIdx.x), q_all = NA * kWarps3<R> * gridDim.x;
  for (int q0 = q_first; q0 < m; q0 = next_item(a.counter2, NA, q_all)) {
    const int q = q0 + g;
    const bool on = q < m;
    const int i = on ? a.queue[q] : 0;
    if (on && sub == 0) a.e_prec[i] = a.e12[q] + a.e3[q] + (FS ? a.fs[2 * (size_t)q] : 0.0);
    const int na = min(NA, m - q0);
    for (int t = 0; t < na; ++t) {
      const size_t qt = (size_t)(q0 + t);
      R* dst = dA + 200 * t;
      const R fp = FS ? (R)a.fs[2 * qt + 1] : R(0);
      for (int o = lane; o < 200; o += 32) {
        const int n = o / 25, lm = o - 25 * n;
        R v = a.dA[qt * 200 + o];
        if (FS) v = fma(fp, a.dAb[qt * 200 + o], v);
        if (n < 3 && lm < 16) v += a.de3[qt * 48 + n * 16 + lm];
        dst[o] = v;
      }
    }
    __syncwarp();
    for (int o = lane; o < 200; o += 32) {
      const int lm = o >> 3, k = o & 7, l = l_of(lm);
      const R nrm = (R)kNorm[lm] * a.inv_n0;
      R* dst = U + kSlot[lm] * 8 + k;
      for (int t = 0; t < na; ++t) {
        R s = R(0);
#pragma unroll
        for (int n = 0; n < 8; ++n) s = fma(Ws[(l * 8 + n) * 8 + k], dA[200 * t + n * 25 + lm], s);
        dst[200 * t] = s * nrm;
      }
    }
    __syncwarp();
    const int nin = on ? a.nin[q] : 0;
    const R wgt = on ? (R)(a.wgt ? a.wgt[i] : 1.0 - (a.lam ? a.lam[i] : 0.0)) : R(0);
    R pix = R(0), piy = R(0), piz = R(0);
    // the pair records kernel 1 kept (displacement and j), the lane's next one loaded a turn ahead
    const typename V<R>::R4* lst = a.list4 + (size_t)q * a.rec;
    typename V<R>::R4 e_n = make_r4(R(0), R(0), R(0), R(0));
    if (sub < nin) e_n = lst[sub];
    for (int slot = sub; slot < nin; slot += L) {
      const auto e = e_n;
      if (slot + L < nin) e_n = lst[slot + L];
      const int j = unpack_j(e.w);
      const R r2 = e.x * e.x + e.y * e.y + e.z * e.z;
      const R ir = rsqrt_(r2);
      R px, py, pz;
      pair_force<R>(U + 200 * g, e.x * ir, e.y * ir, e.z * ir, r2 * ir, ir, a.inv_rc, a.mode, px, py, pz);
      pix += px;
      piy += py;
      piz += pz;
      add_force<R>(a.facc32, a.facc64, a.faccfix, j, -wgt * px, -wgt * py, -wgt * pz);
    }
    __syncwarp();
    pix = lane_sum<R, L>(pix);
    piy = lane_sum<R, L>(piy);
    piz = lane_sum<R, L>(piz);
    if (on && sub == 0) add_force<R>(a.facc32, a.facc64, a.faccfix, i, wgt * pix, wgt * piy, wgt * piz);
    __syncwarp();
  }
}

// The accumulated ACE forces join f and the accumulators are cleared for the next evaluation
// (most atoms have no precise atom in reach and need neither).
__global__ void k_ace_finalize32(int n, float4* __restrict__ acc, double* __restrict__ f) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float4 v = acc[i];
  if (v.x == 0.f && v.y == 0.f && v.z == 0.f) return;
  acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  f[3 * i + 0] += (double)v.x;
  f[3 * i + 1] += (double)v.y;
  f[3 * i + 2] += (double)v.z;
}

__global__ void k_ace_finalize_fix(int n, unsigned long long* __restrict__ acc, double* __restrict__ f) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 3 * n) return;
  const long long v = (long long)acc[i];
  if (v == 0) return;
  acc[i] = 0;
  f[i] += (double)v * (1.0 / kFixScale);
}

__global__ void k_ace_finalize64(int n, double* __restrict__ acc, double* __restrict__ f) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 3 * n) return;
  const double v = acc[i];
  if (v == 0.0) return;
  acc[i] = 0.0;
  f[i] += v;
}

template <typename R>
size_t basis_smem() {
  return sizeof(R) * (320 + 320 + 8 + 320 + 3 * 8) + sizeof(R) * kWarps<R> * (4 * kListCap + kTileWords<R>);
}

template <typename R>
size_t adjoint_smem(int lanes) {
  return sizeof(R) * (320 + kWarps3<R> * 400 * (32 / lanes));
}

// Grid of a persistent kernel over `items` (one warp each) with up to `resident` blocks per SM:
// a whole number of blocks per SM, no more than the items need.
inline int persistent_grid(int num_sms, int resident, int warps, int64_t items) {
  const int64_t per_sm = (items + (int64_t)num_sms * warps - 1) / ((int64_t)num_sms * warps);
  return num_sms * (int)std::max<int64_t>(1, std::min<int64_t>(resident, per_sm));
}

// Lanes per atom of the adjoint for a queue of m atoms: 8 where that still fills every SM
// (FP32: all 24 resident warps twice; FP64: 4 warps per scheduler), a whole warp otherwise.
// Whole force evaluations, 8 against 32 lanes: FP32 3.62 / 3.77 ms (255,840 atoms), 57.8 / 60.0 ms
// (10 steps with 240,000), 3.17 / 3.09 ms (10 steps with 12,700); FP64 4.60 / 4.75 ms (12,700
// atoms), 2.29 / 2.19 ms (energy and gradient, 1,365).
template <typename R>
inline int adjoint_lanes(int num_sms, int64_t m) {
  return m >= (int64_t)num_sms * (sizeof(R) == 4 ? 192 : 64) ? 8 : 32;
}

template <typename K>
int resident_blocks(K kern, int threads, size_t smem) {
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int b = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, threads, smem);
  return b > 0 ? b : 1;
}

template <typename R>
void run_ace(ap_ctx* c, const double* d_lam, const double* d_wgt, const int* d_queue, const int* d_count,
             double* d_e_prec, bool forces, cudaStream_t s) {
  AceArgs<R> a;
  a.queue = d_queue;
  a.count = d_count ? d_count : &c->d_sc->n_precise;
  a.stats = c->d_sc;
  a.counter = &c->d_sc->work_counter;
  a.counter2 = &c->d_sc->work_counter2;
  a.sys = c->d_sys;
  a.atom_sys = c->d_atom_sys;
  if constexpr (sizeof(R) == 4) {
    a.sh = c->d_sh32;
    a.W = c->d_W32;
    a.facc32 = c->d_facc32;
    a.facc64 = nullptr;
  } else {
    a.sh = c->d_sh64;
    a.W = c->d_W64;
    a.facc32 = nullptr;
    a.facc64 = c->d_facc64;
  }
  a.nbr = c->d_nbr_ace;
  a.off = c->stored_off ? c->d_off_ace : nullptr;
  a.cnt = c->d_cnt_ace;
  a.cap = c->cap_ace;
  a.lam = d_lam;
  a.wgt = d_wgt;
  a.faccfix = c->cfg.ace_deterministic ? c->d_faccfix : nullptr;
  a.M2 = a.W + 320;   // the parameter block is [W (320) | M2 (320) | C1 (8) | M2b (320) | C1b (8) | C1l (16)]
  a.C1 = a.W + 640;
  a.M2b = a.W + 648;
  a.C1b = a.W + 968;
  a.C1l = a.W + 976;
  a.fs_on = c->cfg.ace_fs_on;
  a.fs_eps = c->cfg.ace_fs_eps;
  a.dAb = reinterpret_cast<R*>(c->d_ace_dAb);
  a.e12b = c->d_ace_e12b;
  a.fs = c->d_ace_fs;
  a.rc2 = (R)(c->cfg.ace_rc * c->cfg.ace_rc);
  a.inv_rc = (R)(1.0 / c->cfg.ace_rc);
  a.inv_n0 = (R)(1.0 / c->cfg.ace_n0);
  a.mode = c->cfg.fcut_mode;
  a.e_prec = d_e_prec;
  a.list4 = reinterpret_cast<typename V<R>::R4*>(c->d_ace_list);
  a.rec = c->ace_rec_cap;
  a.nin = c->d_ace_nin;
  a.a48 = reinterpret_cast<R*>(c->d_ace_a48);
  a.dA = reinterpret_cast<R*>(c->d_ace_dA);
  a.e12 = c->d_ace_e12;
  a.de3 = reinterpret_cast<R*>(c->d_ace_de3);
  a.e3 = c->d_ace_e3;
  const bool fs = c->cfg.ace_fs_on != 0;

  const int pi = sizeof(R) == 4 ? 0 : 1;
  // the queue's length as of the last synchronisation (its rows were built after it): sizes the
  // grids only, the kernels read the device's own count
  int m = 0;
  std::memcpy(&m, (const char*)c->h_sc + ((const char*)a.count - (const char*)c->d_sc), sizeof(int));
  const int lanes = adjoint_lanes<R>(c->num_sms, m);
  static int b1[2] = {0, 0}, b3[2][2][2] = {};
  const size_t s1 = basis_smem<R>(), s3 = adjoint_smem<R>(lanes);
  if (!b1[pi]) b1[pi] = resident_blocks(k_ace_basis<R>, kWarps<R> * 32, s1);
  auto k3 = lanes == 8 ? (fs ? k_ace_adjoint<R, true, 8> : k_ace_adjoint<R, false, 8>)
                       : (fs ? k_ace_adjoint<R, true, 32> : k_ace_adjoint<R, false, 32>);
  int& r3 = b3[pi][lanes == 8][fs];
  if (forces && !r3) r3 = resident_blocks(k3, kWarps3<R> * 32, s3);
  const int tb = prof_mark(c, s);
  k_ace_basis<R><<<persistent_grid(c->num_sms, b1[pi], kWarps<R>, m), kWarps<R> * 32, s1, s>>>(a);
  prof_add(c, AP_PHASE_ACE_BASIS, tb, prof_mark(c, s));
  c->kernels += launch_ace_nu3<R>(c, a, m, s);
  c->kernels += 2;
  if (!forces) {
    auto ke = fs ? k_ace_energy<R, true> : k_ace_energy<R, false>;
    ke<<<std::max(1, std::min(c->num_sms * 8, (m + 127) / 128)), 128, 0, s>>>(a);
    return;
  }
  const int t0 = prof_mark(c, s);
  k3<<<persistent_grid(c->num_sms, r3, kWarps3<R>, ((int64_t)m * lanes + 31) / 32), kWarps3<R> * 32, s3, s>>>(a);
  prof_add(c, AP_PHASE_ACE_ADJOINT, t0, prof_mark(c, s));
}

}  // namespace

void upload_ace_tables(ap_ctx* c) {
  const AceTables& t = c->ace;
  std::vector<double> p64(c->cfg.ace_W, c->cfg.ace_W + 320);
  p64.insert(p64.end(), t.m2.begin(), t.m2.end());
  p64.insert(p64.end(), t.c1.begin(), t.c1.end());
  p64.insert(p64.end(), t.m2b.begin(), t.m2b.end());
  p64.insert(p64.end(), t.c1b.begin(), t.c1b.end());
  std::vector<float> p32(p64.begin(), p64.end());
  for (const auto* c1 : {&t.c1, &t.c1b})   // the rest of C1 and C1b beyond FP32
    for (double v : *c1) {
      p64.push_back(0.0);
      p32.push_back((float)(v - (double)(float)v));
    }
  cudaMalloc(&c->d_W32, sizeof(float) * p32.size());
  cudaMalloc(&c->d_W64, sizeof(double) * p64.size());
  cudaMemcpy(c->d_W32, p32.data(), sizeof(float) * p32.size(), cudaMemcpyHostToDevice);
  cudaMemcpy(c->d_W64, p64.data(), sizeof(double) * p64.size(), cudaMemcpyHostToDevice);
}

void launch_ace(ap_ctx* c, const double* d_lam, const int* d_queue, double* d_e_prec, bool forces, cudaStream_t s,
                const double* d_wgt, const int* d_count) {
  if (c->cfg.precision == AP_PREC_FP64)
    run_ace<double>(c, d_lam, d_wgt, d_queue, d_count, d_e_prec, forces, s);
  else
    run_ace<float>(c, d_lam, d_wgt, d_queue, d_count, d_e_prec, forces, s);
}

void launch_ace_finalize(ap_ctx* c, double* d_f, cudaStream_t s) {
  c->kernels += 1;
  if (c->cfg.ace_deterministic)
    k_ace_finalize_fix<<<(int)((3 * c->n + 255) / 256), 256, 0, s>>>((int)c->n, c->d_faccfix, d_f);
  else if (c->cfg.precision == AP_PREC_FP64)
    k_ace_finalize64<<<(int)((3 * c->n + 255) / 256), 256, 0, s>>>((int)c->n, c->d_facc64, d_f);
  else
    k_ace_finalize32<<<(int)((c->n + 255) / 256), 256, 0, s>>>((int)c->n, c->d_facc32, d_f);
}

}  // namespace ap
