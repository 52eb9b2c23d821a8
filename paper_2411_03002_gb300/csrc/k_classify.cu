// Precision classification (Appendix A and B): centro-symmetry parameter,
// moving averages, lambda_0, lambda_min spread, minimum-step hysteresis and the
// compacted precise-atom work queue.  Every value that decides a set is computed
// in FP64 with explicit round-to-nearest operations in the order of the
// definitions, so the detected and precise sets are reproducible bit for bit.
// FP32 is used only to pick candidates, with a guard band and an exact fallback.
#include "eam_frame.cuh"

namespace ap {

namespace {

constexpr float kBand = 1e-3f;     // FP32 guard band (A^2) on squared lengths
constexpr int kNN = 12;            // N nearest neighbours of FCC (N_buffer = 0)
constexpr int kHalf = kNN / 2;

__device__ inline const SysInfo& sys_of(const SysInfo* sys, const int* atom_sys, int i) {
  return sys[atom_sys ? atom_sys[i] : 0];
}
__device__ inline int floor_div(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

// f_cut of Appendix B in FP64 with the oracle's operation order.
__device__ inline double fcut_exact(double x, int mode) {
  if (x < 0.0) return 1.0;
  if (x > 1.0) return 0.0;
  double t = x;
  if (mode == 1) t = __dsub_rn(__dmul_rn(2.0, x), 1.0);
  double t2 = __dmul_rn(t, t);
  double t3 = __dmul_rn(t2, t);
  double t5 = __dmul_rn(t3, t2);
  double p = __dsub_rn(__dadd_rn(__dsub_rn(1.0, __dmul_rn(1.875, t)), __dmul_rn(1.25, t3)), __dmul_rn(0.375, t5));
  if (mode == 1) p = __dmul_rn(0.5, p);
  return p;
}

// f_cut in FP32, used only to screen candidates.
__device__ inline float fcut_f(float x, int mode) {
  if (x < 0.f) return 1.f;
  if (x > 1.f) return 0.f;
  const float t = mode == 1 ? 2.f * x - 1.f : x;
  const float t2 = t * t;
  const float p = 1.f - 1.875f * t + 1.25f * t2 * t - 0.375f * t2 * t2 * t;
  return mode == 1 ? 0.5f * p : p;
}

// Cell offset k of a row entry.
__device__ inline void entry_offset(const int* off, size_t e, const SysInfo& S, int wi, int wj, int k[3]) {
  if (off) {
    int p = off[e];
    k[0] = off_x(p);
    k[1] = off_y(p);
    k[2] = off_z(p);
  } else {
    k[0] = wrap_off(cell_x(wj) - cell_x(wi), S.nc[0], S.periodic[0]);
    k[1] = wrap_off(cell_y(wj) - cell_y(wi), S.nc[1], S.periodic[1]);
    k[2] = wrap_off(cell_z(wj) - cell_z(wi), S.nc[2], S.periodic[2]);
  }
}

// Exact displacement (x_j + S L) - x_i for a row entry with cell offset k.
__device__ inline void exact_disp(const double* __restrict__ x, const SysInfo& S, int i, int j, const int4& ci,
                                  const int4& cj, const int k[3], double d[3]) {
  int cu_i[3] = {ci.x, ci.y, ci.z}, cu_j[3] = {cj.x, cj.y, cj.z};
  for (int a = 0; a < 3; ++a) {
    // whole periods between the pair's cell offset and its unwrapped cells (the integer
    // division only where they differ)
    const int t = k[a] - (cu_j[a] - cu_i[a]);
    const int sd = (S.periodic[a] && t != 0) ? t / S.nc[a] : 0;
    // x_j + 0 L is x_j exactly: the FP64 multiply-add (slow on this GPU) only for images
    double shifted = sd == 0 ? x[3 * j + a] : __dadd_rn(x[3 * j + a], __dmul_rn((double)sd, S.L[a]));
    d[a] = __dsub_rn(shifted, x[3 * i + a]);
  }
}

__device__ inline double norm2_exact(const double d[3]) {
  return __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
}

// Candidate order (r^2, j, s) of the definition.
__device__ inline bool cand_less(double ra, int ja, const int* sa, double rb, int jb, const int* sb) {
  if (ra != rb) return ra < rb;
  if (ja != jb) return ja < jb;
  for (int a = 0; a < 3; ++a)
    if (sa[a] != sb[a]) return sa[a] < sb[a];
  return false;
}

__device__ inline void image_of(const SysInfo& S, const int4& ci, const int4& cj, const int k[3], int s[3]) {
  int cu_i[3] = {ci.x, ci.y, ci.z}, cu_j[3] = {cj.x, cj.y, cj.z};
  for (int a = 0; a < 3; ++a) {
    const int t = k[a] - (cu_j[a] - cu_i[a]);
    s[a] = (S.periodic[a] && t != 0) ? t / S.nc[a] : 0;
  }
}

// Row position q of atom i's entry -> exact FP64 displacement.
__device__ inline void exact_entry(const double* __restrict__ x, const SysInfo& S, int i, const int4& ci,
                                   const int* __restrict__ nbr, const int* __restrict__ off,
                                   const int4* __restrict__ cunw, size_t row, int q, double d[3], int& j,
                                   int s[3]) {
  j = nbr[row + q];
  const int4 cj = cunw[j];
  int k[3];
  entry_offset(off, row + q, S, ci.w, cj.w, k);
  exact_disp(x, S, i, j, ci, cj, k, d);
  image_of(S, ci, cj, k, s);
}

// (r2, j, s) ordering of two row entries with equal or different exact r2.
__device__ inline bool entry_less(const double* __restrict__ x, const SysInfo& S, int i, const int4& ci,
                                  const int* __restrict__ nbr, const int* __restrict__ off,
                                  const int4* __restrict__ cunw, size_t row, double ra, int qa, double rb, int qb) {
  if (ra != rb) return ra < rb;
  if (qb < 0) return true;
  double d[3];
  int ja, jb, sa[3], sb[3];
  exact_entry(x, S, i, ci, nbr, off, cunw, row, qa, d, ja, sa);
  exact_entry(x, S, i, ci, nbr, off, cunw, row, qb, d, jb, sb);
  return cand_less(ra, ja, sa, rb, jb, sb);
}

// Ascending FP64 sum of the six pair values (non-negative: their bit patterns order them, in
// integer instructions).
__device__ inline double sum_ascending(double v[kHalf]) {
#pragma unroll
  for (int a = 1; a < kHalf; ++a)
#pragma unroll
    for (int p = a; p > 0; --p)
      if (__double_as_longlong(v[p]) < __double_as_longlong(v[p - 1])) {
        const double t = v[p];
        v[p] = v[p - 1];
        v[p - 1] = t;
      }
  double sum = v[0];
#pragma unroll
  for (int a = 1; a < kHalf; ++a) sum = __dadd_rn(sum, v[a]);
  return sum;
}

// ------------------------------------------------------------------ CSP
// Three kernels share the atoms (launch_csp):
//   k_csp_near   one thread per atom: the 12 nearest and the six smallest pair values found by
//                thresholds, without sorting; in a crystal they stand apart.  Atoms where they
//                do not (surfaces, defects, strong disorder) are handed on.
//   k_csp_sort   one thread per atom: sorted FP32 selections (insertion), for long lists only;
//                what FP32 cannot decide is handed on again.
//   k_csp_exact  one warp per atom, exact selections: what is left, short lists, small systems.
// Structures without shells (a melt, a gas) take all three: updates of a gas of 50,000 / 100,000 /
// 200,000 / 1,000,000 atoms 0.43 / 0.60 / 0.93 / 3.73 ms, where a sorting kernel for all atoms and a
// thread for each of the rest took 0.92 / 0.97 / 1.32 / 3.71 ms.
// FP64 arithmetic issues one warp instruction per 16 cycles and SM: a warp per atom for all
// atoms would take 4 ms on 4,000,000 of them, the 89 FP64 operations of a thread 0.57 ms.

struct CspArgs {
  int n;
  const double* x;
  const uint8_t* ch;
  const SysInfo* sys;
  const int* atom_sys;
  const float4* s32;
  const int4* cunw;
  const int* nbr;
  const int* off;
  const int* cnt;
  int cap;
  float rsf2;
  double rs2;
  double* csp;
  const int* nin;
  float rpf2, stale2;
  int* n_stale;
};

// CSP of atom i by sorted FP32 selections; what FP32 cannot decide (an r_search band hit, an
// ambiguous 12/13 or 6/7 boundary) is appended to `slow`.  All selection arrays are indexed with
// compile-time indices (fully unrolled insertion), so they live in registers.  Rows four entries at
// a time, and no exit but the end: with returns out of the loops the lanes of a warp, which go
// on to the next atom here, no longer met again in the loops (1,000,000 atoms of a gas 10.5 ms,
// 1.2 ms like this).
// With A.nin (rows built at these positions) the row's first nin[i] entries are the ones inside
// r_c^2 = rpf2 at the build (FP32), the rest lie beyond it: when the 13th smallest r^2 of that part
// lies more than two guard bands inside rpf2, the skin part is skipped.  128-thread blocks: the
// shared arrays are indexed by threadIdx.x.
template <bool VEC>
__device__ __forceinline__ void csp_atom(const CspArgs& A, int i, int* __restrict__ slow, int* __restrict__ n_slow) {
  const SysInfo& S = sys_of(A.sys, A.atom_sys, i);
  const float4 si = A.s32[i];
  const int wi = __float_as_int(si.w);
  const int c = A.cnt[i];
  const size_t row = (size_t)i * A.cap;
  const float rsf2 = A.rsf2;

  // 1. the 13 smallest FP32 r^2 among candidates inside r_search
  float tr[kNN + 1];
  int tq[kNN + 1];
#pragma unroll
  for (int a = 0; a <= kNN; ++a) {
    tr[a] = INFINITY;
    tq[a] = -1;
  }
  int n_in = 0;
  bool ok = true;
  int q_end = A.nin ? A.nin[i] : c;
  if (q_end == 0) q_end = c;
  const int* const rowp = A.nbr + row;
  int4 next = c > 0 ? row4<VEC>(rowp, 0, c) : make_int4(0, 0, 0, 0);
  for (int q0 = 0; q0 < q_end; q0 += 4) {
    // four entries at a time, the next four indices loaded ahead of their use
    const int4 jj = next;
    float4 sv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) sv[u] = A.s32[q0 + u < c ? pick(jj, u) : i];
    if (q0 + 4 < c) next = row4<VEC>(rowp, q0 + 4, c);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int q = q0 + u;
      const float4 sj = sv[u];
      int k[3];
      entry_offset(A.off, row + min(q, c - 1), S, wi, __float_as_int(sj.w), k);
      const float dx = (float)k[0] * S.hf[0] + sj.x - si.x;
      const float dy = (float)k[1] * S.hf[1] + sj.y - si.y;
      const float dz = (float)k[2] * S.hf[2] + sj.z - si.z;
      const float r2 = dx * dx + dy * dy + dz * dz;
      const bool in = q < c && r2 <= rsf2 + kBand;
      ok = ok && !(in && r2 >= rsf2 - kBand);
      n_in += in ? 1 : 0;
      if (in && r2 < tr[kNN]) {
        tr[kNN] = r2;
        tq[kNN] = q;
#pragma unroll
        for (int p = kNN; p > 0; --p) {
          const bool sw = tr[p] < tr[p - 1];
          const float lo = fminf(tr[p], tr[p - 1]), hi = fmaxf(tr[p], tr[p - 1]);
          const int ul = sw ? tq[p] : tq[p - 1], uh = sw ? tq[p - 1] : tq[p];
          tr[p - 1] = lo;
          tr[p] = hi;
          tq[p - 1] = ul;
          tq[p] = uh;
        }
      }
    }
    // the in-range part may end within a group of four: the entries after it only make the
    // selection more complete
    if (q0 + 4 >= q_end && q_end < c && !(tr[kNN] + 2.f * kBand < A.rpf2)) q_end = c;
  }
  // Rows older than the positions (stale2 > 0): every atom outside the row lies beyond
  // r_search - 2 m (m the largest displacement since the build), stale2 = that radius
  // squared.  The row's selection is exact when 12 candidates lie inside it with a
  // guard band; otherwise (a nearly isolated atom) the atom is counted and the caller
  // rebuilds the rows and computes the CSP again.
  if (A.stale2 > 0.f && ok && !(n_in >= kNN && tr[kNN - 1] + 2.f * kBand < A.stale2)) atomicAdd(A.n_stale, 1);
  const bool few = n_in < kNN;
  // 2. FP32 decides the 12 nearest unless the 12/13 boundary lies within the guard band
  ok = ok && (few || !(n_in > kNN && tr[kNN] - tr[kNN - 1] <= 2.f * kBand));
  // 3. FP32 vectors of the 12 and the 7 smallest pair values |r_a + r_b|^2.  The 12
  // vectors and row positions live in shared memory, component-major (thread index
  // fastest, conflict-free), not in registers.
  __shared__ float s_v[3][kNN][128];
  __shared__ int s_tq[kNN][128];
  const int tx = threadIdx.x;
  double sum = INFINITY;
  if (ok && !few) {
#pragma unroll
    for (int a = 0; a < kNN; ++a) {
      const int q = tq[a];
      s_tq[a][tx] = q;
      const int j = A.nbr[row + q];
      const float4 sj = A.s32[j];
      int k[3];
      entry_offset(A.off, row + q, S, wi, __float_as_int(sj.w), k);
      s_v[0][a][tx] = (float)k[0] * S.hf[0] + sj.x - si.x;
      s_v[1][a][tx] = (float)k[1] * S.hf[1] + sj.y - si.y;
      s_v[2][a][tx] = (float)k[2] * S.hf[2] + sj.z - si.z;
    }
    float pv[kHalf + 1];
    int pc[kHalf + 1];   // neighbour slots a | b << 8
#pragma unroll
    for (int a = 0; a <= kHalf; ++a) {
      pv[a] = INFINITY;
      pc[a] = 0;
    }
#pragma unroll 1
    for (int a = 0; a < kNN - 1; ++a) {
      const float ax = s_v[0][a][tx], ay = s_v[1][a][tx], az = s_v[2][a][tx];
#pragma unroll 1
      for (int b = a + 1; b < kNN; ++b) {
        const float sx = ax + s_v[0][b][tx], sy = ay + s_v[1][b][tx], sz = az + s_v[2][b][tx];
        const float v = sx * sx + sy * sy + sz * sz;
        if (v < pv[kHalf]) {
          pv[kHalf] = v;
          pc[kHalf] = a | (b << 8);
#pragma unroll
          for (int p = kHalf; p > 0; --p) {
            const bool sw = pv[p] < pv[p - 1];
            const float lo = fminf(pv[p], pv[p - 1]), hi = fmaxf(pv[p], pv[p - 1]);
            const int ul = sw ? pc[p] : pc[p - 1], uh = sw ? pc[p - 1] : pc[p];
            pv[p - 1] = lo;
            pv[p] = hi;
            pc[p - 1] = ul;
            pc[p] = uh;
          }
        }
      }
    }
    // 4. exact values of the six smallest pairs, unless the 6/7 boundary is ambiguous
    ok = pv[kHalf] - pv[kHalf - 1] > 2.f * kBand;
    if (ok) {
      const int4 ci = A.cunw[i];
      double chosen[kHalf];
#pragma unroll
      for (int t = 0; t < kHalf; ++t) {
        double da[3], db[3];
        int ja, jb, sa[3], sb[3];
        exact_entry(A.x, S, i, ci, A.nbr, A.off, A.cunw, row, s_tq[pc[t] & 0xff][tx], da, ja, sa);
        exact_entry(A.x, S, i, ci, A.nbr, A.off, A.cunw, row, s_tq[pc[t] >> 8][tx], db, jb, sb);
        const double s3[3] = {__dadd_rn(da[0], db[0]), __dadd_rn(da[1], db[1]), __dadd_rn(da[2], db[2])};
        chosen[t] = norm2_exact(s3);
      }
      sum = sum_ascending(chosen);
    }
  }
  if (ok) A.csp[i] = sum;
  else slow[atomicAdd(n_slow, 1)] = i;
}

// Atoms per SM on k_csp_near's list up to which k_csp_exact takes them all.  A warp each takes 6 ns
// an atom, the sort 75 us and 2.5 ns an atom; whole updates, sorted and by warps: a gas of 15,000
// atoms 334 and 320 us, 20,000 355 and 347, 25,000 364 and 382, 40,000 404 and 475; 255,840 atoms
// of disordered crystals with 15,500 on the list 975 and 965 us, with 39,000 1,076 and 1,157.
constexpr int kSortFrom = 140;
constexpr int kSortBlocks = 5;   // resident blocks of k_csp_sort per SM (92 registers)

template <bool VEC>
__global__ void __launch_bounds__(128) k_csp_sort(const CspArgs A, const int* __restrict__ list,
                                                  const int* __restrict__ n_list, int* __restrict__ slow,
                                                  int* __restrict__ n_slow, int sort_from) {
  const int m = *n_list;
  if (m <= sort_from) return;
  for (int t0 = blockIdx.x * blockDim.x; t0 < m; t0 += gridDim.x * blockDim.x) {
    if (t0 + threadIdx.x < m) csp_atom<VEC>(A, list[t0 + threadIdx.x], slow, n_slow);
    __syncwarp();
  }
}

// Thread per atom, FP32 screening by thresholds.  The number of entries walked gives the density
// and that the first shell's r^2 in an FCC crystal, r1^2 = R^2 (4 sqrt(2) pi/3 / N)^(2/3).  Entries
// below 1.6 r1^2 go to a short list in shared memory; a threshold (1.6 r1^2 or a little less)
// that leaves exactly 12 of them is looked for (the second shell lies at twice the first one's
// r^2), and the next entry must lie more than two guard bands further out.  Likewise the six
// pairs below r1^2/4 (opposite neighbours; other pairs leave about r1^2 or more), if they are six
// and stand apart.  Sorting networks over 13 entries and 7 pairs, which this replaces for the
// atoms of a crystal, were 4 of 5 instructions: 4,000,000 atoms 2.74 -> 1.44 ms,
// and 0.25 ms less for the exact selections.
constexpr int kNear = 24;
#ifndef AP_CSP_MINB
#define AP_CSP_MINB 8   // resident blocks per SM k_csp_near is compiled for
#endif
template <bool VEC>
__global__ void __launch_bounds__(128, AP_CSP_MINB) k_csp_near(const CspArgs A, int* __restrict__ list, int* __restrict__ n_list) {
  __shared__ float s_r2[kNear][128];
  __shared__ unsigned short s_q[kNear][128];
  const int i = blockIdx.x * 128 + threadIdx.x, tx = threadIdx.x;
  if (i >= A.n) return;
  if (A.ch && !A.ch[i]) {
    A.csp[i] = 0.0;
    return;
  }
  const SysInfo& S = sys_of(A.sys, A.atom_sys, i);
  const float4 si = A.s32[i];
  const int wi = __float_as_int(si.w);
  // with nin only the in-range part is walked: the rest lies beyond rpf2
  const int c = A.nin ? A.nin[i] : A.cnt[i];
  const size_t row = (size_t)i * A.cap;
  const float r1 = (A.nin ? A.rpf2 : A.rsf2) * exp2f((2.f / 3.f) * log2f(5.924f / (float)(c + 1)));   // r1^2
  float top = 1.6f * r1, rest = INFINITY;
  int n = 0;
  {
    // four entries at a time, the next four indices loaded ahead of their use
    const int* const rowp = A.nbr + row;
    int4 next = c > 0 ? row4<VEC>(rowp, 0, c) : make_int4(0, 0, 0, 0);
    for (int q0 = 0; q0 < c; q0 += 4) {
      const int4 jj = next;
      float4 sv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) sv[u] = A.s32[q0 + u < c ? pick(jj, u) : i];
      if (q0 + 4 < c) next = row4<VEC>(rowp, q0 + 4, c);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int q = q0 + u;
        if (q >= c) break;
        const float4 sj = sv[u];
        int k[3];
        entry_offset(A.off, row + q, S, wi, __float_as_int(sj.w), k);
        const float dx = (float)k[0] * S.hf[0] + sj.x - si.x;
        const float dy = (float)k[1] * S.hf[1] + sj.y - si.y;
        const float dz = (float)k[2] * S.hf[2] + sj.z - si.z;
        const float r2 = dx * dx + dy * dy + dz * dz;
        if (r2 < top) {
          if (n < kNear) {
            s_r2[n][tx] = r2;
            s_q[n][tx] = (unsigned short)q;
          }
          ++n;
        } else {
          rest = fminf(rest, r2);
        }
      }
    }
  }
  // the threshold that leaves 12 of the list
  bool ok = n <= kNear;
  int m = 0;
  float far = 0.f;
  for (int turn = 0; ok && turn < 4; ++turn, top *= 0.92f) {
    float out = INFINITY;   // the nearest entry of the list beyond the threshold
    m = 0;
    far = 0.f;
    for (int k = 0; k < n; ++k) {
      const float r2 = s_r2[k][tx];
      const bool in = r2 < top;
      m += in ? 1 : 0;
      far = in ? fmaxf(far, r2) : far;
      out = in ? out : fminf(out, r2);
    }
    if (m <= kNN) {
      rest = fminf(rest, out);
      break;
    }
  }
  m = 0;
  for (int k = 0; ok && k < n; ++k)
    if (s_r2[k][tx] <= far && m < kNear) s_q[m++][tx] = s_q[k][tx];
  // the 12 nearest, surely inside r_search, and surely nearer than what was not walked or what
  // rows older than the positions may miss
  ok = ok && m == kNN && rest - far > 2.f * kBand && far < A.rsf2 - kBand && (!A.nin || far + 2.f * kBand < A.rpf2) &&
       (!(A.stale2 > 0.f) || far + 2.f * kBand < A.stale2);
  unsigned lo = 0, hi = 0;   // the pairs found, a | b << 4, the last one in the low byte
  if (ok) {
    float v[kNN][3];
#pragma unroll
    for (int a = 0; a < kNN; ++a) {
      const int q = s_q[a][tx];
      const float4 sj = A.s32[A.nbr[row + q]];
      int k[3];
      entry_offset(A.off, row + q, S, wi, __float_as_int(sj.w), k);
      v[a][0] = (float)k[0] * S.hf[0] + sj.x - si.x;
      v[a][1] = (float)k[1] * S.hf[1] + sj.y - si.y;
      v[a][2] = (float)k[2] * S.hf[2] + sj.z - si.z;
    }
    const float lim = 0.25f * r1;
    float big = 0.f, next = INFINITY;
    int pairs = 0;
#pragma unroll
    for (int a = 0; a < kNN; ++a)
#pragma unroll
      for (int b = a + 1; b < kNN; ++b) {
        const float sx = v[a][0] + v[b][0], sy = v[a][1] + v[b][1], sz = v[a][2] + v[b][2];
        const float p = sx * sx + sy * sy + sz * sz;
        if (p < lim) {
          hi = __funnelshift_l(lo, hi, 8);
          lo = lo << 8 | (unsigned)(a | b << 4);
          ++pairs;
          big = fmaxf(big, p);
        } else {
          next = fminf(next, p);
        }
      }
    ok = pairs == kHalf && next - big > 2.f * kBand;
  }
  if (!ok) {
    list[atomicAdd(n_list, 1)] = i;
    return;
  }
  // exact values of the six pairs, summed in ascending order
  const int4 ci = A.cunw[i];
  double chosen[kHalf];
#pragma unroll
  for (int t = 0; t < kHalf; ++t) {
    const unsigned ab = t < 4 ? lo >> (8 * t) : hi >> (8 * (t - 4));
    double d[2][3];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int q = s_q[(e ? ab >> 4 : ab) & 15][tx];
      int j, s[3];
      exact_entry(A.x, S, i, ci, A.nbr, A.off, A.cunw, row, q, d[e], j, s);
    }
    const double s3[3] = {__dadd_rn(d[0][0], d[1][0]), __dadd_rn(d[0][1], d[1][1]), __dadd_rn(d[0][2], d[1][2])};
    chosen[t] = norm2_exact(s3);
  }
  A.csp[i] = sum_ascending(chosen);
}

template <typename K>
__device__ inline K warp_min_key(K v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const K u = __shfl_xor_sync(0xffffffffu, v, o);
    v = u < v ? u : v;
  }
  return v;
}

// One warp per atom: the atoms of list[0, *n_list) or, with a null list, all n atoms.  The 13
// nearest in FP32 by 13 warp minima over the row (key: r^2 bits, row position); the exact
// (r^2, j, image) selection instead where FP32 cannot decide the 12/13 boundary.  Then all 66
// pair values in FP64, two or three per lane, and six minima of their bit patterns.
// list2: what k_csp_sort handed on, when it ran.
__global__ void __launch_bounds__(128) k_csp_exact(const CspArgs A, const int* __restrict__ list,
                                                   const int* __restrict__ n_list, const int* __restrict__ list2,
                                                   const int* __restrict__ n_list2, int sort_from) {
  const int lane = threadIdx.x & 31, warps = (gridDim.x * blockDim.x) >> 5;
  const bool sorted = list && *n_list > sort_from;
  const int m = !list ? A.n : sorted ? *n_list2 : *n_list;
  const unsigned long long none = ~0ull;
  for (int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < m; w += warps) {
    const int i = !list ? w : sorted ? list2[w] : list[w];
    if (A.ch && !A.ch[i]) {
      if (lane == 0) A.csp[i] = 0.0;
      continue;
    }
    const SysInfo& S = sys_of(A.sys, A.atom_sys, i);
    const float4 si = A.s32[i];
    const int4 ci = A.cunw[i];
    const int c = A.cnt[i];
    const size_t row = (size_t)i * A.cap;
    // FP32 key of row position t; none outside r_search (decided exactly in its guard band)
    auto key = [&](int t) -> unsigned long long {
      const int j = A.nbr[row + t];
      const float4 sj = A.s32[j];
      int k[3];
      entry_offset(A.off, row + t, S, ci.w, __float_as_int(sj.w), k);
      const float dx = (float)k[0] * S.hf[0] + sj.x - si.x;
      const float dy = (float)k[1] * S.hf[1] + sj.y - si.y;
      const float dz = (float)k[2] * S.hf[2] + sj.z - si.z;
      const float r2 = dx * dx + dy * dy + dz * dz;
      if (r2 > A.rsf2 + kBand) return none;
      if (r2 >= A.rsf2 - kBand) {
        double d[3];
        exact_disp(A.x, S, i, j, ci, A.cunw[j], k, d);
        if (!(norm2_exact(d) < A.rs2)) return none;
      }
      return (unsigned long long)__float_as_uint(r2) << 32 | (unsigned)t;
    };
    constexpr int kKeep = 5;   // keys of the first 160 row positions stay in registers
    unsigned long long ks[kKeep];
    int n_in = 0;
#pragma unroll
    for (int u = 0; u < kKeep; ++u) {
      const int t = lane + 32 * u;
      ks[u] = t < c ? key(t) : none;
      n_in += __popc(__ballot_sync(0xffffffffu, ks[u] != none));
    }
    for (int t0 = 32 * kKeep; t0 < c; t0 += 32) {
      const int t = t0 + lane;
      n_in += __popc(__ballot_sync(0xffffffffu, t < c && key(t) != none));
    }
    int mine = 0;   // lane a < 12: row position of the a-th neighbour
    float r12 = INFINITY, r13 = INFINITY;
    unsigned long long last = 0;
    for (int a = 0; a <= kNN && a < n_in; ++a) {
      unsigned long long best = none;
#pragma unroll
      for (int u = 0; u < kKeep; ++u)
        if ((a == 0 || ks[u] > last) && ks[u] < best) best = ks[u];
      for (int t = 32 * kKeep + lane; t < c; t += 32) {
        const unsigned long long v = key(t);
        if ((a == 0 || v > last) && v < best) best = v;
      }
      last = warp_min_key(best);
      if (a == kNN - 1) r12 = __uint_as_float((unsigned)(last >> 32));
      if (a == kNN) r13 = __uint_as_float((unsigned)(last >> 32));
      if (lane == a) mine = (int)(unsigned)last;
    }
    // rows older than the positions: see csp_atom
    if (A.stale2 > 0.f && !(n_in >= kNN && r12 + 2.f * kBand < A.stale2) && lane == 0) atomicAdd(A.n_stale, 1);
    if (n_in < kNN) {
      if (lane == 0) A.csp[i] = INFINITY;
      continue;
    }
    if (n_in > kNN && r13 - r12 <= 2.f * kBand) {
      // exact order: the next entry after (r_l, t_l) by (r^2, j, image), 12 times
      double r_l = -1.0;
      int t_l = -1;
      for (int a = 0; a < kNN; ++a) {
        double r_b = INFINITY;
        int t_b = -1;
        for (int t = lane; t < c; t += 32) {
          double d[3];
          int j, s[3];
          exact_entry(A.x, S, i, ci, A.nbr, A.off, A.cunw, row, t, d, j, s);
          const double r2 = norm2_exact(d);
          if (!(r2 < A.rs2)) continue;
          if (t_l >= 0 && (t == t_l || !entry_less(A.x, S, i, ci, A.nbr, A.off, A.cunw, row, r_l, t_l, r2, t))) continue;
          if (t_b < 0 || entry_less(A.x, S, i, ci, A.nbr, A.off, A.cunw, row, r2, t, r_b, t_b)) {
            r_b = r2;
            t_b = t;
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const double r_o = __shfl_xor_sync(0xffffffffu, r_b, o);
          const int t_o = __shfl_xor_sync(0xffffffffu, t_b, o);
          if (t_o >= 0 && (t_b < 0 || (t_o != t_b && entry_less(A.x, S, i, ci, A.nbr, A.off, A.cunw, row, r_o, t_o, r_b, t_b)))) {
            r_b = r_o;
            t_b = t_o;
          }
        }
        r_l = r_b;
        t_l = t_b;
        if (lane == a) mine = t_b;
      }
    }
    double d[3] = {0.0, 0.0, 0.0};
    if (lane < kNN) {
      int j, s[3];
      exact_entry(A.x, S, i, ci, A.nbr, A.off, A.cunw, row, mine, d, j, s);
    }
    long long pv[3];
#pragma unroll
    for (int u = 0; u < 3; ++u) {
      int p = lane + 32 * u, a = 0;   // pair p of the 66: (a, b), a < b
      const bool have = p < kNN * (kNN - 1) / 2;
      if (!have) p = 0;
#pragma unroll
      for (int e = kNN - 1; e > 0; --e)
        if (a == kNN - 1 - e && p >= e) {
          p -= e;
          ++a;
        }
      const int b = a + 1 + p;
      double s3[3];
#pragma unroll
      for (int e = 0; e < 3; ++e)
        s3[e] = __dadd_rn(__shfl_sync(0xffffffffu, d[e], a), __shfl_sync(0xffffffffu, d[e], b));
      pv[u] = have ? __double_as_longlong(norm2_exact(s3)) : 0x7fffffffffffffffll;
    }
    double sum = 0.0;
    for (int t = 0; t < kHalf; ++t) {
      const long long best = pv[0] < pv[1] ? (pv[0] < pv[2] ? pv[0] : pv[2]) : (pv[1] < pv[2] ? pv[1] : pv[2]);
      const long long v = warp_min_key(best);
      // one copy of the value is used up (equal values are taken one after the other)
      const unsigned who = __ballot_sync(0xffffffffu, best == v);
      if (lane == __ffs(who) - 1) {
        if (pv[0] == v) pv[0] = 0x7fffffffffffffffll;
        else if (pv[1] == v) pv[1] = 0x7fffffffffffffffll;
        else pv[2] = 0x7fffffffffffffffll;
      }
      sum = t == 0 ? __longlong_as_double(v) : __dadd_rn(sum, __longlong_as_double(v));
    }
    if (lane == 0) A.csp[i] = sum;
  }
}

// Canonical moving average over a ring buffer [ns][n]: oldest -> newest, then / ns.
__device__ inline double ring_mean(const double* __restrict__ hist, int ns, int newest, size_t n, int i) {
  int q0 = (newest + 1) % ns;
  double s = hist[(size_t)q0 * n + i];
  for (int q = 1; q < ns; ++q) s = __dadd_rn(s, hist[(size_t)((newest + 1 + q) % ns) * n + i]);
  return __ddiv_rn(s, (double)ns);
}

// Push CSP, average, lambda_0 (Eq. lambda_1_i), detected flag, lambda_min init.
__global__ void k_lambda0(int n, const uint8_t* __restrict__ ch, const double* __restrict__ csp,
                          double* __restrict__ hist, int ns, int pos, int fill, double csp_lo, double csp_hi,
                          int mode, double* __restrict__ csp_avg, double* __restrict__ lam0,
                          double* __restrict__ lam_min, int* __restrict__ flag, float* __restrict__ vmin_f,
                          int* __restrict__ n_det1) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) *n_det1 = 0;   // for the spread that follows
  if (i >= n) return;
  vmin_f[i] = 3.4e38f;       // the FP32 minima of the spread start above any estimate
  double c = csp[i];
  if (fill) {
    for (int q = 0; q < ns; ++q) hist[(size_t)q * n + i] = c;
  } else {
    hist[(size_t)pos * n + i] = c;
  }
  double avg = ring_mean(hist, ns, pos, (size_t)n, i);
  csp_avg[i] = avg;
  bool changeable = !ch || ch[i];
  double l0 = 1.0;
  if (changeable) {
    double y = __ddiv_rn(__dsub_rn(csp_hi, avg), __dsub_rn(csp_hi, csp_lo));
    l0 = __dsub_rn(1.0, fcut_exact(y, mode));
  }
  lam0[i] = l0;
  lam_min[i] = changeable ? l0 : 1.0;
  flag[i] = (changeable && l0 < 1.0) ? 1 : 0;
}

__global__ void k_compact(int n, const int* __restrict__ flag, const int* __restrict__ scan, int* __restrict__ out,
                          int* __restrict__ count32, long long* __restrict__ count64) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n && flag[i]) out[scan[i]] = i;
  if (i == 0) {
    int tot = scan[n];
    if (count32) *count32 = tot;
    if (count64) *count64 = tot;
  }
}

// lambda_min spread (Eq. lambda_2_i): one warp per detected atom i scans the cells
// within r_hi; for every image j with r_ij < r_hi it lowers lambda_min,j to
// 1 - (1 - lambda_0,i) f_cut((r_ij - r_lo)/(r_hi - r_lo)) by a 64-bit atomicMin on
// the bit pattern (order-free and exact for non-negative doubles).
// The warp takes the stencil cells 32 at a time; the cells that can reach r_hi form,
// through a warp scan of their atom counts, one stream of candidate atoms that the
// lanes share out (lane k takes candidates k, k + 32, ...; its cell is found by a
// binary search over the 32 prefix sums), so lanes stay busy whatever the cells hold.
constexpr int kSpreadWarps = 8;

// The exact value 1 - (1 - lambda_0,i) f_cut((r_ij - r_lo)/(r_hi - r_lo)) of pair (i, j),
// j in the stencil cell of periodic image img relative to i's wrapped cell cw_i; false if
// r_ij >= r_hi.  Image relative to the input positions: s = img + nwrap_i - nwrap_j.
__device__ inline bool spread_value(const double* __restrict__ x, const SysInfo& S, int i, int j, const int4& ci,
                                    const int4& cj, const int img[3], double rh2, double r_lo, double width,
                                    double one_minus, int mode, double& v) {
  const int cwi[3] = {cell_x(ci.w), cell_y(ci.w), cell_z(ci.w)};
  const int cwj[3] = {cell_x(cj.w), cell_y(cj.w), cell_z(cj.w)};
  const int cu_i[3] = {ci.x, ci.y, ci.z}, cu_j[3] = {cj.x, cj.y, cj.z};
  double d[3];
  for (int q = 0; q < 3; ++q) {
    int sd = 0;
    if (S.periodic[q]) sd = img[q] + (cu_i[q] - cwi[q]) / S.nc[q] - (cu_j[q] - cwj[q]) / S.nc[q];
    const double shifted = sd == 0 ? x[3 * j + q] : __dadd_rn(x[3 * j + q], __dmul_rn((double)sd, S.L[q]));
    d[q] = __dsub_rn(shifted, x[3 * i + q]);
  }
  const double r2 = norm2_exact(d);
  if (!(r2 < rh2)) return false;
  const double r = __dsqrt_rn(r2);
  const double f = fcut_exact(__ddiv_rn(__dsub_rn(r, r_lo), width), mode);
  v = __dsub_rn(1.0, __dmul_rn(one_minus, f));
  return true;
}
#ifndef AP_SPREAD_UNROLL
#define AP_SPREAD_UNROLL 1   // unroll depth of the per-lane candidate loop (compile-time tuning)
#endif
constexpr int kSpreadUnroll = AP_SPREAD_UNROLL;
#ifndef AP_SPREAD_QUEUE
#define AP_SPREAD_QUEUE 1   // walk only the cells that can reach r_hi, 32 at a time (compile-time tuning)
#endif

// Two passes over the same candidates, since FP64 is slow on this GPU.  PHASE 0 (FP32): a
// pair surely inside r_lo has f_cut = 1, so its exact value 1 - (1 - lambda_0,i) needs no
// distance and goes straight into lambda_min,j; vmin_f[j] = the smallest FP32 estimate
// (error < 1e-5) over the pairs surely inside r_hi.  PHASE 1: the exact value of the other
// pairs only where it can set the final minimum: the estimate can go below the current
// lambda_min,j and, for a pair surely inside r_hi, lies within 1e-4 of vmin_f[j] (a pair in
// the guard band around r_hi is always evaluated).  Without the first pass every new
// running minimum, and every pair inside r_lo (they tie), took an exact value.
template <int PHASE>
__global__ void __launch_bounds__(kSpreadWarps * 32) k_spread(
    const int* __restrict__ det, const int* __restrict__ n_det, const double* __restrict__ x,
    const uint8_t* __restrict__ ch, const SysInfo* __restrict__ sys, const int* __restrict__ atom_sys,
    const float4* __restrict__ s32, const int4* __restrict__ cunw, const int* __restrict__ cstart,
    const int* __restrict__ catoms, const double* __restrict__ lam0, double r_lo, double r_hi, int mode, int sx,
    int sy, int sz, double* __restrict__ lam_min, float margin, float* __restrict__ vmin_f,
    int* __restrict__ det1, int* __restrict__ n_det1) {
  // per warp: inclusive prefix of candidate counts, first catoms slot, stencil offset
  __shared__ int s_pre[kSpreadWarps][32], s_beg[kSpreadWarps][32], s_t[kSpreadWarps][32], s_img[kSpreadWarps][32];
  __shared__ int4 s_q[kSpreadWarps][64];   // per warp: queued cells (first slot, count, stencil index, image)
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  const int m = *n_det;
  const double rh2 = __dmul_rn(r_hi, r_hi);
  const float rhf2 = (float)rh2;
  const float rlo2f = (float)__dmul_rn(r_lo, r_lo);
  // cells older than the positions (atoms up to `margin` from their cells): prune beyond r_hi + margin
  const float rprune = (float)r_hi + margin, prune2 = rprune * rprune;
  const double width = __dsub_rn(r_hi, r_lo);
  const float r_lo_f = (float)r_lo, inv_w_f = (float)(1.0 / width);
  const int wx = 2 * sx + 1, wy = 2 * sy + 1, wz = 2 * sz + 1;
  const int ncell = wx * wy * wz;
  for (int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < m; w += warps) {
    const int i = det[w];
    const SysInfo& S = sys_of(sys, atom_sys, i);
    const float4 si = s32[i];
    const int4 ci = cunw[i];
    const double one_minus = __dsub_rn(1.0, lam0[i]);
    const float one_minus_f = (float)one_minus;
    const double v_in = __dsub_rn(1.0, __dmul_rn(one_minus, 1.0));   // the value of a pair inside r_lo
    bool need = false;   // PHASE 0: a pair outside r_lo that can still go below lambda_min,j
    const int cw[3] = {cell_x(ci.w), cell_y(ci.w), cell_z(ci.w)};
    // the scan of a batch of cells' atom counts and the stream of their candidates
    auto walk = [&](int cnt, int beg, int t, int imgp) {
      int pre = cnt;   // inclusive warp scan of the counts
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, pre, o);
        if (lane >= o) pre += v;
      }
      const int total = __shfl_sync(0xffffffffu, pre, 31);
      s_pre[wib][lane] = pre;
      s_beg[wib][lane] = beg;
      s_t[wib][lane] = t;
      s_img[wib][lane] = imgp;
      __syncwarp();
#if AP_SPREAD_UNROLL > 1
#pragma unroll kSpreadUnroll
#endif
      for (int k = lane; k < total; k += 32) {
        // cell of candidate k: the first c with s_pre[c] > k
        int lo = 0, hi = 31;
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (s_pre[wib][mid] > k) hi = mid;
          else lo = mid + 1;
        }
        const int c = lo;
        const int a = s_beg[wib][c] + k - (c ? s_pre[wib][c - 1] : 0);
        const int tt = s_t[wib][c], ip = s_img[wib][c];
        const int dx = tt % wx - sx, dy = (tt / wx) % wy - sy, dz = tt / (wx * wy) - sz;
        const int j = catoms[a];
        if (j == i && dx == 0 && dy == 0 && dz == 0) continue;
        if (ch && !ch[j]) continue;
        const float ox = (float)dx * S.hf[0] - si.x;
        const float oy = (float)dy * S.hf[1] - si.y;
        const float oz = (float)dz * S.hf[2] - si.z;
        const float4 sj = s32[j];
        const float ddx = ox + sj.x, ddy = oy + sj.y, ddz = oz + sj.z;
        const float r2f = ddx * ddx + ddy * ddy + ddz * ddz;
        if (r2f > rhf2 + kBand) continue;
        // FP32 estimate of the candidate value (error < 1e-5)
        const float vf = fmaxf(0.f, 1.f - one_minus_f * fcut_f((sqrtf(r2f) - r_lo_f) * inv_w_f, mode));
        const bool inside = r2f < rhf2 - kBand;
        if constexpr (PHASE == 0) {
          // a pair that cannot go below the current lambda_min,j (which only decreases) is never the minimum
          if ((double)vf - 1e-4 >= __ldcg(&lam_min[j])) continue;
          if (r2f < rlo2f - kBand) {
            // surely inside r_lo: f_cut = 1, and the exact value 1 - (1 - lambda_0,i) needs no distance
            if (v_in < __ldcg(&lam_min[j]))
              atomicMin((unsigned long long*)&lam_min[j], (unsigned long long)__double_as_longlong(v_in));
            if (vf < __ldcg(&vmin_f[j])) atomicMin((unsigned int*)&vmin_f[j], __float_as_uint(vf));
            continue;
          }
          need = true;   // the second pass may take this pair's exact value
          if (inside && vf < __ldcg(&vmin_f[j])) atomicMin((unsigned int*)&vmin_f[j], __float_as_uint(vf));
          continue;
        }
        if (r2f < rlo2f - kBand) continue;   // applied by the first pass
        // if even its lower bound cannot go below the current lambda_min,j (which only
        // decreases), or a surely-inside pair's estimate lies above the smallest one by
        // more than twice the error, the exact value cannot be the final minimum
        if ((double)vf - 1e-4 >= __ldcg(&lam_min[j])) continue;
        if (inside && vf > __ldcg(&vmin_f[j]) + 1e-4f) continue;
        const int img[3] = {off_x(ip), off_y(ip), off_z(ip)};
        double v;
        if (!spread_value(x, S, i, j, ci, cunw[j], img, rh2, r_lo, width, one_minus, mode, v)) continue;
        atomicMin((unsigned long long*)&lam_min[j], (unsigned long long)__double_as_longlong(v));
      }
      __syncwarp();
    };
    int queued = 0;
    for (int t0 = 0; t0 < ncell; t0 += 32) {
      // this lane's cell of the chunk: kept if it exists and can reach r_hi
      const int t = t0 + lane;
      int cnt = 0, beg = 0, imgp = 0;
      if (t < ncell) {
        const int dx = t % wx - sx, dy = (t / wx) % wy - sy, dz = t / (wx * wy) - sz;
        int tc[3] = {cw[0] + dx, cw[1] + dy, cw[2] + dz};
        int img[3] = {0, 0, 0};
        bool skip = false;
        for (int a = 0; a < 3; ++a) {
          if (S.periodic[a]) {
            img[a] = floor_div(tc[a], S.nc[a]);
            tc[a] -= img[a] * S.nc[a];
          } else if (tc[a] < 0 || tc[a] >= S.nc[a]) {
            skip = true;
          }
        }
        if (!skip) {
          const float gx = fmaxf(0.f, fmaxf((float)dx * S.hf[0] - si.x, si.x - (float)(dx + 1) * S.hf[0]));
          const float gy = fmaxf(0.f, fmaxf((float)dy * S.hf[1] - si.y, si.y - (float)(dy + 1) * S.hf[1]));
          const float gz = fmaxf(0.f, fmaxf((float)dz * S.hf[2] - si.z, si.z - (float)(dz + 1) * S.hf[2]));
          if (gx * gx + gy * gy + gz * gz <= prune2 + kBand) {
            const int cid = S.cell_base + (tc[2] * S.nc[1] + tc[1]) * S.nc[0] + tc[0];
            beg = cstart[cid];
            cnt = cstart[cid + 1] - beg;
            // periodic image of the cell, 8 bits per component biased by 128
            imgp = pack_off(img[0], img[1], img[2]);
          }
        }
      }
#if AP_SPREAD_QUEUE
      // queue the cells that can reach r_hi; walk them 32 at a time
      const unsigned vm = __ballot_sync(0xffffffffu, cnt > 0);
      if (cnt > 0) s_q[wib][queued + __popc(vm & lt)] = make_int4(beg, cnt, t, imgp);
      queued += __popc(vm);
      __syncwarp();
      const bool last = t0 + 32 >= ncell;
      while (queued >= 32 || (last && queued > 0)) {
        const int take_n = queued < 32 ? queued : 32;
        const int4 e = lane < take_n ? s_q[wib][lane] : make_int4(0, 0, 0, 0);
        __syncwarp();
        if (lane + 32 < queued) s_q[wib][lane] = s_q[wib][lane + 32];
        queued -= take_n;
        __syncwarp();
        walk(e.y, e.x, e.z, e.w);
      }
#else
      walk(cnt, beg, t, imgp);
#endif
    }
    // the second pass visits only the detected atoms with such a pair (lambda_min only
    // decreases, so a pair screened out here stays out)
    if constexpr (PHASE == 0) {
      if (__any_sync(0xffffffffu, need) && lane == 0) det1[atomicAdd(n_det1, 1)] = i;
    }
  }
}

// Push lambda_min, average (Eq. lambda_3_i), hysteresis (Eq. lambda_4_i), flag precise.
__global__ void k_lambda_final(int n, const uint8_t* __restrict__ ch, const double* __restrict__ lam_min,
                               double* __restrict__ hist, int ns, int pos, int fill, double dlam_min,
                               double* __restrict__ lam_avg, double* __restrict__ lam_prev, double* __restrict__ lam,
                               int* __restrict__ flag) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double lm = lam_min[i];
  if (fill) {
    for (int q = 0; q < ns; ++q) hist[(size_t)q * n + i] = lm;
  } else {
    hist[(size_t)pos * n + i] = lm;
  }
  double avg = ring_mean(hist, ns, pos, (size_t)n, i);
  lam_avg[i] = avg;
  double prev = fill ? avg : lam_prev[i];
  bool take = fabs(__dsub_rn(avg, prev)) >= dlam_min || avg == 0.0 || avg == 1.0;
  double l = take ? avg : prev;
  if (ch && !ch[i]) l = 1.0;
  lam_prev[i] = l;
  lam[i] = l;
  flag[i] = l < 1.0 ? 1 : 0;
}

inline int nblk(int64_t n, int t) { return (int)((n + t - 1) / t); }

}  // namespace

void launch_csp(ap_ctx* c, const double* d_x, const uint8_t* d_ch, cudaStream_t s, bool fresh_rows,
                double stale_disp) {
  double r = c->cfg.eam_rc + c->cfg.skin;
  double rs2 = r * r;
  const int* off = c->stored_off ? c->d_off_eam : nullptr;
  int* n_slow = &c->d_sc->n_csp_slow;
  // n_csp_slow, n_csp_list and, for rows older than the positions, n_stale_bad
  cudaMemsetAsync(n_slow, 0, (stale_disp > 0.0 ? 3 : 2) * sizeof(int), s);
  // Rows older than the positions: stale2 = the radius inside which they are complete.
  // The build's split still bounds the skin part from below: its entries were beyond r_c
  // at the build and are now beyond r_c - 2 m, the radius the in-range part is tested
  // against before the skin part is skipped.
  float stale2 = 0.f;
  const int* nin = fresh_rows ? c->d_lim_eam : nullptr;
  float rpf2 = c->split_rpf2;
  if (stale_disp > 0.0) {
    const double rin = r - 2.0 * stale_disp;
    stale2 = rin > 0.0 ? (float)(rin * rin) : 1e-30f;
    const double rp = std::sqrt((double)c->split_rpf2) - 2.0 * stale_disp;
    nin = c->d_split_eam;
    rpf2 = rp > 0.0 ? (float)(rp * rp) : 0.f;
  }
  CspArgs A;
  A.n = (int)c->n;
  A.x = d_x;
  A.ch = d_ch;
  A.sys = c->d_sys;
  A.atom_sys = c->d_atom_sys;
  A.s32 = c->d_sh32;
  A.cunw = c->d_cunw;
  A.nbr = c->d_nbr_eam;
  A.off = off;
  A.cnt = c->d_cnt_eam;
  A.cap = c->cap_eam;
  A.rsf2 = (float)rs2;
  A.rs2 = rs2;
  A.csp = c->d_csp;
  A.nin = nin;
  A.rpf2 = rpf2;
  A.stale2 = stale2;
  A.n_stale = &c->d_sc->n_stale_bad;
  const int sort_from = kSortFrom * c->num_sms;
  // a few thousand atoms: a warp each at once (237 atoms 14 us; a thread each took 64 us, since
  // one atom's chain is that long)
  if (c->n <= 32 * c->num_sms) {
    k_csp_exact<<<nblk(c->n, 4), 128, 0, s>>>(A, nullptr, nullptr, nullptr, nullptr, 0);
    c->kernels += 1;
    return;
  }
  int* n_list = &c->d_sc->n_csp_list;
  auto near = c->cap_eam % 4 == 0 ? k_csp_near<true> : k_csp_near<false>;
  near<<<nblk(c->n, 128), 128, 0, s>>>(A, c->d_csp_slow, n_list);
  // the handed-over atoms, grid-stride over the device-side counts; d_det1 is free until the spread
  auto sort = c->cap_eam % 4 == 0 ? k_csp_sort<true> : k_csp_sort<false>;
  if (c->n > sort_from)
    sort<<<c->num_sms * kSortBlocks, 128, 0, s>>>(A, c->d_csp_slow, n_list, c->d_det1, n_slow, sort_from);
  k_csp_exact<<<c->num_sms * 8, 128, 0, s>>>(A, c->d_csp_slow, n_list, c->d_det1, n_slow, sort_from);
  c->kernels += c->n > sort_from ? 3 : 2;
}

// d_score: the detection score pushed into the history (CSP, or the selector's p),
// with thresholds (lo, hi) in the f_cut argument (hi - avg)/(hi - lo).
void launch_lambda0(ap_ctx* c, const uint8_t* d_ch, const double* d_score, double lo, double hi, cudaStream_t s) {
  int ns = c->cfg.n_csp_avg;
  int fill = c->hist_started ? 0 : 1;
  int pos = fill ? 0 : (c->csp_pos + 1) % ns;
  c->csp_pos = pos;
  k_lambda0<<<nblk(c->n, 256), 256, 0, s>>>((int)c->n, d_ch, d_score, c->d_csp_hist, ns, pos, fill, lo, hi,
                                            c->cfg.fcut_mode, c->d_csp_avg, c->d_lam0, c->d_lam_min, c->d_flag,
                                            c->d_vmin_f, &c->d_sc->n_det1);
  c->kernels += 2 + scan_exclusive(c->d_flag, c->d_scan, (int)c->n, c->d_scan_tmp, s);
  k_compact<<<nblk(c->n, 256), 256, 0, s>>>((int)c->n, c->d_flag, c->d_scan, c->d_detected, &c->d_sc->n_detected,
                                            nullptr);
}

void launch_spread(ap_ctx* c, const double* d_x, const uint8_t* d_ch, cudaStream_t s) {
  int grid = c->num_sms * 8;
  const int* st = c->cells_stale ? c->sten_spread_stale : c->sten_spread;
  const float margin = c->cells_stale ? (float)c->stale_m : 0.f;
  k_spread<0><<<grid, kSpreadWarps * 32, 0, s>>>(c->d_detected, &c->d_sc->n_detected, d_x, d_ch, c->d_sys,
                                                 c->d_atom_sys, c->d_sh32, c->d_cunw, c->d_cell_start,
                                                 c->d_cell_atoms, c->d_lam0, c->cfg.r_lo, c->cfg.r_hi,
                                                 c->cfg.fcut_mode, st[0], st[1], st[2], c->d_lam_min, margin,
                                                 c->d_vmin_f, c->d_det1, &c->d_sc->n_det1);
  k_spread<1><<<grid, kSpreadWarps * 32, 0, s>>>(c->d_det1, &c->d_sc->n_det1, d_x, d_ch, c->d_sys,
                                                 c->d_atom_sys, c->d_sh32, c->d_cunw, c->d_cell_start,
                                                 c->d_cell_atoms, c->d_lam0, c->cfg.r_lo, c->cfg.r_hi,
                                                 c->cfg.fcut_mode, st[0], st[1], st[2], c->d_lam_min, margin,
                                                 c->d_vmin_f, nullptr, nullptr);
  c->kernels += 2;
}

void launch_lambda_final(ap_ctx* c, const uint8_t* d_ch, double* d_lam, int* d_queue, int64_t* d_nq64,
                         cudaStream_t s) {
  int ns = c->cfg.n_lam_avg;
  int fill = c->hist_started ? 0 : 1;
  int pos = fill ? 0 : (c->lam_pos + 1) % ns;
  c->lam_pos = pos;
  c->hist_started = true;
  k_lambda_final<<<nblk(c->n, 256), 256, 0, s>>>((int)c->n, d_ch, c->d_lam_min, c->d_lam_hist, ns, pos, fill,
                                                 c->cfg.dlam_min, c->d_lam_avg, c->d_lam_prev, d_lam, c->d_flag);
  c->kernels += 2 + scan_exclusive(c->d_flag, c->d_scan, (int)c->n, c->d_scan_tmp, s);
  k_compact<<<nblk(c->n, 256), 256, 0, s>>>((int)c->n, c->d_flag, c->d_scan, d_queue, &c->d_sc->n_precise,
                                            (long long*)(d_nq64 ? d_nq64 : (int64_t*)&c->d_sc->n_precise64));
}

}  // namespace ap
