// Local thermostat (Appendix C): energy errors of a lambda update and their
// momentum-conserving correction.
//
//   k_th_delta     Delta lambda_i = lambda_i^c - lambda_i^d and the ACE weights -Delta lambda_i
//                  of the difference force (F^c - F^d is linear in Delta lambda: an EAM
//                  pass with weights Delta lambda plus an ACE pass over K = {Delta lambda != 0}
//                  with weights -Delta lambda, run by the caller);
//   k_th_energy    Delta E_i = Delta T_i + Delta V_i (Eqs. Delta_T_i, Delta_V_i, Delta_E_i)
//                  from F^d, F^c - F^d, v(t + dt/2), E^f and E^p, for mobile atoms;
//   k_th_bin/...   the atoms with Delta E_i != 0 binned into sweep cells of edge
//                  >= 2 (r_row + skin), sorted by index inside a cell;
//   k_th_rescale   one warp per cell of one colour (8 launches): for every atom of
//                  the cell in ascending index, Omega_i = {i} + the distinct mobile
//                  atoms of its EAM row, v_cm, the relative kinetic energy, beta
//                  (Eq. beta_omega_i) and v_j <- v_cm + beta (v_j - v_cm)
//                  (Eq. p_resc_omega).  Cells of one colour are a cell apart, so
//                  their groups are disjoint and run concurrently.
#include <cmath>

#include "ap_internal.cuh"

namespace ap {

namespace {

constexpr double kAcc = 1.602176634e-19 / 1.66053906660e-27 * 1e-20 / 1e-10;   // A/fs^2 per eV/(A amu)

__global__ void k_th_delta(int n, const double* __restrict__ lam_c, const double* __restrict__ lam_d,
                           double* __restrict__ dlam, double* __restrict__ wneg, int* __restrict__ flag) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double d = lam_c[i] - lam_d[i];
  dlam[i] = d;
  wneg[i] = -d;
  flag[i] = d != 0.0 ? 1 : 0;
}

__global__ void k_th_energy(int n, const double* __restrict__ dlam, const double* __restrict__ e_fast,
                            const double* __restrict__ e_prec_k, const double* __restrict__ f_d,
                            const double* __restrict__ df, const double* __restrict__ v_half,
                            const double* __restrict__ mass, const uint8_t* __restrict__ fixed, double dt,
                            double* __restrict__ dE, int* __restrict__ flag) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double e = 0.0;
  if (!(fixed && fixed[i])) {
    // F^c^2 - F^d^2 written as d (2 F^d + d) with d = F^c - F^d: exactly 0 where the
    // difference force is 0 (a contracted fc*fc - fd*fd would leave a rounding residue).
    const double c1 = dt * dt * kAcc / (8.0 * mass[i]);
    for (int a = 0; a < 3; ++a) {
      const double fd = f_d[3 * i + a];
      const double d = df[3 * i + a];
      e += d * (c1 * (2.0 * fd + d) + 0.5 * dt * v_half[3 * i + a]);
    }
    const double dl = dlam[i];
    if (dl != 0.0) e += dl * (e_fast[i] - e_prec_k[i]);
  }
  dE[i] = e;
  flag[i] = e != 0.0 ? 1 : 0;
}

struct ThCells {
  double lo[3], h[3];
  int nc[3], periodic[3];
  double L[3];
};

__device__ inline int th_cell(const ThCells& T, const double* x) {
  int c[3];
  for (int d = 0; d < 3; ++d) {
    double s = x[d] - T.lo[d];
    if (T.periodic[d]) {
      s = fmod(s, T.L[d]);
      if (s < 0) s += T.L[d];
    }
    int k = (int)floor(s / T.h[d]);
    c[d] = k < 0 ? 0 : (k >= T.nc[d] ? T.nc[d] - 1 : k);
  }
  return (c[2] * T.nc[1] + c[1]) * T.nc[0] + c[0];
}

__global__ void k_th_count(const int* __restrict__ q, const int* __restrict__ m, const double* __restrict__ x,
                           ThCells T, int* __restrict__ cell_of, int* __restrict__ count) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= *m) return;
  const int c = th_cell(T, &x[3 * q[k]]);
  cell_of[k] = c;
  atomicAdd(&count[c], 1);
}

__global__ void k_th_scatter(const int* __restrict__ q, const int* __restrict__ m, const int* __restrict__ cell_of,
                             const int* __restrict__ start, int* __restrict__ fill, int* __restrict__ atoms) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= *m) return;
  const int c = cell_of[k];
  atoms[start[c] + atomicAdd(&fill[c], 1)] = q[k];
}

// Ascending index inside every cell: one block per cell, each thread counting the smaller
// indices of the cell (tiles in shared memory) to place its atom.  An insertion sort by one
// thread per cell took 130 us for 150 atoms a cell and grows with the square; cells of a
// small or oddly sized box hold up to a few thousand atoms.
constexpr int kSortThreads = 128;
__global__ void __launch_bounds__(kSortThreads) k_th_sort(const int* __restrict__ start,
                                                          const int* __restrict__ atoms, int* __restrict__ sorted) {
  __shared__ int tile[kSortThreads];
  const int b = start[blockIdx.x], e = start[blockIdx.x + 1];
  for (int a0 = b; a0 < e; a0 += kSortThreads) {
    const int a = a0 + threadIdx.x;
    const int v = a < e ? atoms[a] : 0;
    int rank = 0;
    for (int t0 = b; t0 < e; t0 += kSortThreads) {
      __syncthreads();
      if (t0 + threadIdx.x < e) tile[threadIdx.x] = atoms[t0 + threadIdx.x];
      __syncthreads();
      const int m = min(kSortThreads, e - t0);
      for (int u = 0; u < m; ++u) rank += tile[u] < v ? 1 : 0;
    }
    if (a < e) sorted[b + rank] = v;
  }
}

template <typename T>
__device__ inline T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Total mass and centre-of-mass velocity from the lanes' masses and momenta: four sums over the
// warp in 6 additions per lane instead of 20 (FP64 additions issue at one per 16 cycles here):
// the halves of the warp first split the four values among themselves, then every group of 8
// lanes reduces one of them and divides it by the mass.
__device__ inline void warp_centre(double& sm, double& px, double& py, double& pz) {
  const int lane = threadIdx.x & 31;
  const bool hi = lane & 16, mid = lane & 8;
  double k0 = hi ? py : sm, k1 = hi ? pz : px;
  k0 += __shfl_xor_sync(0xffffffffu, hi ? sm : py, 16);
  k1 += __shfl_xor_sync(0xffffffffu, hi ? px : pz, 16);
  double k = mid ? k1 : k0;
  k += __shfl_xor_sync(0xffffffffu, mid ? k0 : k1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
  sm = __shfl_sync(0xffffffffu, k, 0);
  k = k / sm;
  px = __shfl_sync(0xffffffffu, k, 8);
  py = __shfl_sync(0xffffffffu, k, 16);
  pz = __shfl_sync(0xffffffffu, k, 24);
}

// Member test for row entry t of atom i: a mobile atom other than i that, with DEDUP, does
// not appear earlier in the row.  Only a box narrower than five search cells (DEDUP; there
// the cell offsets are stored) can put two images of one atom, or one of i itself, in a row:
// otherwise every period is at least 2.5 row radii.
template <bool DEDUP>
__device__ inline bool member(const int* __restrict__ row, int t, int i, const uint8_t* __restrict__ fixed) {
  const int j = row[t];
  if (j == i || (fixed && fixed[j])) return false;
  if constexpr (DEDUP) {
    for (int u = 0; u < t; ++u)
      if (row[u] == j) return false;
  }
  return true;
}

// One warp per cell of one colour; the corrections of a cell form a serial chain (each needs
// the velocities that the last one left), so the latency of one correction is the cost.  Each
// lane keeps up to kMem members' velocities in registers between the three sums, what is no
// member carries mass 0 at index i, and what the chain needs of the coming atoms is loaded one
// turn ahead (three turns of indices).  Rows beyond 32 kMem entries take the loop over memory.
// The time of an update follows the number of corrections, few while a run is young.  On a slab of
// 358,012 atoms with 405 / 5,970 / 21,750 / 32,700 of them (third, fourth, fifth and 48th update)
// the thermostat takes 1.7 / 4.1 / 6.6 / 8.5 ms; 23 / 64 / 108 / 145 ms with a membership test over
// the whole row for boxes that cannot need it.  Loading ahead took 2.4 ms off an update of some
// 28,000.  What is left is the FP64 chain of two divisions, a square root and 11 dependent additions.
constexpr int kMem = 6;   // 192 row entries: the default row capacity is 160
template <bool DEDUP>
__global__ void __launch_bounds__(32) k_th_rescale(
    ThCells T, int color, const int* __restrict__ start, const int* __restrict__ atoms, const int* __restrict__ nbr,
    const int* __restrict__ cnt, int cap, const uint8_t* __restrict__ fixed, const double* __restrict__ mass,
    const double* __restrict__ dE, double* __restrict__ v, DevScalars* __restrict__ sc) {
  const int lane = threadIdx.x & 31;
  const int px = color & 1, py = (color >> 1) & 1, pz = (color >> 2) & 1;
  const int mx = (T.nc[0] + 1 - px) / 2, my = (T.nc[1] + 1 - py) / 2, mz = (T.nc[2] + 1 - pz) / 2;
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= mx * my * mz) return;
  const int cx = 2 * (w % mx) + px, cy = 2 * ((w / mx) % my) + py, cz = 2 * (w / (mx * my)) + pz;
  const int cell = (cz * T.nc[1] + cy) * T.nc[0] + cx;
  const int a_end = start[cell + 1];
  const int a0 = start[cell];
  if (a0 >= a_end) return;
  unsigned long long n_ok = 0, n_bad = 0;
  double e_sum = 0.0;
  // What the chain needs of the coming atoms is loaded a turn before it is used, without branches
  // on loaded values: the atom of turn a + 4, the row length of a + 3, the row entries of a + 2,
  // masses, fixed flags and Delta E of a + 1.
  int i4 = -1, i3 = -1, c3 = 0, i2 = -1, c2 = 0, i1 = -1, c1 = 0;
  int j2[kMem], j1[kMem];
  double m1[kMem], de1 = 0.0;
  unsigned f1[kMem];
#pragma unroll
  for (int u = 0; u < kMem; ++u) {
    j2[u] = j1[u] = -1;
    m1[u] = 0.0;
    f1[u] = 0;
  }
  for (int a = a0 - 4; a < a_end; ++a) {
    const int i = i1, c = c1;
    const double de = de1;
    const bool in_regs = c <= 32 * kMem;
    int j[kMem];
    double m[kMem], ux[kMem], uy[kMem], uz[kMem];
    double vx = 0.0, vy = 0.0, vz = 0.0, mi = 0.0;
    if (a >= a0 && in_regs) {
#pragma unroll
      for (int u = 0; u < kMem; ++u) {
        const int t = lane + 32 * u;
        bool is = t < c && j1[u] != i && f1[u] == 0;
        if constexpr (DEDUP) is = is && member<DEDUP>(nbr + (size_t)i * cap, t, i, fixed);
        j[u] = is ? j1[u] : i;
        m[u] = is ? m1[u] : 0.0;
        ux[u] = uy[u] = uz[u] = 0.0;
        if (is) {
          ux[u] = v[3 * j[u]];
          uy[u] = v[3 * j[u] + 1];
          uz[u] = v[3 * j[u] + 2];
        }
      }
    }
    if (a >= a0 && lane == 0) {
      mi = mass[i];
      vx = v[3 * i];
      vy = v[3 * i + 1];
      vz = v[3 * i + 2];
    }
    // turn a + 1: the row entries have arrived
    i1 = i2;
    c1 = c2;
    if (i1 >= 0) {
      de1 = dE[i1];
#pragma unroll
      for (int u = 0; u < kMem; ++u) {
        const bool in = lane + 32 * u < c1;
        j1[u] = j2[u];
        m1[u] = in ? mass[j2[u]] : 0.0;
        f1[u] = in && fixed ? fixed[j2[u]] : 0u;
      }
    }
    // turn a + 2: its row; turn a + 3: its length; turn a + 4: the atom
    i2 = i3;
    c2 = c3;
    if (i2 >= 0) {
      const int* row2 = nbr + (size_t)i2 * cap;
#pragma unroll
      for (int u = 0; u < kMem; ++u) {
        const int t = lane + 32 * u;
        j2[u] = t < c2 && c2 <= 32 * kMem ? row2[t] : i2;
      }
    }
    i3 = i4;
    c3 = i3 >= 0 ? cnt[i3] : 0;
    i4 = a + 4 < a_end && a + 4 >= a0 ? atoms[a + 4] : -1;
    if (a < a0) continue;
    const int* row = nbr + (size_t)i * cap;
    // total mass and momentum of Omega_i (atom i itself in lane 0)
    double sm = mi, spx = mi * vx, spy = mi * vy, spz = mi * vz;
    if (in_regs) {
#pragma unroll
      for (int u = 0; u < kMem; ++u) {
        if (32 * u >= c) break;
        sm += m[u];
        spx = fma(m[u], ux[u], spx);
        spy = fma(m[u], uy[u], spy);
        spz = fma(m[u], uz[u], spz);
      }
    } else {
      for (int t = lane; t < c; t += 32) {
        if (!member<DEDUP>(row, t, i, fixed)) continue;
        const int q = row[t];
        const double mq = mass[q];
        sm += mq;
        spx += mq * v[3 * q];
        spy += mq * v[3 * q + 1];
        spz += mq * v[3 * q + 2];
      }
    }
    double vcx = spx, vcy = spy, vcz = spz;
    warp_centre(sm, vcx, vcy, vcz);
    // relative kinetic energy
    double k = 0.0;
    if (lane == 0) {
      vx -= vcx;
      vy -= vcy;
      vz -= vcz;
      k = mi * (vx * vx + vy * vy + vz * vz);
    }
    if (in_regs) {
#pragma unroll
      for (int u = 0; u < kMem; ++u) {
        if (32 * u >= c) break;
        ux[u] -= vcx;
        uy[u] -= vcy;
        uz[u] -= vcz;
        k = fma(m[u], ux[u] * ux[u] + uy[u] * uy[u] + uz[u] * uz[u], k);
      }
    } else {
      for (int t = lane; t < c; t += 32) {
        if (!member<DEDUP>(row, t, i, fixed)) continue;
        const int q = row[t];
        const double ax = v[3 * q] - vcx, ay = v[3 * q + 1] - vcy, az = v[3 * q + 2] - vcz;
        k += mass[q] * (ax * ax + ay * ay + az * az);
      }
    }
    k = warp_sum(k) * (0.5 / kAcc);
    // a group of atom i alone has no relative velocity, whatever (m v) / m rounds to
    if (sm == __shfl_sync(0xffffffffu, mi, 0)) k = 0.0;
    const double rad = k > 0.0 ? de / k + 1.0 : (de == 0.0 ? 1.0 : -1.0);
    if (rad < 0.0) {
      ++n_bad;
      continue;
    }
    const double beta = sqrt(rad);
    ++n_ok;
    e_sum += de;
    // rescale the relative velocities (every member written by one lane)
    if (lane == 0) {
      v[3 * i] = fma(beta, vx, vcx);
      v[3 * i + 1] = fma(beta, vy, vcy);
      v[3 * i + 2] = fma(beta, vz, vcz);
    }
    if (in_regs) {
#pragma unroll
      for (int u = 0; u < kMem; ++u) {
        if (m[u] != 0.0) {
          v[3 * j[u]] = fma(beta, ux[u], vcx);
          v[3 * j[u] + 1] = fma(beta, uy[u], vcy);
          v[3 * j[u] + 2] = fma(beta, uz[u], vcz);
        }
      }
    } else {
      for (int t = lane; t < c; t += 32) {
        if (!member<DEDUP>(row, t, i, fixed)) continue;
        const int q = row[t];
        v[3 * q] = vcx + beta * (v[3 * q] - vcx);
        v[3 * q + 1] = vcy + beta * (v[3 * q + 1] - vcy);
        v[3 * q + 2] = vcz + beta * (v[3 * q + 2] - vcz);
      }
    }
    __syncwarp();
  }
  if (lane == 0) {
    if (n_bad) {
      atomicOr(&sc->err, kErrRadicand);
      atomicAdd(&sc->th_bad, n_bad);
    }
    if (n_ok) {
      atomicAdd(&sc->th_n, n_ok);
      atomicAdd(&sc->th_e, e_sum);
    }
  }
}

inline int nblk(int64_t n, int t) { return (int)((n + t - 1) / t); }

ThCells th_cells(const ap_ctx* c) {
  const SysInfo& S = c->h_sys[0];
  ThCells T;
  const double hmin = 2.0 * (c->cfg.eam_rc + c->cfg.skin + c->cfg.skin);
  for (int d = 0; d < 3; ++d) {
    int nc = (int)std::floor(S.L[d] / hmin);
    if (nc < 1) nc = 1;
    if (S.periodic[d] && nc > 1 && (nc & 1)) --nc;
    T.nc[d] = nc;
    T.lo[d] = S.lo[d];
    T.L[d] = S.L[d];
    T.h[d] = S.L[d] / nc;
    T.periodic[d] = S.periodic[d];
  }
  return T;
}

}  // namespace

int th_cell_count(const ap_ctx* c) {
  ThCells T = th_cells(c);
  return T.nc[0] * T.nc[1] * T.nc[2];
}

void launch_th_delta(ap_ctx* c, const double* d_lam_c, const double* d_lam_d, cudaStream_t s) {
  const int n = (int)c->n;
  k_th_delta<<<nblk(n, 256), 256, 0, s>>>(n, d_lam_c, d_lam_d, c->d_th_dlam, c->d_th_w, c->d_flag);
  c->kernels += 1;
}

void launch_th_energy(ap_ctx* c, const double* d_f, const double* d_v, const double* d_mass, const uint8_t* d_fixed,
                      cudaStream_t s) {
  const int n = (int)c->n;
  k_th_energy<<<nblk(n, 256), 256, 0, s>>>(n, c->d_th_dlam, c->d_efast, c->d_th_ep, d_f, c->d_th_df, d_v, d_mass,
                                           d_fixed, c->cfg.dt, c->d_th_de, c->d_flag);
  c->kernels += 1;
}

// Bin the queue d_q (count *d_m) into sweep cells and run the 8 colour sweeps.
void launch_th_correct(ap_ctx* c, const int* d_q, const int* d_m, const double* d_x, const uint8_t* d_fixed,
                       const double* d_mass, double* d_v, cudaStream_t s) {
  const int n = (int)c->n;
  ThCells T = th_cells(c);
  const int nc = T.nc[0] * T.nc[1] * T.nc[2];
  cudaMemsetAsync(c->d_th_ccount, 0, sizeof(int) * (size_t)nc, s);
  k_th_count<<<nblk(n, 256), 256, 0, s>>>(d_q, d_m, d_x, T, c->d_th_cellof, c->d_th_ccount);
  c->kernels += 1 + scan_exclusive(c->d_th_ccount, c->d_th_cstart, nc, c->d_scan_tmp, s);
  cudaMemsetAsync(c->d_th_ccount, 0, sizeof(int) * (size_t)nc, s);
  k_th_scatter<<<nblk(n, 256), 256, 0, s>>>(d_q, d_m, c->d_th_cellof, c->d_th_cstart, c->d_th_ccount, c->d_th_atoms);
  int* sorted = c->d_th_cellof;   // free once the scatter has read it
  k_th_sort<<<nc, kSortThreads, 0, s>>>(c->d_th_cstart, c->d_th_atoms, sorted);
  c->kernels += 2;
  auto rescale = c->stored_off ? k_th_rescale<true> : k_th_rescale<false>;
  for (int color = 0; color < 8; ++color) {
    const int px = color & 1, py = (color >> 1) & 1, pz = (color >> 2) & 1;
    const int cells = ((T.nc[0] + 1 - px) / 2) * ((T.nc[1] + 1 - py) / 2) * ((T.nc[2] + 1 - pz) / 2);
    if (cells <= 0) continue;
    rescale<<<nblk(32 * cells, 32), 32, 0, s>>>(T, color, c->d_th_cstart, sorted, c->d_nbr_eam, c->d_cnt_eam,
                                                c->cap_eam, d_fixed, d_mass, c->d_th_de, d_v, c->d_sc);
    c->kernels += 1;
  }
}

}  // namespace ap
