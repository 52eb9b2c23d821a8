// Cell list and neighbour rows (section 2.4: the per-domain neighbour search that
// the paper delegates to LAMMPS).  Row i of a list holds every image (j, s) with
// |x_j + s L - x_i|^2 < r_list^2, decided by that FP64 expression; an FP32
// cell-relative pre-filter only skips candidates that are clearly in or out.
#include <algorithm>
#include <cmath>

#include "ap_internal.cuh"

namespace ap {

namespace {

constexpr int kScanThreads = 512;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

__global__ void k_scan_block(const int* __restrict__ in, int* __restrict__ out, int m, int n_in,
                             int* __restrict__ bsum) {
  __shared__ int ws[kScanThreads / 32];
  const int base = blockIdx.x * kScanTile + threadIdx.x * kScanItems;
  int v[kScanItems];
  int tsum = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    int idx = base + k;
    v[k] = (idx < n_in) ? in[idx] : 0;
    tsum += v[k];
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int x = tsum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[wid] = x;
  __syncthreads();
  if (wid == 0) {
    int w = (lane < kScanThreads / 32) ? ws[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < kScanThreads / 32) ws[lane] = w;
  }
  __syncthreads();
  int run = x - tsum + (wid > 0 ? ws[wid - 1] : 0);
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    int idx = base + k;
    if (idx < m) out[idx] = run;
    run += v[k];
  }
  if (threadIdx.x == kScanThreads - 1) bsum[blockIdx.x] = run;
}

__global__ void k_scan_add(int* __restrict__ out, int m, const int* __restrict__ offs) {
  int b = blockIdx.x;
  int add = offs[b];
  for (int k = threadIdx.x; k < kScanTile; k += blockDim.x) {
    int idx = b * kScanTile + k;
    if (idx < m) out[idx] += add;
  }
}

int scan_rec(const int* in, int n_in, int* out, int m, int* tmp, cudaStream_t s) {
  int nb = (m + kScanTile - 1) / kScanTile;
  int k = 1;
  k_scan_block<<<nb, kScanThreads, 0, s>>>(in, out, m, n_in, tmp);
  if (nb > 1) {
    int* offs = tmp + nb;
    k += scan_rec(tmp, nb, offs, nb, tmp + 2 * nb, s);
    k_scan_add<<<nb, 256, 0, s>>>(out, m, offs);
    ++k;
  }
  return k;
}

__device__ inline int floor_div(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

__device__ inline const SysInfo& sys_of(const SysInfo* sys, const int* atom_sys, int i) {
  return sys[atom_sys ? atom_sys[i] : 0];
}

// ------------------------------------------------------------------ binning
// Cell of every atom, its shadow (the k_shadow arithmetic) and the copy of it that the
// displacement since this build is taken from.
__global__ void k_bin(int n, const double* __restrict__ x, const int32_t* __restrict__ species,
                      const SysInfo* __restrict__ sys, const int* __restrict__ atom_sys, int* __restrict__ cell,
                      int* __restrict__ slot, int4* __restrict__ cunw, int* __restrict__ cell_count,
                      const double* __restrict__ org, float4* __restrict__ s32, double4_32a* __restrict__ s64,
                      float4* __restrict__ s32b, DevScalars* sc) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) {
    sc->max_disp2_bits = 0;
    sc->max_dispa2_bits = 0x7f7f7f7fu;   // the ACE rows' reference shadows belong to the old cells: until the next ACE build
  }
  if (i >= n) return;
  const SysInfo& S = sys_of(sys, atom_sys, i);
  int cw[3], cu[3];
  int bad = 0;
  if (species && species[i] != 0) bad |= kErrArg;
  for (int d = 0; d < 3; ++d) {
    double xv = x[3 * i + d];
    if ((__double2hiint(xv) & 0x7ff00000) == 0x7ff00000) {   // inf or nan
      bad |= kErrNonfinite;
      cw[d] = 0;
      cu[d] = 0;
      continue;
    }
    double rel = xv - S.lo[d];
    // FP32 decides the cell unless the atom lies within 1e-3 of a cell's edge (its error is below
    // 3e-4 cells), or within 1e-2 of the box's: the two FP64 divisions were most of this kernel
    // (4,000,000 atoms 412 -> 79 us)
    const float qf = (float)rel * (1.f / S.hf[d]);
    const int ci = (int)qf;
    const float fr = qf - (float)ci;
    if (qf > 0.01f && qf < (float)S.nc[d] - 0.01f && fr > 1e-3f && fr < 0.999f) {
      cw[d] = cu[d] = ci;
      continue;
    }
    int nw = 0;
    if (S.periodic[d]) {
      nw = (int)floor(rel / S.L[d]);
      rel = rel - (double)nw * S.L[d];
    } else if (rel < 0.0 || rel >= S.L[d]) {
      bad |= kErrBox;
    }
    int c = (int)floor(rel / S.h[d]);
    c = c < 0 ? 0 : (c >= S.nc[d] ? S.nc[d] - 1 : c);
    cw[d] = c;
    cu[d] = c + nw * S.nc[d];
  }
  if (bad) atomicOr(&sc->err, bad);
  int id = S.cell_base + (cw[2] * S.nc[1] + cw[1]) * S.nc[0] + cw[0];
  cell[i] = id;
  const int4 c4 = make_int4(cu[0], cu[1], cu[2], pack_cell(cw[0], cw[1], cw[2]));
  cunw[i] = c4;
  slot[i] = atomicAdd(&cell_count[id], 1);
  const double xi[3] = {x[3 * i + 0], x[3 * i + 1], x[3 * i + 2]};
  double sh[3];
  cell_shadow(S, org, c4, xi, sh);
  const float4 s4 = make_float4((float)sh[0], (float)sh[1], (float)sh[2], __int_as_float(c4.w));
  s32[i] = s4;
  s32b[i] = s4;
  if (s64) s64[i] = make_double4_32a(sh[0], sh[1], sh[2], (double)c4.w);
}

__global__ void k_cell_scatter(int n, const int* __restrict__ cell, const int* __restrict__ slot,
                               const int* __restrict__ start, int* __restrict__ atoms) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  atoms[start[cell[i]] + slot[i]] = i;
}

// Sort each cell's atoms by index so that rows come out in a deterministic order.
__global__ void k_cell_sort(int n_cells, const int* __restrict__ start, int* __restrict__ atoms) {
  int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n_cells) return;
  int b = start[c], e = start[c + 1];
  for (int a = b + 1; a < e; ++a) {
    int t = atoms[a];
    int p = a - 1;
    while (p >= b && atoms[p] > t) {
      atoms[p + 1] = atoms[p];
      --p;
    }
    atoms[p + 1] = t;
  }
}

// Cell-relative coordinates s = (x - lo) - c_unw h; w = packed wrapped cell.
__global__ void k_shadow(int n, const double* __restrict__ x, const SysInfo* __restrict__ sys,
                         const int* __restrict__ atom_sys, const double* __restrict__ org,
                         const int4* __restrict__ cunw, float4* __restrict__ s32, double4_32a* __restrict__ s64) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const SysInfo& S = sys_of(sys, atom_sys, i);
  const int4 c = cunw[i];
  const double xi[3] = {x[3 * i + 0], x[3 * i + 1], x[3 * i + 2]};
  double sh[3];
  cell_shadow(S, org, c, xi, sh);
  s32[i] = make_float4((float)sh[0], (float)sh[1], (float)sh[2], __int_as_float(c.w));
  if (s64) s64[i] = make_double4_32a(sh[0], sh[1], sh[2], (double)c.w);
}

__global__ void k_wrap(int n, double* __restrict__ x, const SysInfo* __restrict__ sys, const int* __restrict__ atom_sys) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const SysInfo& S = sys_of(sys, atom_sys, i);
  for (int d = 0; d < 3; ++d) {
    if (!S.periodic[d]) continue;
    double xv = x[3 * i + d];
    double rel = xv - S.lo[d];
    if (rel >= 0.0 && rel < S.L[d]) continue;
    int nw = (int)floor(rel / S.L[d]);
    x[3 * i + d] = __dsub_rn(xv, __dmul_rn((double)nw, S.L[d]));
  }
}

// ------------------------------------------------------------------ row builds
// The exact decision: |(x_j + S L) - x_i|^2 < rc2 with explicit round-to-nearest
// operations (no contraction), S the image of j relative to the input positions.
__device__ inline bool exact_within(const double* __restrict__ x, const SysInfo& S, int i, int j, const int4& ci,
                                    const int4& cj, const int img[3], double rc2) {
  int cwi[3] = {cell_x(ci.w), cell_y(ci.w), cell_z(ci.w)};
  int cwj[3] = {cell_x(cj.w), cell_y(cj.w), cell_z(cj.w)};
  int cui[3] = {ci.x, ci.y, ci.z};
  int cuj[3] = {cj.x, cj.y, cj.z};
  double r2 = 0.0;
  double dd[3];
  for (int d = 0; d < 3; ++d) {
    int Sd = 0;
    if (S.periodic[d]) Sd = img[d] + (cui[d] - cwi[d]) / S.nc[d] - (cuj[d] - cwj[d]) / S.nc[d];
    double shifted = Sd == 0 ? x[3 * j + d] : __dadd_rn(x[3 * j + d], __dmul_rn((double)Sd, S.L[d]));
    dd[d] = __dsub_rn(shifted, x[3 * i + d]);
  }
  r2 = __dadd_rn(__dadd_rn(__dmul_rn(dd[0], dd[0]), __dmul_rn(dd[1], dd[1])), __dmul_rn(dd[2], dd[2]));
  return r2 < rc2;
}

// One warp builds one row (used for the long ACE rows).  The lanes test the stencil cells
// ((2 sten + 1)^3 around atom i's cell) 32 at a time against the cell-box distance and
// queue the cells that pass in a per-warp shared-memory buffer; each full batch of 32
// queued cells is walked with one cell per lane, the lanes iterating their cells' atoms in
// lock-step, and accepted (j, offset) are appended with ballot compaction.  Entry order:
// (batch, atom slot, lane) -- deterministic.  Returns the full count (may exceed cap).
// With cells older than the positions (atoms moved up to `margin` since the cell build),
// a cell is pruned only beyond r + margin, and the stencil must reach r + 2 margin.
// buf: this warp's 64-entry shared-memory queue (first atom slot, count, cell offset,
// image).
__device__ inline int build_row_warp(int i, const double* __restrict__ x, const SysInfo& S,
                                     const float4* __restrict__ s32, const int4* __restrict__ cunw,
                                     const int* __restrict__ cstart, const int* __restrict__ catoms, float rcf2,
                                     double rc2, float band, int cap, int* __restrict__ row,
                                     int* __restrict__ offrow, int sten, float margin, int4* buf) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const float4 si = s32[i];
  const int4 ci = cunw[i];
  const int cw[3] = {cell_x(ci.w), cell_y(ci.w), cell_z(ci.w)};
  const float rprune = sqrtf(rcf2) + margin, prune2 = rprune * rprune + band;
  const int W = 2 * sten + 1, ncell = W * W * W;
  int cnt = 0, queued = 0;
  for (int t0 = 0; t0 < ncell; t0 += 32) {
    const int t = t0 + lane;
    const int dx = t % W - sten, dy = (t / W) % W - sten, dz = t / (W * W) - sten;
    int tc[3] = {cw[0] + dx, cw[1] + dy, cw[2] + dz};
    int img[3] = {0, 0, 0};
    bool valid = t < ncell;
    for (int d = 0; d < 3 && valid; ++d) {
      if (S.periodic[d]) {
        img[d] = floor_div(tc[d], S.nc[d]);
        tc[d] -= img[d] * S.nc[d];
      } else if (tc[d] < 0 || tc[d] >= S.nc[d]) {
        valid = false;
      }
    }
    if (valid) {
      const float gx = fmaxf(0.f, fmaxf((float)dx * S.hf[0] - si.x, si.x - (float)(dx + 1) * S.hf[0]));
      const float gy = fmaxf(0.f, fmaxf((float)dy * S.hf[1] - si.y, si.y - (float)(dy + 1) * S.hf[1]));
      const float gz = fmaxf(0.f, fmaxf((float)dz * S.hf[2] - si.z, si.z - (float)(dz + 1) * S.hf[2]));
      valid = gx * gx + gy * gy + gz * gz <= prune2;
    }
    int b = 0, len = 0;
    if (valid) {
      const int cid = S.cell_base + (tc[2] * S.nc[1] + tc[1]) * S.nc[0] + tc[0];
      b = cstart[cid];
      len = cstart[cid + 1] - b;
    }
    const unsigned vm = __ballot_sync(0xffffffffu, len > 0);
    if (len > 0) buf[queued + __popc(vm & lt)] = make_int4(b, len, pack_off(dx, dy, dz), pack_off(img[0], img[1], img[2]));
    queued += __popc(vm);
    __syncwarp();
    // walk a full batch, or what is left after the last stencil cell
    const bool last = t0 + 32 >= ncell;
    while (queued >= 32 || (last && queued > 0)) {
      const int take_n = queued < 32 ? queued : 32;
      int4 e = make_int4(0, 0, 0, 0);
      if (lane < take_n) e = buf[lane];
      __syncwarp();
      if (lane + 32 < queued) buf[lane] = buf[lane + 32];   // the rest moves to the front
      queued -= take_n;
      __syncwarp();
      const int ox_i = off_x(e.z), oy_i = off_y(e.z), oz_i = off_z(e.z);
      const int im[3] = {off_x(e.w), off_y(e.w), off_z(e.w)};
      const float ox = (float)ox_i * S.hf[0] - si.x;
      const float oy = (float)oy_i * S.hf[1] - si.y;
      const float oz = (float)oz_i * S.hf[2] - si.z;
      const bool self_cell = ox_i == 0 && oy_i == 0 && oz_i == 0;
      const int maxlen = __reduce_max_sync(0xffffffffu, e.y);
      for (int k = 0; k < maxlen; ++k) {
        bool take = false;
        int j = 0;
        if (k < e.y) {
          j = catoms[e.x + k];
          if (!(j == i && self_cell)) {
            const float4 sj = s32[j];
            const float ddx = ox + sj.x, ddy = oy + sj.y, ddz = oz + sj.z;
            const float r2f = ddx * ddx + ddy * ddy + ddz * ddz;
            if (r2f < rcf2 - band) {
              take = true;
            } else if (r2f <= rcf2 + band) {
              take = exact_within(x, S, i, j, ci, cunw[j], im, rc2);
            }
          }
        }
        const unsigned m = __ballot_sync(0xffffffffu, take);
        const int pos = cnt + __popc(m & lt);
        if (take && pos < cap) {
          row[pos] = j;
          if (offrow) offrow[pos] = e.z;
        }
        cnt += __popc(m);
      }
    }
  }
  return cnt;
}

// ---- EAM rows, one block per group of cells (2 x 2 x 2, or a single one in small systems).
//   * The block stages the candidates of the whole group once, in shared memory: the stencil is
//     walked as pencils of cells along x, contiguous in cell order and cut to the reach of the
//     group's box; of their atoms those within reach of the box are kept, in stencil order.
//   * Each warp takes one cell of the group (or a share of the single cell's atoms) and lists the
//     staged candidates within reach of the box around its atoms (about 250 of the 560 in a
//     cell's 5^3 stencil in FCC copper, of which each atom takes 85 to 110).
//   * Each lane tests a block of consecutive listed candidates against the warp's atoms, three
//     at a time, and keeps a bit per candidate and atom; a scan over the lanes' counts gives
//     every accepted candidate its place in the row.
// A thread per row walked all 560 candidates in one dependent chain and wrote 32 rows at once,
// 4 bytes each: 999,180 atoms at 6.5 A 1.48 -> 1.28 ms, 32,000 atoms 206 -> 64 us, 237 atoms
// 160 -> 13 us (the dependent chain was the cost there).  What binds it now is instruction
// issue: the tests (about 35 % of the instructions) and the writes of the accepted entries.
//
// Row order: first the entries whose FP32 distance lies inside the potential cutoff
// (rpf2 = r_c^2), in stencil order, then the skin entries, last of the stencil first; nin
// receives the length of the first part.  The EAM density pass records, per atom, where the
// in-range entries end at the current positions (it re-tests every entry), so the force pass
// walks only that prefix; the split at build time only makes the prefix short.  The CSP on
// rows built at its own positions may stop after the first part.
constexpr int kBuildWarps = 8;     // warps per block
constexpr int kStage = 1024;       // staged candidates per block; a fuller stage is used up in rounds
// listed candidates per warp (13 or 16 per lane), used up in turns likewise
template <bool ACE>
constexpr int kList = ACE ? 512 : 416;
constexpr int kCentres = 3;        // atoms tested together against a listed candidate

struct BuildArgs {
  const double* x;
  const SysInfo* sys;
  int n_sys, group;         // cells per edge of a block's group: 2 or 1
  const float4* s32c;       // shadows in cell order
  const int4* cunw;
  const int* cstart;
  const int* catoms;
  float rcf2;
  double rc2;
  float rpf2, band;
  // LIST: the groups that hold atoms (ACE rows: queued atoms); with more than list_max of them,
  // thinly filled then, another kernel builds the rows (k_build_thin, k_build_ace)
  const int* groups;
  const int* n_list;
  int list_max;
  // ACE rows only: the queue position of every atom (-1: none), the atoms' own shadows, the
  // stencil's half-width and the atoms' displacement since the cells were built (build_row_warp)
  const int* qpos;
  const float4* s32;
  int sten, n_groups;
  float margin;
  int cap;
  int* nbr;
  int* off;
  int* cnt;
  int* nin;
  DevScalars* sc;
};

// The exact decision for a candidate in the guard band around the cutoff, at cell offset o
// (pack_off) of atom i if `stored`, else at the one that follows from the two atoms' cells.
// Out of line: hardly any pair comes here.
__device__ __noinline__ bool decide(const BuildArgs& A, const SysInfo& S, int i, int j, int o, bool stored) {
  const int4 ci = A.cunw[i], cj = A.cunw[j];
  const int cw[3] = {cell_x(ci.w), cell_y(ci.w), cell_z(ci.w)}, cv[3] = {cell_x(cj.w), cell_y(cj.w), cell_z(cj.w)};
  const int ko[3] = {off_x(o), off_y(o), off_z(o)};
  int img[3];
  for (int d = 0; d < 3; ++d) {
    const int k = stored ? ko[d] : wrap_off(cv[d] - cw[d], S.nc[d], S.periodic[d]);
    img[d] = S.periodic[d] ? floor_div(cw[d] + k, S.nc[d]) : 0;
  }
  return exact_within(A.x, S, i, j, ci, cj, img, A.rc2);
}

__device__ inline float warp_min(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ inline float warp_max(float v) { return -warp_min(-v); }

#ifndef AP_BUILD_MINB
#define AP_BUILD_MINB 4   // resident blocks per SM the row build is compiled for (registers)
#endif
// STORED: the box is narrower than five cells in a periodic dimension and rows carry the cell
// offsets; otherwise they follow from the two atoms' cells.
// ACE: the rows of the queued atoms, in queue order, at the ACE radius (no split).
// LIST: the groups that hold atoms (queued ones) come from a list, several to a block; one block
// per group otherwise.
template <bool STORED, bool ACE, bool LIST = ACE>
__global__ void __launch_bounds__(kBuildWarps * 32, AP_BUILD_MINB)
    k_build_rows(const __grid_constant__ BuildArgs A) {
  constexpr int T = kBuildWarps * 32;
  __shared__ float4 s_pos[kStage];                      // position relative to the group's first cell, atom index
  __shared__ int s_cell[STORED ? kStage : 1];           // cell relative to the group's first cell (pack_off)
  __shared__ unsigned short s_list[kBuildWarps][kList<ACE>];
  __shared__ int s_beg[T], s_pre[T + 1], s_run[T];      // runs: first slot, candidates before, cell (pack_off) and image
  __shared__ int s_sum[kBuildWarps + 1];
  __shared__ int s_own[ACE ? kBuildWarps : 1][ACE ? 32 : 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int sten = ACE ? A.sten : kStencil;
  const float margin = ACE ? A.margin : 0.f;
  const int n_work = LIST ? *A.n_list : A.n_groups;
  if (LIST && n_work > A.list_max) return;
  for (int item = blockIdx.x; item < n_work; item += gridDim.x) {
    const int group_id = LIST ? A.groups[item] : item;
    __syncthreads();   // the shared arrays of the last item
    // the system and the group of cells
    int sys = 0;
    for (int lo = 0, hi = A.n_sys - 1; lo <= hi;) {
      const int mid = (lo + hi) >> 1;
      if (A.sys[mid].grp_base <= group_id) {
        sys = mid;
        lo = mid + 1;
      } else {
        hi = mid - 1;
      }
    }
    const SysInfo& S = A.sys[sys];
    const int nx = S.nc[0], ny = S.nc[1], nz = S.nc[2];
    const float hx = S.hf[0], hy = S.hf[1], hz = S.hf[2];
    const int gx = (nx + A.group - 1) / A.group, gy = (ny + A.group - 1) / A.group;
    const int gid = group_id - S.grp_base;
    const int x0 = gid % gx * A.group, y0 = gid / gx % gy * A.group, z0 = gid / (gx * gy) * A.group;
    const int mx = min(A.group, nx - x0), my = min(A.group, ny - y0), mz = min(A.group, nz - z0);
    const float reach2 = A.rcf2 + A.band, r_sure = A.rcf2 - A.band;
    // r_sure is rounded and may lie further from rcf2 than the guard band: the exact decision takes
    // every pair that is not surely inside (the difference itself is exact)
    const float band = fmaxf(A.band, A.rcf2 - r_sure);
    // this warp's cell of the group, or its share of the single cell's atoms
    const int parts = A.group == 1 ? kBuildWarps : 1, part = A.group == 1 ? warp : 0;
    const int wx = warp & 1, wy = (warp >> 1) & 1, wz = warp >> 2;
    int b = 0, own = 0, ux = 0, uy = 0, uz = 0;
    if (A.group == 1 || (wx < mx && wy < my && wz < mz)) {
      if (A.group != 1) {
        ux = wx;
        uy = wy;
        uz = wz;
      }
      const int cell = S.cell_base + ((z0 + uz) * ny + y0 + uy) * nx + x0 + ux;
      b = A.cstart[cell];
      own = max(0, (A.cstart[cell + 1] - b - part + parts - 1) / parts);   // atoms part, part + parts, ...
    }
    // ---- the runs of the group's stencil: pencil (dy, dz), periodic image ix along x.  Cells are
    // cut at the reach plus the margin of the group's box grown by the margin.
    const int py = my + 2 * sten, pz = mz + 2 * sten;
    const int ix_lo = S.periodic[0] ? floor_div(x0 - sten, nx) : 0;
    const int n_im = S.periodic[0] ? floor_div(x0 + mx - 1 + sten, nx) - ix_lo + 1 : 1;
    const int n_runs = py * pz * n_im;   // at most T: 36 x 5 for the EAM stencil; launch_build_ace checks
    const float blo = -margin - 1e-3f;
    const float gxh = (float)mx * hx - blo, gyh = (float)my * hy - blo, gzh = (float)mz * hz - blo;
    const float prune = sqrtf(A.rcf2) + margin, prune2 = prune * prune + A.band;
    int len = 0;
    if (threadIdx.x < n_runs) {
      const int pen = threadIdx.x / n_im, ix = ix_lo + threadIdx.x - pen * n_im;
      const int dz = pen / py - sten, dy = pen % py - sten;
      int ty = y0 + dy, tz = z0 + dz;
      bool valid = true;
      if (S.periodic[1]) ty -= floor_div(ty, ny) * ny;
      else valid = valid && ty >= 0 && ty < ny;
      if (S.periodic[2]) tz -= floor_div(tz, nz) * nz;
      else valid = valid && tz >= 0 && tz < nz;
      const float ay = fmaxf(0.f, fmaxf((float)dy * hy - gyh, blo - (float)(dy + 1) * hy));
      const float az = fmaxf(0.f, fmaxf((float)dz * hz - gzh, blo - (float)(dz + 1) * hz));
      const float left = prune2 - ay * ay - az * az;
      if (valid && left >= 0.f) {
        const float ax = sqrtf(left) + 2e-3f;   // cells that the reach along x touches, slack for the division
        const int c0 = max(max(-sten, (int)floorf((blo - ax) / hx)) + x0 - ix * nx, 0);
        const int c1 = min(min(mx - 1 + sten, (int)floorf((gxh + ax) / hx)) + x0 - ix * nx, nx - 1);
        if (c0 <= c1) {
          const int row0 = S.cell_base + (tz * ny + ty) * nx;
          const int beg = A.cstart[row0 + c0];
          len = A.cstart[row0 + c1 + 1] - beg;
          s_beg[threadIdx.x] = beg;
          s_run[threadIdx.x] = pack_off(0, dy, dz) | (ix - ix_lo) << 24;
        }
      }
    }
    int pre = len;   // inclusive scan of the lengths over the block
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, pre, o);
      if (lane >= o) pre += v;
    }
    if (lane == 31) s_sum[warp] = pre;
    __syncthreads();
    if (warp == 0) {
      int v = lane < kBuildWarps ? s_sum[lane] : 0;
#pragma unroll
      for (int o = 1; o < kBuildWarps; o <<= 1) {
        const int w = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += w;
      }
      if (lane < kBuildWarps) s_sum[lane] = v;
    }
    __syncthreads();
    const int total = s_sum[kBuildWarps - 1];
    s_pre[threadIdx.x + 1] = pre + (warp ? s_sum[warp - 1] : 0);
    if (threadIdx.x == 0) s_pre[0] = 0;
    __syncthreads();
    if (total == 0) {   // no atom in the group either
      if constexpr (LIST) continue;
      else return;
    }

    // ---- rounds: stage candidates (ordered), then test them against every warp's atoms
    int at = 0, staged = 0;   // uniform over the block
    bool first_round = true;
    while (true) {
      bool full = false;
      while (at < total) {
        const int f = at + threadIdx.x;
        bool keep = false;
        float px = 0.f, py_ = 0.f, pz_ = 0.f;
        int j = 0, ko = 0;
        if (f < total) {
          int lo = 0, hi = n_runs - 1;   // the run of candidate f: the last one with s_pre <= f
          while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_pre[mid] <= f) lo = mid;
            else hi = mid - 1;
          }
          const int slot = s_beg[lo] + f - s_pre[lo], o = s_run[lo];
          j = A.catoms[slot];
          const float4 sj = ACE ? A.s32[j] : A.s32c[slot];
          const int kx = cell_x(__float_as_int(sj.w)) + (ix_lo + (o >> 24)) * nx - x0;
          ko = (o & 0xffffff) + kx;
          px = fmaf((float)kx, hx, sj.x);
          py_ = fmaf((float)off_y(o), hy, sj.y);
          pz_ = fmaf((float)off_z(o), hz, sj.z);
          const float ax = fmaxf(0.f, fmaxf(blo - px, px - gxh)), ay = fmaxf(0.f, fmaxf(blo - py_, py_ - gyh)),
                      az = fmaxf(0.f, fmaxf(blo - pz_, pz_ - gzh));
          keep = ax * ax + ay * ay + az * az <= reach2;
        }
        const unsigned mk = __ballot_sync(0xffffffffu, keep);
        __syncthreads();
        if (lane == 0) s_sum[warp] = __popc(mk);
        __syncthreads();
        int before = 0, sum = 0;
#pragma unroll
        for (int w = 0; w < kBuildWarps; ++w) {
          const int v = s_sum[w];
          before += w < warp ? v : 0;
          sum += v;
        }
        if (staged + sum > kStage) {   // uniform: no room, test what is staged first
          full = true;
          break;
        }
        if (keep) {
          const int q = staged + before + __popc(mk & lt);
          s_pos[q] = make_float4(px, py_, pz_, __int_as_float(j));
          if (STORED) s_cell[q] = ko;
        }
        staged += sum;
        at += T;
      }
      __syncthreads();
      for (int c0 = 0; c0 < own; c0 += 32) {   // up to 32 of the warp's atoms, one per lane
        int nc = min(32, own - c0);
        int slot = b + part + (c0 + min(lane, nc - 1)) * parts;
        if constexpr (ACE) {   // the queued ones of them
          const unsigned queued = __ballot_sync(0xffffffffu, lane < nc && A.qpos[A.catoms[slot]] >= 0);
          if (!queued) continue;
          if (queued >> lane & 1) s_own[warp][__popc(queued & lt)] = slot;
          nc = __popc(queued);
          __syncwarp();
          slot = s_own[warp][min(lane, nc - 1)];
          __syncwarp();
        }
        const int me_i = A.catoms[slot];
        const int me_row = ACE ? A.qpos[me_i] : me_i;
        const float4 sm = ACE ? A.s32[me_i] : A.s32c[slot];
        const float mex = fmaf((float)ux, hx, sm.x), mey = fmaf((float)uy, hy, sm.y), mez = fmaf((float)uz, hz, sm.z);
        int n_in = 0, n_skin = 0;   // entries found so far for this lane's atom
        if (!first_round) {
          n_in = ACE ? A.cnt[me_row] : A.nin[me_row];
          n_skin = ACE ? 0 : A.cnt[me_row];
        }
        const float xlo = warp_min(mex), xhi = warp_max(mex), ylo = warp_min(mey), yhi = warp_max(mey),
                    zlo = warp_min(mez), zhi = warp_max(mez);
        unsigned short* const list = s_list[warp];
        int from = 0;
        bool first = first_round && !full, direct = false;
        do {
          // list the staged candidates within reach of this warp's atoms
          int listed = 0;
          while (from < staged) {
            const int t = from + lane;
            bool keep = false;
            if (t < staged) {
              const float4 p = s_pos[t];
              const float ax = fmaxf(0.f, fmaxf(xlo - p.x, p.x - xhi)), ay = fmaxf(0.f, fmaxf(ylo - p.y, p.y - yhi)),
                          az = fmaxf(0.f, fmaxf(zlo - p.z, p.z - zhi));
              keep = fmaf(ax, ax, fmaf(ay, ay, az * az)) <= reach2;
            }
            const unsigned mk = __ballot_sync(0xffffffffu, keep);
            if (listed + __popc(mk) > kList<ACE>) break;
            if (keep) list[listed + __popc(mk & lt)] = (unsigned short)t;
            listed += __popc(mk);
            from += 32;
          }
          __syncwarp();
          direct = first && from >= staged;   // all candidates are in the list: rows are written in place
          first = false;
          // lane t takes candidates K t .. K t + K - 1 of the list
          const int K = (listed + 31) >> 5, base = K * lane, nk = min(K, listed - base);
          for (int u0 = 0; u0 < nc; u0 += kCentres) {
            float cx[kCentres], cy[kCentres], cz[kCentres];
            int ci[kCentres];
            unsigned m[kCentres];   // bit k: candidate k is inside r_c; bit 16 + k: in the skin
#pragma unroll
            for (int u = 0; u < kCentres; ++u) {
              const int src = min(u0 + u, nc - 1);
              cx[u] = __shfl_sync(0xffffffffu, mex, src);
              cy[u] = __shfl_sync(0xffffffffu, mey, src);
              cz[u] = __shfl_sync(0xffffffffu, mez, src);
              ci[u] = __shfl_sync(0xffffffffu, me_i, src);
              m[u] = 0;
            }
            for (int k = 0; k < nk; ++k) {
              const float4 p = s_pos[list[base + k]];
              const unsigned b_in = 1u << k, b_sk = 0x10000u << k;
#pragma unroll
              for (int u = 0; u < kCentres; ++u) {
                const float dx = p.x - cx[u], dy = p.y - cy[u], dz = p.z - cz[u];
                const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
                const unsigned bit = r2 < A.rpf2 ? b_in : b_sk;
                if (r2 < r_sure) m[u] |= bit;
                if (fabsf(r2 - A.rcf2) <= band || r2 < 1e-6f) {
                  const int j = __float_as_int(p.w);
                  const int o = STORED ? s_cell[list[base + k]] - (pack_off(ux, uy, uz) - pack_off(0, 0, 0)) : 0;
                  if (r2 < 1e-6f && j == ci[u] && (!STORED || o == pack_off(0, 0, 0))) {
                    m[u] &= ~bit;   // the atom itself
                  } else if (fabsf(r2 - A.rcf2) <= band) {
                    m[u] &= ~bit;
                    if (decide(A, S, ci[u], j, o, STORED)) m[u] |= bit;
                  }
                }
              }
            }
            __syncwarp();
#pragma unroll
            for (int u = 0; u < kCentres; ++u) {
              if (u0 + u >= nc) break;
              const int cnt = __popc(m[u] & 0xffffu) | (__popc(m[u] >> 16) << 16);
              int sum = cnt;   // inclusive scan of both counts
#pragma unroll
              for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, sum, o);
                if (lane >= o) sum += v;
              }
              const int tot = __shfl_sync(0xffffffffu, sum, 31);
              const int ni = __shfl_sync(0xffffffffu, n_in, u0 + u), ns = __shfl_sync(0xffffffffu, n_skin, u0 + u);
              sum -= cnt;
              // in-range entries fill the row from the front; skin entries from the row's end, or,
              // while more candidates are to come, from the end of its capacity
              int q_in = ni + (sum & 0xffff);
              int q_sk = (direct ? ni + (tot & 0xffff) + ns + (tot >> 16) : A.cap) - 1 - ns - (sum >> 16);
              const size_t row = (size_t)(ACE ? __shfl_sync(0xffffffffu, me_row, u0 + u) : ci[u]) * A.cap;
              unsigned bits = m[u];
              while (bits) {
                const int k = __ffs(bits) - 1;
                bits &= bits - 1;
                const int q = k < 16 ? q_in++ : q_sk--;
                if (q >= 0 && q < A.cap) {
                  const int t = list[base + (k & 15)];
                  A.nbr[row + q] = __float_as_int(s_pos[t].w);
                  if (STORED) A.off[row + q] = s_cell[t] - (pack_off(ux, uy, uz) - pack_off(0, 0, 0));
                }
              }
              if (lane == u0 + u) {
                n_in = ni + (tot & 0xffff);
                n_skin = ns + (tot >> 16);
              }
            }
          }
          __syncwarp();
        } while (from < staged);
        if (full) {   // another round follows
          if (lane < nc) {
            if (!ACE) A.nin[me_row] = n_in;
            A.cnt[me_row] = ACE ? n_in : n_skin;
          }
          continue;
        }
        // rows of more than one turn: the skin entries move from [cap - n_skin, cap) to [n_in, cnt),
        // each run of 32 read in full before it is written; its destinations lie below every source
        // of the later runs.  An overflowing row holds cap valid entries (the capacity error makes
        // the caller rebuild or fail before any result is used).
        const int cnt = n_in + n_skin;
        for (int u = 0; !ACE && !direct && u < nc; ++u) {
          const int i = __shfl_sync(0xffffffffu, me_i, u), ni = __shfl_sync(0xffffffffu, n_in, u),
                    ns = __shfl_sync(0xffffffffu, n_skin, u);
          if (ni + ns >= A.cap) continue;
          for (int which = 0; which < (STORED ? 2 : 1); ++which) {
            int* r = (which ? A.off : A.nbr) + (size_t)i * A.cap;
            for (int k0 = 0; k0 < ns; k0 += 32) {
              const int k = k0 + lane;
              const int v = k < ns ? r[A.cap - ns + k] : 0;
              __syncwarp();
              if (k < ns) r[ni + k] = v;
            }
          }
        }
        if (lane < nc) {
          A.cnt[me_row] = min(cnt, A.cap);
          if constexpr (!ACE)
            A.nin[me_row] = min(n_in, A.cap);   // the in-range part (read by the CSP on rows built at its positions)
          else if (min(cnt, A.cap) > __ldcg(&A.sc->ace_row_max))   // only a new maximum takes the (same-address) atomic
            atomicMax(&A.sc->ace_row_max, min(cnt, A.cap));
          if (cnt > A.cap) {
            atomicMax(ACE ? &A.sc->need_ace : &A.sc->need_eam, cnt);
            atomicOr(&A.sc->err, kErrCapacity);
          }
        }
      }
      if (!full) break;
      first_round = false;
      staged = 0;
      __syncthreads();   // the stage is refilled
    }
    if constexpr (!LIST) return;   // one block per group
  }
}

// EAM rows where a group of cells holds a few atoms only (a dilute gas): one thread per row, in cell
// order, with the row order of k_build_rows.  In-range entries fill the row from the front, skin
// entries from the end of its capacity, and the gap is closed at the end.  Only if the list of groups
// is longer than list_max.
__global__ void __launch_bounds__(128, 9) k_build_thin(int n, const int* __restrict__ atom_sys,
                                                       const __grid_constant__ BuildArgs A) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n || *A.n_list <= A.list_max) return;
  const int i = A.catoms[t];
  const SysInfo& S = sys_of(A.sys, atom_sys, i);
  const float4 si = A.s32[i];
  const int4 ci = A.cunw[i];
  const int cw[3] = {cell_x(ci.w), cell_y(ci.w), cell_z(ci.w)};
  const float reach2 = A.rcf2 + A.band, r_sure = A.rcf2 - A.band;
  int* const row = A.nbr + (size_t)i * A.cap;
  int* const offrow = A.off ? A.off + (size_t)i * A.cap : nullptr;
  int n_in = 0, n_skin = 0;
  for (int dz = -kStencil; dz <= kStencil; ++dz) {
    int tz = cw[2] + dz, iz = 0;
    if (S.periodic[2]) {
      iz = floor_div(tz, S.nc[2]);
      tz -= iz * S.nc[2];
    } else if (tz < 0 || tz >= S.nc[2]) {
      continue;
    }
    const float oz = (float)dz * S.hf[2] - si.z, gz = fmaxf(0.f, fmaxf(oz, -oz - S.hf[2]));
    for (int dy = -kStencil; dy <= kStencil; ++dy) {
      int ty = cw[1] + dy, iy = 0;
      if (S.periodic[1]) {
        iy = floor_div(ty, S.nc[1]);
        ty -= iy * S.nc[1];
      } else if (ty < 0 || ty >= S.nc[1]) {
        continue;
      }
      const float oy = (float)dy * S.hf[1] - si.y, gy = fmaxf(0.f, fmaxf(oy, -oy - S.hf[1]));
      if (gz * gz + gy * gy > reach2) continue;
      const int row0 = S.cell_base + (tz * S.nc[1] + ty) * S.nc[0];
      for (int dx = -kStencil; dx <= kStencil; ++dx) {
        int tx = cw[0] + dx, ix = 0;
        if (S.periodic[0]) {
          ix = floor_div(tx, S.nc[0]);
          tx -= ix * S.nc[0];
        } else if (tx < 0 || tx >= S.nc[0]) {
          continue;
        }
        const float ox = (float)dx * S.hf[0] - si.x, gx = fmaxf(0.f, fmaxf(ox, -ox - S.hf[0]));
        if (gz * gz + gy * gy + gx * gx > reach2) continue;
        const int b = A.cstart[row0 + tx], e = A.cstart[row0 + tx + 1];
        for (int a = b; a < e; ++a) {
          if (a == t && dx == 0 && dy == 0 && dz == 0) continue;   // the atom itself
          const float4 sj = A.s32c[a];
          const int j = A.catoms[a];
          const float ddx = ox + sj.x, ddy = oy + sj.y, ddz = oz + sj.z;
          const float r2 = ddx * ddx + ddy * ddy + ddz * ddz;
          if (r2 > reach2) continue;
          if (!(r2 < r_sure)) {
            const int img[3] = {ix, iy, iz};
            if (!exact_within(A.x, S, i, j, ci, A.cunw[j], img, A.rc2)) continue;
          }
          const bool in = r2 < A.rpf2;
          if (n_in + n_skin < A.cap) {
            const int pos = in ? n_in : A.cap - 1 - n_skin;
            row[pos] = j;
            if (offrow) offrow[pos] = pack_off(dx, dy, dz);
          }
          n_in += in ? 1 : 0;
          n_skin += in ? 0 : 1;
        }
      }
    }
  }
  const int cnt = n_in + n_skin;
  if (cnt < A.cap)   // destinations lie below every later source
    for (int k = 0; k < n_skin; ++k) {
      row[n_in + k] = row[A.cap - n_skin + k];
      if (offrow) offrow[n_in + k] = offrow[A.cap - n_skin + k];
    }
  A.cnt[i] = min(cnt, A.cap);
  A.nin[i] = min(n_in, A.cap);
  if (cnt > A.cap) {
    atomicMax(&A.sc->need_eam, cnt);
    atomicOr(&A.sc->err, kErrCapacity);
  }
}

// The list of the cell groups with queued atoms (in any order: it only orders the work), and
// qpos[i] = queue position of atom i (the others hold -1).  flag: one int per group, 0.  A null
// queue stands for all n atoms (no qpos then).
__global__ void k_queue_groups(int n, const int* __restrict__ queue, const int* __restrict__ nq,
                               const SysInfo* __restrict__ sys, const int* __restrict__ atom_sys,
                               const int4* __restrict__ cunw, int group, int* __restrict__ qpos,
                               int* __restrict__ flag, int* __restrict__ list, int* __restrict__ n_list) {
  const int m = queue ? *nq : n;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < m; q += gridDim.x * blockDim.x) {
    const int i = queue ? queue[q] : q;
    if (queue) qpos[i] = q;
    const SysInfo& S = sys_of(sys, atom_sys, i);
    const int w = cunw[i].w;
    const int gx = (S.nc[0] + group - 1) / group, gy = (S.nc[1] + group - 1) / group;
    const int g = S.grp_base + (cell_z(w) / group * gy + cell_y(w) / group) * gx + cell_x(w) / group;
    if (flag[g] == 0 && atomicExch(&flag[g], 1) == 0) list[atomicAdd(n_list, 1)] = g;
  }
}

// FP32 shadows in cell order (s32c[a] = s32[catoms[a]]), for the EAM row build.
__global__ void k_shadow_cells(int n, const int* __restrict__ catoms, const float4* __restrict__ s32,
                               float4* __restrict__ s32c) {
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a < n) s32c[a] = s32[catoms[a]];
}

__global__ void __launch_bounds__(256) k_build_ace(const int* __restrict__ queue, const int* __restrict__ nq,
                                                   const double* __restrict__ x, const SysInfo* __restrict__ sys,
                                                   const int* __restrict__ atom_sys, const float4* __restrict__ s32,
                                                   const int4* __restrict__ cunw, const int* __restrict__ cstart,
                                                   const int* __restrict__ catoms, float rcf2, double rc2,
                                                   float band, int cap, int* __restrict__ nbr, int* __restrict__ off,
                                                   int* __restrict__ cnt, DevScalars* sc, int sten, float margin,
                                                   const int* __restrict__ n_list, int list_max) {
  __shared__ int4 s_buf[8][64];   // per warp: the stencil cells queued for the walk
  if (n_list && *n_list <= list_max) return;   // k_build_rows has built them
  const int wib = threadIdx.x >> 5;
  const int m = *nq;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  for (int q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < m; q += warps) {
    const int i = queue[q];
    const SysInfo& S = sys_of(sys, atom_sys, i);
    const int c = build_row_warp(i, x, S, s32, cunw, cstart, catoms, rcf2, rc2, band, cap, nbr + (size_t)q * cap,
                                 off ? off + (size_t)q * cap : nullptr, sten, margin, s_buf[wib]);
    if ((threadIdx.x & 31) == 0) {
      cnt[q] = c < cap ? c : cap;
      const int kept_c = c < cap ? c : cap;   // only a new maximum takes the (same-address) atomic
      if (kept_c > __ldcg(&sc->ace_row_max)) atomicMax(&sc->ace_row_max, kept_c);
      if (c > cap) {
        atomicMax(&sc->need_ace, c);
        atomicOr(&sc->err, kErrCapacity);
      }
    }
  }
}

// Export: entry (j, k) -> image s relative to the build positions.
__global__ void k_export(int rows, int cap_in, int cap_out, const int* __restrict__ row_atom,
                         const int* __restrict__ nbr, const int* __restrict__ off, const int* __restrict__ cnt_in,
                         const SysInfo* __restrict__ sys, const int* __restrict__ atom_sys,
                         const int4* __restrict__ cunw, int* __restrict__ cnt_out, int* __restrict__ idx_out,
                         int* __restrict__ shift_out) {
  int r = blockIdx.x;
  if (r >= rows) return;
  int i = row_atom ? row_atom[r] : r;
  const SysInfo& S = sys_of(sys, atom_sys, i);
  int c = cnt_in[r];
  if (threadIdx.x == 0) cnt_out[r] = c < cap_out ? c : cap_out;
  int4 ci = cunw[i];
  for (int q = threadIdx.x; q < c && q < cap_out; q += blockDim.x) {
    int j = nbr[(size_t)r * cap_in + q];
    int4 cj = cunw[j];
    int k[3];
    if (off) {
      int p = off[(size_t)r * cap_in + q];
      k[0] = off_x(p);
      k[1] = off_y(p);
      k[2] = off_z(p);
    } else {
      k[0] = wrap_off(cell_x(cj.w) - cell_x(ci.w), S.nc[0], S.periodic[0]);
      k[1] = wrap_off(cell_y(cj.w) - cell_y(ci.w), S.nc[1], S.periodic[1]);
      k[2] = wrap_off(cell_z(cj.w) - cell_z(ci.w), S.nc[2], S.periodic[2]);
    }
    int cu_i[3] = {ci.x, ci.y, ci.z}, cu_j[3] = {cj.x, cj.y, cj.z};
    idx_out[(size_t)r * cap_out + q] = j;
    for (int d = 0; d < 3; ++d) {
      int sd = 0;
      if (S.periodic[d]) sd = (k[d] - (cu_j[d] - cu_i[d])) / S.nc[d];
      shift_out[((size_t)r * cap_out + q) * 3 + d] = sd;
    }
  }
}

inline int nblk(int64_t n, int t) { return (int)((n + t - 1) / t); }

}  // namespace

size_t scan_tmp_bytes(int n) { return sizeof(int) * ((size_t)n / 512 + 256); }

int scan_exclusive(const int* d_in, int* d_out, int n, int* d_tmp, cudaStream_t s) {
  return scan_rec(d_in, n, d_out, n + 1, d_tmp, s);
}

void launch_wrap_positions(ap_ctx* c, double* d_x, cudaStream_t s) {
  k_wrap<<<nblk(c->n, 256), 256, 0, s>>>((int)c->n, d_x, c->d_sys, c->d_atom_sys);
  c->kernels += 1;
}

void launch_bin(ap_ctx* c, const double* d_x, const int32_t* d_species, cudaStream_t s) {
  cudaMemsetAsync(c->d_cell_count, 0, sizeof(int) * (size_t)c->n_cells, s);
  k_bin<<<nblk(c->n, 256), 256, 0, s>>>((int)c->n, d_x, d_species, c->d_sys, c->d_atom_sys, c->d_cell, c->d_slot,
                                        c->d_cunw, c->d_cell_count, c->d_org, c->d_sh32,
                                        c->cfg.precision == AP_PREC_FP64 ? c->d_sh64 : nullptr, c->d_sh32b, c->d_sc);
  c->kernels += 1;
}

void launch_cell_sort(ap_ctx* c, cudaStream_t s) {
  c->kernels += 2 + scan_exclusive(c->d_cell_count, c->d_cell_start, c->n_cells, c->d_scan_tmp, s);
  k_cell_scatter<<<nblk(c->n, 256), 256, 0, s>>>((int)c->n, c->d_cell, c->d_slot, c->d_cell_start, c->d_cell_atoms);
  k_cell_sort<<<nblk(c->n_cells, 128), 128, 0, s>>>(c->n_cells, c->d_cell_start, c->d_cell_atoms);
}

void launch_shadow(ap_ctx* c, const double* d_x, cudaStream_t s) {
  k_shadow<<<nblk(c->n, 256), 256, 0, s>>>((int)c->n, d_x, c->d_sys, c->d_atom_sys, c->d_org, c->d_cunw, c->d_sh32,
                                           c->cfg.precision == AP_PREC_FP64 ? c->d_sh64 : nullptr);
  c->kernels += 1;
}

static constexpr float kBand = 1e-3f;   // guard band on r^2 (A^2) around the cutoff

// Sum of the row counts (block sums, one 64-bit atomic per block).
__global__ void k_row_total(int rows, const int* __restrict__ cnt, unsigned long long* __restrict__ out) {
  __shared__ unsigned long long part[8];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long v = i < rows ? (unsigned long long)cnt[i] : 0ull;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long s = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += part[w];
    atomicAdd(out, s);
  }
}

void launch_row_total(ap_ctx* c, int which, int rows, cudaStream_t s) {
  cudaMemsetAsync(&c->d_sc->row_total, 0, sizeof(unsigned long long), s);
  if (rows > 0)
    k_row_total<<<nblk(rows, 256), 256, 0, s>>>(
        rows, which == 0 ? c->d_cnt_eam : which == 1 ? c->d_cnt_ace : c->d_lim_eam, &c->d_sc->row_total);
}

void launch_build_eam(ap_ctx* c, const double* d_x, cudaStream_t s) {
  double r = c->cfg.eam_rc + c->cfg.skin;
  double rc2 = r * r;
  // the potential's own cutoff: rows are split at it (the Mishin rc may lie below eam_rc)
  const double rp = c->cfg.eam_type == AP_EAM_MISHIN ? c->cfg.eam_mishin[28] : c->cfg.eam_rc;
  c->split_rpf2 = (float)(rp * rp);
  k_shadow_cells<<<nblk(c->n, 256), 256, 0, s>>>((int)c->n, c->d_cell_atoms, c->d_sh32, c->d_sh32c);
  c->kernels += 1;
  BuildArgs A;
  A.x = d_x;
  A.sys = c->d_sys;
  A.n_sys = c->n_sys;
  A.group = c->build_group;
  A.s32c = c->d_sh32c;
  A.cunw = c->d_cunw;
  A.cstart = c->d_cell_start;
  A.catoms = c->d_cell_atoms;
  A.rcf2 = (float)rc2;
  A.rc2 = rc2;
  A.rpf2 = c->split_rpf2;
  A.band = kBand;
  A.cap = c->cap_eam;
  A.nbr = c->d_nbr_eam;
  A.off = c->stored_off ? c->d_off_eam : nullptr;
  A.cnt = c->d_cnt_eam;
  A.nin = c->d_lim_eam;
  A.sc = c->d_sc;
  A.qpos = A.groups = A.n_list = nullptr;
  A.list_max = 0;
  A.s32 = c->d_sh32;
  A.sten = kStencil;
  A.n_groups = c->n_groups;
  A.margin = 0.f;
  c->kernels += 1;
  // Fewer than 32 atoms a group on average (a crystal of copper's density fills one with 44): the
  // groups that hold atoms are listed first (about 8 us), since a block that finds its group empty
  // costs 4.3 ns, and the list's length decides.  A few thousand full groups in a large box are built
  // from the list (whole builds of 10,976 atoms in 400 A 0.63 -> 0.13 ms, of 108,000 in 800 A
  // 4.6 -> 0.34 ms); many groups, at 10 ns each however few their atoms, by a thread per row: a
  // gas of a tenth of the crystal's density, 1,000,000 atoms 2.8 -> 0.86 ms, 100,000 0.34 -> 0.19, but
  // 20,000 0.14 -> 0.18; a crystal of 0.6 of it, 1,000,000 atoms 1.44 -> 1.08 ms.  From 32 atoms a
  // group on a block per group is as fast or faster (1,000,000 atoms at 0.8: 1.30 and 1.35 ms).
  if (c->n_groups > 4096 && c->n < 32 * (int64_t)c->n_groups) {
    int* flag = c->d_cell_count;   // free after the cell sort, like d_slot; n_groups <= n_cells
    int* list = c->d_slot;
    int* n_list = &c->d_sc->n_row_groups;   // cleared by build_checked
    cudaMemsetAsync(flag, 0, sizeof(int) * (size_t)c->n_groups, s);
    k_queue_groups<<<std::min(c->num_sms * 4, nblk(c->n, 256)), 256, 0, s>>>(
        (int)c->n, nullptr, nullptr, c->d_sys, c->d_atom_sys, c->d_cunw, c->build_group, nullptr, flag, list, n_list);
    A.groups = list;
    A.n_list = n_list;
    A.list_max = 5000 + (int)c->n / 60;
    c->kernels += 1;
    auto build = c->stored_off ? k_build_rows<true, false, true> : k_build_rows<false, false, true>;
    build<<<std::min(c->n_groups, c->num_sms * AP_BUILD_MINB * 2), kBuildWarps * 32, 0, s>>>(A);
    if (std::min<int64_t>(c->n, c->n_groups) > A.list_max) {
      k_build_thin<<<nblk(c->n, 128), 128, 0, s>>>((int)c->n, c->d_atom_sys, A);
      c->kernels += 1;
    }
    return;
  }
  auto build = c->stored_off ? k_build_rows<true, false> : k_build_rows<false, false>;
  build<<<c->n_groups, kBuildWarps * 32, 0, s>>>(A);
}

void launch_build_ace(ap_ctx* c, const double* d_x, const int* d_queue, const int* d_nq, int m, bool unique,
                      cudaStream_t s) {
  const double r = c->cfg.ace_rc + c->cfg.skin;
  // Cells older than the positions (ap_step kept the EAM lists): the atoms moved up to
  // m = stale_m since the cell build, so a cell is pruned only beyond r + m and the
  // stencil reaches r + 2 m.  The rows stay complete while no atom moves more than skin/2
  // from its position at this build, which ap_step checks after every drift.
  int sten = kStencil;
  float margin = 0.f;
  if (c->cells_stale) {
    margin = (float)c->stale_m;
    for (const SysInfo& S : c->h_sys)
      for (int d = 0; d < 3; ++d) sten = std::max(sten, (int)std::ceil((r + 2.0 * c->stale_m) / S.h[d]));
  }
  double rc2 = r * r;
  // Cell groups, as for the EAM rows, for long queues in which every atom stands once, where the
  // stencil's runs fit a block's threads (k_build_rows: 255,840 atoms at 8 A 0.59 ms, a warp per
  // row 0.83; 240,000 of 4,000,000 at 7.7 A 0.76 and 0.97); a warp per row otherwise (12,700 atoms
  // 43 us, by groups 51 and the list 5; 83,000 in narrow boxes 0.267 and 0.266 ms), and where the
  // list shows that the queue is scattered over groups with fewer than 20 of its atoms (energies of
  // 500,000 atoms' random parts, by groups and by warps: 5.5 a group 0.86 and 0.61 ms, 18 a group 1.62
  // and 1.60, 26 a group 2.13 and 2.31).
  int runs = 0;
  for (const SysInfo& S : c->h_sys) {
    const int e = c->build_group + 2 * sten, im = S.periodic[0] ? (e + S.nc[0] - 1) / S.nc[0] + 1 : 1;
    runs = std::max(runs, e * e * im);
  }
  const int* listed = nullptr;
  const int list_max = m / 20;
  if (m >= 400 * c->num_sms && unique && runs <= kBuildWarps * 32) {
    int* flag = c->d_cell_count;   // free after the cell sort; n_groups <= n_cells
    int* list = c->d_slot;         // free after the cell sort; at most one group per atom
    int* n_list = &c->d_sc->n_row_groups;   // cleared by build_ace_checked
    cudaMemsetAsync(flag, 0, sizeof(int) * (size_t)c->n_groups, s);
    cudaMemsetAsync(c->d_qpos, 0xff, sizeof(int) * (size_t)c->n, s);
    k_queue_groups<<<c->num_sms * 4, 256, 0, s>>>((int)c->n, d_queue, d_nq, c->d_sys, c->d_atom_sys, c->d_cunw, c->build_group,
                                                  c->d_qpos, flag, list, n_list);
    BuildArgs A = {};
    A.x = d_x;
    A.sys = c->d_sys;
    A.n_sys = c->n_sys;
    A.group = c->build_group;
    A.cunw = c->d_cunw;
    A.cstart = c->d_cell_start;
    A.catoms = c->d_cell_atoms;
    A.rcf2 = (float)rc2;
    A.rc2 = rc2;
    A.rpf2 = 3.4e38f;   // no split
    A.band = kBand;
    A.qpos = c->d_qpos;
    A.groups = list;
    A.n_list = listed = n_list;
    A.list_max = list_max;
    A.s32 = c->d_sh32;
    A.sten = sten;
    A.margin = margin;
    A.cap = c->cap_ace;
    A.nbr = c->d_nbr_ace;
    A.off = c->stored_off ? c->d_off_ace : nullptr;
    A.cnt = c->d_cnt_ace;
    A.sc = c->d_sc;
    auto build = c->stored_off ? k_build_rows<true, true> : k_build_rows<false, true>;
    build<<<std::max(1, std::min(c->n_groups, c->num_sms * AP_BUILD_MINB * 2)), kBuildWarps * 32, 0, s>>>(A);
    c->kernels += 2;
    if (c->n_groups <= list_max) return;
  }
  int grid = c->num_sms * 8;
  k_build_ace<<<grid, 256, 0, s>>>(d_queue, d_nq, d_x, c->d_sys, c->d_atom_sys, c->d_sh32, c->d_cunw,
                                   c->d_cell_start, c->d_cell_atoms, (float)rc2, rc2, kBand, c->cap_ace,
                                   c->d_nbr_ace, c->stored_off ? c->d_off_ace : nullptr, c->d_cnt_ace, c->d_sc, sten,
                                   margin, listed, list_max);
  c->kernels += 1;
}

void launch_export_rows(ap_ctx* c, int which, int rows, int cap_out, int* d_cnt, int* d_idx, int* d_shift,
                        cudaStream_t s) {
  if (rows <= 0) return;
  if (which == 0)
    k_export<<<rows, 128, 0, s>>>(rows, c->cap_eam, cap_out, nullptr, c->d_nbr_eam,
                                  c->stored_off ? c->d_off_eam : nullptr, c->d_cnt_eam, c->d_sys, c->d_atom_sys,
                                  c->d_cunw, d_cnt, d_idx, d_shift);
  else
    k_export<<<rows, 128, 0, s>>>(rows, c->cap_ace, cap_out, c->d_precise, c->d_nbr_ace,
                                  c->stored_off ? c->d_off_ace : nullptr, c->d_cnt_ace, c->d_sys, c->d_atom_sys,
                                  c->d_cunw, d_cnt, d_idx, d_shift);
}

}  // namespace ap
