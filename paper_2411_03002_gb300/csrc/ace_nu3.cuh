// ACE kernel 2: nu = 3 energy and gradient of the atoms of the precise queue, as straight-line
// code over the merged monomials of the basis (ace_nu3.inc), with A and dE/dA in registers and
// the coefficients in the kernels' parameter space.  E3 follows from Euler's identity for a
// homogeneous cubic, E3 = (1/3) sum A dE3/dA.
// Finnis-Sinclair form (FS): a first pass gives the nu = 3 part of phi^(2), hence phi^(2), F and
// F'; the gradient pass then uses the coefficients c1 + F' c2, and E3 of phi^(1) is
// E3(c1 + F' c2) - F' E3(c2).
#pragma once

#include <algorithm>
#include <cstring>

#include "ace_args.cuh"

namespace ap {

namespace {

#include "ace_nu3.inc"

// nu = 3 coefficients, passed by value (kernel parameter space), in the order of kNu3Key; the
// ones of phi^(2) (second) only in the Finnis-Sinclair form.
template <typename R, bool FS>
struct Nu3Coef {
  R c[AP_NU3_N];
  __device__ R second(int) const { return R(0); }
};
template <typename R>
struct Nu3Coef<R, true> {
  R c[AP_NU3_N], c2[AP_NU3_N];
  __device__ R second(int t) const { return c2[t]; }
};

template <typename R>
__device__ inline void load48(const R* p, R A[48]) {   // rows of 48 entries: 4-wide loads
  const auto* src = reinterpret_cast<const typename V<R>::R4*>(p);
#pragma unroll
  for (int v = 0; v < 12; ++v) {
    const auto t = src[v];
    A[4 * v] = t.x;
    A[4 * v + 1] = t.y;
    A[4 * v + 2] = t.z;
    A[4 * v + 3] = t.w;
  }
}

// phi^(2) of an atom from its nu = 3 part -> F, F'
template <typename R>
__device__ inline void embed_fs(const AceArgs<R>& a, int q, double e3b, double& F, R& fp) {
  const double phi2 = a.e12b[q] + e3b;
  const double sq = sqrt(fabs(phi2) + a.fs_eps * a.fs_eps);
  F = phi2 > 0.0 ? sq - a.fs_eps : (phi2 < 0.0 ? a.fs_eps - sq : 0.0);
  fp = (R)(0.5 / sq);
}

#define NU3_GROUP_BEGIN(x, y) \
  {                           \
    const R p_ = A[x] * A[y]; \
    R s_ = R(0);
// the energy part of the phi^(2) pass (ENERGY), or the gradient
#define NU3_COEF(t) (FS ? fma(fp, P.second(t), P.c[t]) : P.c[t])
#define NU3_TERM(t, z)                          \
  if constexpr (ENERGY) {                       \
    s_ = fma(P.second(t), A[z], s_);            \
  } else {                                      \
    s_ = fma(NU3_COEF(t), A[z], s_);            \
    dA[z] = fma(NU3_COEF(t), p_, dA[z]);        \
  }
#define NU3_GROUP_END(x, y)       \
  if constexpr (ENERGY) {         \
    eb = fma(p_, s_, eb);         \
  } else {                        \
    dA[x] = fma(s_, A[y], dA[x]); \
    dA[y] = fma(s_, A[x], dA[y]); \
  }                               \
  }

template <int N>
struct Int {
  static constexpr int value = N;
};

// Part PART of the monomials (PART = -1: all of them).
template <typename R, bool FS, bool ENERGY, int PART>
__device__ __forceinline__ void nu3_body(const R A[48], R dA[48], R& eb, R fp, const Nu3Coef<R, FS>& P) {
  if constexpr (PART == -1) {
    AP_NU3_BODY
  } else if constexpr (PART == 0) {
    AP_NU3_BODY_0
  } else if constexpr (PART == 1) {
    AP_NU3_BODY_1
  } else if constexpr (PART == 2) {
    AP_NU3_BODY_2
  } else if constexpr (PART == 3) {
    AP_NU3_BODY_3
  } else if constexpr (PART == 4) {
    AP_NU3_BODY_4
  } else if constexpr (PART == 5) {
    AP_NU3_BODY_5
  } else if constexpr (PART == 6) {
    AP_NU3_BODY_6
  } else {
    AP_NU3_BODY_7
  }
}
#undef NU3_GROUP_BEGIN
#undef NU3_COEF
#undef NU3_TERM
#undef NU3_GROUP_END
static_assert(AP_NU3_PARTS == 8, "nu3_body and k_ace_nu3_parts take eight parts");

// Long queues (FP32): one lane per atom.  The body is 6,000 FMAs of straight-line code, so this
// takes 30 us (FP64: 235 us) however few the atoms are.
template <typename R, bool FS>
__global__ void __launch_bounds__(128) k_ace_nu3(AceArgs<R> a, const __grid_constant__ Nu3Coef<R, FS> P) {
  const int m = *a.count;
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.counter = *a.counter2 = 0;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < m; q += gridDim.x * blockDim.x) {
    R A[48], dA[48];
    load48(a.a48 + (size_t)q * 48, A);
#pragma unroll
    for (int v = 0; v < 48; ++v) dA[v] = R(0);
    R fp = R(0), eb = R(0), e = R(0);
    double F = 0.0;
    if constexpr (FS) {
      nu3_body<R, FS, true, -1>(A, dA, eb, fp, P);
      embed_fs(a, q, (double)eb, F, fp);
    }
    nu3_body<R, FS, false, -1>(A, dA, e, fp, P);
#pragma unroll
    for (int v = 0; v < 48; ++v) e = fma(A[v], dA[v], e);
    auto* dst = reinterpret_cast<typename V<R>::R4*>(a.de3 + (size_t)q * 48);
#pragma unroll
    for (int v = 0; v < 12; ++v) dst[v] = make_r4(dA[4 * v], dA[4 * v + 1], dA[4 * v + 2], dA[4 * v + 3]);
    a.e3[q] = (double)e * (1.0 / 3.0) - (FS ? (double)fp * (double)eb : 0.0);
    if (FS) {
      a.fs[2 * (size_t)q] = F;
      a.fs[2 * (size_t)q + 1] = (double)fp;
    }
  }
}

// Short queues: a block of 8 warps works on 32 atoms, each warp on an eighth of the monomials;
// the partial gradients are summed in shared memory in a fixed order.  The chain that one warp
// walks is an eighth, and there are 8 times as many warps.  Taken by FP64 always (1,365 atoms
// 235 -> 66 us, 12,700 atoms 236 -> 196 us) and by FP32 while the queue is one wave of its blocks,
// two per SM: 155 atoms 33 -> 14 us, but 12,700 atoms 28 us with a lane per atom against 32.
template <typename R, bool FS>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 2 : 1) k_ace_nu3_parts(AceArgs<R> a, const __grid_constant__ Nu3Coef<R, FS> P) {
  extern __shared__ __align__(32) unsigned char smem_raw[];
  R* part = reinterpret_cast<R*>(smem_raw);   // [8][48][32] partial gradients
  __shared__ R s_e[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int m = *a.count;
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.counter = *a.counter2 = 0;
  for (int q0 = blockIdx.x * 32; q0 < m; q0 += gridDim.x * 32) {
    const int q = q0 + lane;
    const R* src = a.a48 + (size_t)min(q, m - 1) * 48;
    R fp = R(0), eb = R(0);
    double F = 0.0;
    auto run = [&](auto part_c, auto energy_c) {
      constexpr int PART = decltype(part_c)::value;
      constexpr bool ENERGY = decltype(energy_c)::value;
      R A[48], dA[48];
      load48(src, A);
#pragma unroll
      for (int v = 0; v < 48; ++v) dA[v] = R(0);
      R e = R(0);
      nu3_body<R, FS, ENERGY, PART>(A, dA, e, fp, P);
      if (ENERGY) {
        s_e[PART][lane] = e;
      } else {
#pragma unroll
        for (int v = 0; v < 48; ++v) part[(PART * 48 + v) * 32 + lane] = dA[v];
      }
    };
    auto all_parts = [&](auto energy_c) {
      switch (warp) {
        case 0: run(Int<0>(), energy_c); break;
        case 1: run(Int<1>(), energy_c); break;
        case 2: run(Int<2>(), energy_c); break;
        case 3: run(Int<3>(), energy_c); break;
        case 4: run(Int<4>(), energy_c); break;
        case 5: run(Int<5>(), energy_c); break;
        case 6: run(Int<6>(), energy_c); break;
        default: run(Int<7>(), energy_c); break;
      }
    };
    if constexpr (FS) {
      all_parts(Int<1>());
      __syncthreads();
#pragma unroll
      for (int w = 0; w < 8; ++w) eb += s_e[w][lane];
      embed_fs(a, min(q, m - 1), (double)eb, F, fp);
      __syncthreads();
    }
    all_parts(Int<0>());
    __syncthreads();
    // warp w sums entries 6 w .. 6 w + 5 over the parts
    R e = R(0);
#pragma unroll
    for (int u = 0; u < 6; ++u) {
      const int v = 6 * warp + u;
      R s = part[v * 32 + lane];
#pragma unroll
      for (int w = 1; w < 8; ++w) s += part[(w * 48 + v) * 32 + lane];
      e = fma(src[v], s, e);
      if (q < m) a.de3[(size_t)q * 48 + v] = s;
    }
    s_e[warp][lane] = e;
    __syncthreads();
    if (warp == 0 && q < m) {
      R t = s_e[0][lane];
#pragma unroll
      for (int w = 1; w < 8; ++w) t += s_e[w][lane];
      a.e3[q] = (double)t * (1.0 / 3.0) - (FS ? (double)fp * (double)eb : 0.0);
      if (FS) {
        a.fs[2 * (size_t)q] = F;
        a.fs[2 * (size_t)q + 1] = (double)fp;
      }
    }
    __syncthreads();
  }
}

template <typename R>
constexpr size_t kPartBytes = sizeof(R) * 8 * 48 * 32;
#ifndef AP_NU3_LONG
#define AP_NU3_LONG 64   // atoms per SM from which FP32 queues take one lane per atom
#endif

template <typename R, bool FS>
void run_nu3(ap_ctx* c, const AceArgs<R>& a, int m, cudaStream_t s) {
  Nu3Coef<R, FS> P;
  const R* src;
  if constexpr (sizeof(R) == 4) src = c->ace.nu3_f32.data();
  else src = c->ace.nu3_coef.data();
  std::memcpy(P.c, src, sizeof(P.c));
  if constexpr (FS) std::memcpy(P.c2, sizeof(R) == 4 ? src + AP_NU3_N : (const R*)c->ace.nu3_coef2.data(), sizeof(P.c2));
  if constexpr (sizeof(R) == 4) {
    if (m >= AP_NU3_LONG * c->num_sms) {
      k_ace_nu3<R, FS><<<c->num_sms * 8, 128, 0, s>>>(a, P);
      return;
    }
  }
  cudaFuncSetAttribute(k_ace_nu3_parts<R, FS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPartBytes<R>);
  const int blocks = std::max(1, std::min((m + 31) / 32, c->num_sms * (sizeof(R) == 4 ? 4 : 2)));
  k_ace_nu3_parts<R, FS><<<blocks, 256, kPartBytes<R>, s>>>(a, P);
}

}  // namespace

template <typename R>
int launch_ace_nu3(ap_ctx* c, const AceArgs<R>& a, int m, cudaStream_t s) {
  if (c->cfg.ace_fs_on) run_nu3<R, true>(c, a, m, s);
  else run_nu3<R, false>(c, a, m, s);
  return 1;
}

}  // namespace ap
