// Arguments and small helpers shared by the ACE kernels (k_ace.cu, k_ace_nu3.cu).
#pragma once

#include "ap_internal.cuh"

namespace ap {

template <typename R>
struct V;
template <>
struct V<float> {
  using S4 = float4;
  using R4 = float4;
  static __device__ inline int code(const float4& s) { return __float_as_int(s.w); }
};
template <>
struct V<double> {
  using S4 = double4_32a;
  using R4 = double4_32a;
  static __device__ inline int code(const double4_32a& s) { return (int)s.w; }
};

__device__ inline float pack_j(int j, float) { return __int_as_float(j); }
__device__ inline double pack_j(int j, double) { return __longlong_as_double((long long)j); }
__device__ inline int unpack_j(float v) { return __float_as_int(v); }
__device__ inline float4 make_r4(float a, float b, float c, float d) { return make_float4(a, b, c, d); }
__device__ inline double4_32a make_r4(double a, double b, double c, double d) { return make_double4_32a(a, b, c, d); }
__device__ inline int unpack_j(double v) { return (int)__double_as_longlong(v); }

// Arguments of the three ACE kernels.  Scratch indexed by the queue position q
// carries the per-atom state from one kernel to the next.
template <typename R>
struct AceArgs {
  const int* queue;
  const int* count;        // queue length (device)
  DevScalars* stats;
  int* counter;
  int* counter2;
  const SysInfo* sys;
  const int* atom_sys;
  const typename V<R>::S4* sh;
  const int* nbr;
  const int* off;
  const int* cnt;
  int cap;
  const double* lam;
  const double* wgt;       // explicit weights w_i (NULL: w_i = 1 - lambda_i)
  const R* W;
  const R* M2;
  const R* C1;
  const R* M2b;      // phi^(2) tables of the Finnis-Sinclair form
  const R* C1b;
  const R* C1l;      // [16] what FP32 rounds off C1 and C1b
  R rc2, inv_rc, inv_n0;
  int mode;
  int fs_on;
  double fs_eps;
  double* e_prec;
  float4* facc32;
  double* facc64;
  unsigned long long* faccfix;   // fixed-point accumulator [n][3], or NULL (float atomics)
  typename V<R>::R4* list4;   // [q][rec] in-range (d, j) records in row order (kernel 1 -> 3)
  int rec;                    // record slots per queue position (>= every ACE row's length)
  int* nin;          // [q] their number
  R* a48;            // [q][48] A entries with n <= 2, l <= 3 (input of nu = 3)
  R* dA;             // [q][200] dE/dA of nu = 1, 2
  double* e12;       // [q] E of nu = 1, 2
  R* de3;            // [q][48] dE3/dA (Finnis-Sinclair form: of phi^(1) + F' phi^(2))
  double* e3;        // [q] E3 (of phi^(1))
  R* dAb;            // [q][200] dphi^(2)_12/dA                 (Finnis-Sinclair form only)
  double* e12b;      // [q] phi^(2)_12                          (Finnis-Sinclair form only)
  double* fs;        // [q][2] F(phi^(2)), F'(phi^(2))          (Finnis-Sinclair form only)
};

// Kernel 2 (k_ace_nu3.cu) for a queue of about m atoms; returns the number of kernels launched.
template <typename R>
int launch_ace_nu3(ap_ctx* c, const AceArgs<R>& a, int m, cudaStream_t s);

}  // namespace ap
