// lbpf_lattice.cuh -- lattices, storage codecs and the per-simulation descriptor.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

namespace lbpf {

// ---------------------------------------------------------------- lattices
// Table 1 (e_i) and Table 2 (w_i, A_i, B_i, e^2) of Sec. 3.4.
template <int Q>
struct Lat;

template <>
struct Lat<7> {
  static constexpr double e2 = 0.25;
  static constexpr bool has_y = true;  // links along the kernel's y axis (false: a 2D lattice in the xz plane)
  static constexpr int diag0 = 1;      // first index of the diagonal weight class (none: an axis index)
  __host__ __device__ static constexpr int cls(int i) { return i == 0 ? 0 : 1; }  // 0 rest, 1 axis, 2 diagonal
  __host__ __device__ static constexpr int ex(int i) { return i == 1 ? 1 : (i == 3 ? -1 : 0); }
  __host__ __device__ static constexpr int ey(int i) { return i == 2 ? 1 : (i == 4 ? -1 : 0); }
  __host__ __device__ static constexpr int ez(int i) { return i == 5 ? 1 : (i == 6 ? -1 : 0); }
  __host__ __device__ static constexpr int opp(int i) {
    return i == 0 ? 0 : (i == 1 ? 3 : (i == 2 ? 4 : (i == 3 ? 1 : (i == 4 ? 2 : (i == 5 ? 6 : 5)))));
  }
  __host__ __device__ static constexpr double w(int i) { return i == 0 ? 0.25 : 0.125; }
  __host__ __device__ static constexpr double B(int i) { return i == 0 ? -0.75 : 0.125; }
};

// The accessors are switch expressions so that, with the population loops
// unrolled, every lookup folds to an immediate.
template <>
struct Lat<15> {
  static constexpr double e2 = 1.0 / 3.0;
  static constexpr bool has_y = true;
  static constexpr int diag0 = 7;
  __host__ __device__ static constexpr int cls(int i) { return i == 0 ? 0 : (i <= 6 ? 1 : 2); }
  // e_0..e_6 as D3Q7, then the cube diagonals
  __host__ __device__ static constexpr int ex(int i) {
    switch (i) {
      case 1: case 7: case 10: case 11: case 14: return 1;
      case 3: case 8: case 9: case 12: case 13: return -1;
      default: return 0;
    }
  }
  __host__ __device__ static constexpr int ey(int i) {
    switch (i) {
      case 2: case 7: case 8: case 11: case 12: return 1;
      case 4: case 9: case 10: case 13: case 14: return -1;
      default: return 0;
    }
  }
  __host__ __device__ static constexpr int ez(int i) {
    switch (i) {
      case 5: case 7: case 8: case 9: case 10: return 1;
      case 6: case 11: case 12: case 13: case 14: return -1;
      default: return 0;
    }
  }
  __host__ __device__ static constexpr int opp(int i) {
    switch (i) {
      case 1: return 3; case 2: return 4; case 3: return 1; case 4: return 2; case 5: return 6; case 6: return 5;
      case 7: return 13; case 8: return 14; case 9: return 11; case 10: return 12;
      case 11: return 9; case 12: return 10; case 13: return 7; case 14: return 8;
      default: return 0;
    }
  }
  __host__ __device__ static constexpr double w(int i) {
    return i == 0 ? 2.0 / 9.0 : (i <= 6 ? 1.0 / 9.0 : 1.0 / 72.0);
  }
  __host__ __device__ static constexpr double B(int i) {
    return i == 0 ? -7.0 / 9.0 : (i <= 6 ? 1.0 / 9.0 : 1.0 / 72.0);
  }
};

template <>
struct Lat<19> {
  static constexpr double e2 = 1.0 / 3.0;
  static constexpr bool has_y = true;
  static constexpr int diag0 = 7;
  __host__ __device__ static constexpr int cls(int i) { return i == 0 ? 0 : (i <= 6 ? 1 : 2); }
  // e_0..e_6 as D3Q7, then the twelve edge diagonals
  __host__ __device__ static constexpr int ex(int i) {
    switch (i) {
      case 1: case 7: case 9: case 11: case 13: return 1;
      case 3: case 8: case 10: case 12: case 14: return -1;
      default: return 0;
    }
  }
  __host__ __device__ static constexpr int ey(int i) {
    switch (i) {
      case 2: case 7: case 8: case 15: case 17: return 1;
      case 4: case 9: case 10: case 16: case 18: return -1;
      default: return 0;
    }
  }
  __host__ __device__ static constexpr int ez(int i) {
    switch (i) {
      case 5: case 11: case 12: case 15: case 16: return 1;
      case 6: case 13: case 14: case 17: case 18: return -1;
      default: return 0;
    }
  }
  __host__ __device__ static constexpr int opp(int i) {
    switch (i) {
      case 1: return 3; case 2: return 4; case 3: return 1; case 4: return 2; case 5: return 6; case 6: return 5;
      case 7: return 10; case 8: return 9; case 9: return 8; case 10: return 7;
      case 11: return 14; case 12: return 13; case 13: return 12; case 14: return 11;
      case 15: return 18; case 16: return 17; case 17: return 16; case 18: return 15;
      default: return 0;
    }
  }
  __host__ __device__ static constexpr double w(int i) {
    return i == 0 ? 1.0 / 3.0 : (i <= 6 ? 1.0 / 18.0 : 1.0 / 36.0);
  }
  __host__ __device__ static constexpr double B(int i) {
    return i == 0 ? -2.0 / 3.0 : (i <= 6 ? 1.0 / 18.0 : 1.0 / 36.0);
  }
};
// Table 3 (e_i) and Table 4 (w_i, A_i, B_i, e^2) of Sec. 3.4: the 2D lattices.  A 2D
// grid (nx, ny) runs as a kernel grid (nx, 1, ny): the paper's y axis becomes the
// kernel's marching axis z, so ey() below is always 0 and ez() holds the paper's e_y.
// Population order and memory layout are unchanged (one kernel plane row per paper row).
template <>
struct Lat<5> {
  static constexpr double e2 = 1.0 / 3.0;
  static constexpr bool has_y = false;
  static constexpr int diag0 = 1;
  __host__ __device__ static constexpr int cls(int i) { return i == 0 ? 0 : 1; }
  __host__ __device__ static constexpr int ex(int i) { return i == 1 ? 1 : (i == 3 ? -1 : 0); }
  __host__ __device__ static constexpr int ey(int) { return 0; }
  __host__ __device__ static constexpr int ez(int i) { return i == 2 ? 1 : (i == 4 ? -1 : 0); }
  __host__ __device__ static constexpr int opp(int i) { return i == 0 ? 0 : (i <= 2 ? i + 2 : i - 2); }
  __host__ __device__ static constexpr double w(int i) { return i == 0 ? 1.0 / 3.0 : 1.0 / 6.0; }
  __host__ __device__ static constexpr double B(int i) { return i == 0 ? -2.0 / 3.0 : 1.0 / 6.0; }
};

template <>
struct Lat<9> {
  static constexpr double e2 = 1.0 / 3.0;
  static constexpr bool has_y = false;
  static constexpr int diag0 = 5;
  __host__ __device__ static constexpr int cls(int i) { return i == 0 ? 0 : (i <= 4 ? 1 : 2); }
  // paper's e_0..e_4 as D2Q5, then (1,1), (-1,1), (-1,-1), (1,-1); second component in ez()
  __host__ __device__ static constexpr int ex(int i) {
    switch (i) {
      case 1: case 5: case 8: return 1;
      case 3: case 6: case 7: return -1;
      default: return 0;
    }
  }
  __host__ __device__ static constexpr int ey(int) { return 0; }
  __host__ __device__ static constexpr int ez(int i) {
    switch (i) {
      case 2: case 5: case 6: return 1;
      case 4: case 7: case 8: return -1;
      default: return 0;
    }
  }
  __host__ __device__ static constexpr int opp(int i) {
    switch (i) {
      case 1: return 3; case 2: return 4; case 3: return 1; case 4: return 2;
      case 5: return 7; case 6: return 8; case 7: return 5; case 8: return 6;
      default: return 0;
    }
  }
  __host__ __device__ static constexpr double w(int i) {
    return i == 0 ? 4.0 / 9.0 : (i <= 4 ? 1.0 / 9.0 : 1.0 / 36.0);
  }
  __host__ __device__ static constexpr double B(int i) {
    return i == 0 ? -5.0 / 9.0 : (i <= 4 ? 1.0 / 9.0 : 1.0 / 36.0);
  }
};
// A_i = 1 for the rest population and 0 otherwise on all five lattices.

// Populations with e_y != 0 cross block rows during the moment gather and go
// through shared memory; yslot(i) numbers them 0..NY-1 (-1 for e_y = 0).
template <int Q>
struct YSlots {
  __host__ __device__ static constexpr int count() {
    int c = 0;
    for (int i = 0; i < Q; ++i) c += Lat<Q>::ey(i) != 0;
    return c;
  }
  __host__ __device__ static constexpr int slot(int i) {
    if (Lat<Q>::ey(i) == 0) return -1;
    int c = 0;
    for (int j = 0; j < i; ++j) c += Lat<Q>::ey(j) != 0;
    return c;
  }
};
template <int Q>
struct NYOf {
  static constexpr int value = YSlots<Q>::count();
};
template <>
struct NYOf<0> {
  static constexpr int value = 0;
};

// ---------------------------------------------------------------- storage codec
// FP64/FP32: stored as is.  FP16/BF16: stored = (f - shift) * scale, decoded to
// FP32; `shift` removes the bulk value so the stored number is the small part.
template <typename S>
struct Codec;
// raw(s) / pack(v): the stored number itself as T and back (round to nearest), for
// arithmetic done directly in the scaled units (f - shift) * scale.
// dec64 / enc64: the same codec evaluated in FP64 for state import and export: with a
// power-of-two scale, s / scale + shift is exact in FP64, so export then import returns
// every stored number unchanged.
template <>
struct Codec<double> {
  using T = double;
  static constexpr bool shifted = false;
  __device__ static __forceinline__ T dec(double s, T, T) { return s; }
  __device__ static __forceinline__ double enc(T v, T, T) { return v; }
  __device__ static __forceinline__ T raw(double s) { return s; }
  __device__ static __forceinline__ double pack(T v) { return v; }
  __device__ static __forceinline__ double dec64(double s, double, double) { return s; }
  __device__ static __forceinline__ double enc64(double v, double, double) { return v; }
};
template <>
struct Codec<float> {
  using T = float;
  static constexpr bool shifted = false;
  __device__ static __forceinline__ T dec(float s, T, T) { return s; }
  __device__ static __forceinline__ float enc(T v, T, T) { return v; }
  __device__ static __forceinline__ T raw(float s) { return s; }
  __device__ static __forceinline__ float pack(T v) { return v; }
  __device__ static __forceinline__ double dec64(float s, double, double) { return (double)s; }
  __device__ static __forceinline__ float enc64(double v, double, double) { return (float)v; }
};
template <>
struct Codec<__half> {
  using T = float;
  static constexpr bool shifted = true;
  __device__ static __forceinline__ T dec(__half s, T shift, T inv_scale) {
    return fmaf(__half2float(s), inv_scale, shift);
  }
  __device__ static __forceinline__ __half enc(T v, T shift, T scale) { return __float2half_rn((v - shift) * scale); }
  __device__ static __forceinline__ T raw(__half s) { return __half2float(s); }
  __device__ static __forceinline__ __half pack(T v) { return __float2half_rn(v); }
  __device__ static __forceinline__ double dec64(__half s, double shift, double inv_scale) {
    return (double)__half2float(s) * inv_scale + shift;
  }
  __device__ static __forceinline__ __half enc64(double v, double shift, double scale) {
    return __double2half((v - shift) * scale);
  }
};
template <>
struct Codec<__nv_bfloat16> {
  using T = float;
  static constexpr bool shifted = true;
  __device__ static __forceinline__ T dec(__nv_bfloat16 s, T shift, T inv_scale) {
    return fmaf(__bfloat162float(s), inv_scale, shift);
  }
  __device__ static __forceinline__ __nv_bfloat16 enc(T v, T shift, T scale) {
    return __float2bfloat16_rn((v - shift) * scale);
  }
  __device__ static __forceinline__ T raw(__nv_bfloat16 s) { return __bfloat162float(s); }
  __device__ static __forceinline__ __nv_bfloat16 pack(T v) { return __float2bfloat16_rn(v); }
  __device__ static __forceinline__ double dec64(__nv_bfloat16 s, double shift, double inv_scale) {
    return (double)__bfloat162float(s) * inv_scale + shift;
  }
  __device__ static __forceinline__ __nv_bfloat16 enc64(double v, double shift, double scale) {
    return __double2bfloat16((v - shift) * scale);
  }
};

// ---------------------------------------------------------------- descriptors
// The constants of a simulation in the compute type T, so that no thread converts them.
template <typename T>
struct Consts {
  T inv2dx;       // 1 / (2 dx)
  T inv2dx2;      // its square
  T c_eta;        // e^-2 (W0^2/tau0) dt/dx^2: eta_phi = c_eta a_s^2 + 1/2 (Eq. LBE_RelaxationTime)
  T inv_eta1;     // 1/eta_phi at a_s = 1
  T c_N;          // e^-2 (dt/dx) W0^2/tau0: the N term of g^(0) (Eq. Feq_Phase)
  T dt_tau0;      // dt / tau0
  T lamM, lam;    // lambda Mc_inf, lambda (Eq. LBE_SourceTerm)
  T a0, a4, a6;   // a_s = a0 + a4 sum n^4 + a6 nx^2 ny^2 nz^2 (Eq. Anisotropic-Function_As, As_K41-K61)
  T aniso, eps1, eps2;  // 0: Eq. Anisotropic-Function_As, 1: Eq. As_K41-K61, and its parameters
  T grad2_min;
  T k;
  T inv_etaU;     // 1 / eta_U (Eq. RelaxationTime_Concentration)
  T c_J;          // e^-2 dt/dx of the U lattice (Eq. Feq_Transport)
  T D_dx2;        // D / dx^2
  T D;
  T at_amp;       // W0 / (2 sqrt2), Eq. (AntiTrapping_Current)
  T dt, inv_dt;
  T inv_etaT;     // 1 / eta_theta (Eq. ThermalDiffusivity)
  T theta0;
  T shift_h, shift_f;       // FP16/BF16 codec: h shifted by w_i U0; f initially by w_i theta0
  T scale[3], inv_scale[3]; // FP16/BF16 codec scales of g, h, f (powers of two)
};

// Per-simulation constants and buffers, resident in device memory.
struct SimDev {
  int nx, ny, nz, q_theta;
  int antitrapping;
  long long nsite;
  void* pop[2][3];  // [buffer][g, h, f] in the storage type, [Q][z][y][x]
  void* phi[3];     // phi levels (compute type); level s%3 is phi^n at step s
  void* U[2];       // U^n at buffer s%2
  void* th[3];      // theta levels (unused when q_theta == 0); level s%3 is theta^n at step s
  Consts<double> c64;
  Consts<float> c32;
};
template <typename T>
__device__ __forceinline__ const Consts<T>& consts_of(const SimDev& sd) {
  if constexpr (sizeof(T) == 8) return sd.c64;
  else return sd.c32;
}

}  // namespace lbpf
