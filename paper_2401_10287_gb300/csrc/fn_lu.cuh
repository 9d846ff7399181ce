// Register-resident LU of one small orbital matrix per thread.
#pragma once
#include <stdint.h>

#include "fn_device.cuh"

namespace fn {

// Widening of a stored orbital entry to the determinant type.  FP32 -> FP64 goes through
// integer bit operations (sign, exponent re-biased by 1023 - 127, mantissa shifted into the
// top of the 52-bit field): exact for every normal FP32 value, FP32 subnormals become signed
// zero, infinities and NaNs keep their class.  It keeps the conversions off the FP64 pipe,
// which sets the pace of this stage.
template <typename Det, typename PhiT> __device__ __forceinline__ Det widen(PhiT v) { return (Det)v; }
template <> __device__ __forceinline__ double widen<double, float>(float f) {
  const uint32_t u = __float_as_uint(f);
  const uint32_t ex = (u >> 23) & 0xFFu, sign = u & 0x80000000u, man = u & 0x7FFFFFu;
  const uint32_t ex64 = ex == 0 ? 0u : (ex == 0xFFu ? 0x7FFu : ex + 896u);
  const uint32_t hi = sign | (ex64 << 20) | (ex == 0 ? 0u : (man >> 3));
  const uint32_t lo = ex == 0 ? 0u : (man << 29);
  return __hiloint2double((int)hi, (int)lo);
}

// The same with FP32 subnormals kept: they are scaled into the normal range (exactly) first.
template <typename Det, typename PhiT> __device__ __forceinline__ Det widen_all(PhiT v) { return (Det)v; }
template <> __device__ __forceinline__ double widen_all<double, float>(float f) {
  const bool sub = (__float_as_uint(f) & 0x7F800000u) == 0u;
  const uint32_t u = __float_as_uint(sub ? f * 0x1p64f : f);
  const uint32_t ex = (u >> 23) & 0xFFu, sign = u & 0x80000000u, man = u & 0x7FFFFFu;
  const uint32_t ex64 = ex == 0 ? 0u : (ex == 0xFFu ? 0x7FFu : ex + (sub ? 832u : 896u));
  return __hiloint2double((int)(sign | (ex64 << 20) | (man >> 3)), (int)(man << 29));
}

// Pivot search key: |v| as an unsigned integer (the bit patterns of non-negative IEEE
// numbers order like their values), so the comparisons leave the FP64 pipe alone.
__device__ __forceinline__ unsigned long long abs_key(double v) {
  return (unsigned long long)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
}
__device__ __forceinline__ unsigned int abs_key(float v) { return __float_as_uint(v) & 0x7FFFFFFFu; }

// Register-resident LU of one n x n block (n <= 8 known at compile time): one elimination
// step per template instance, so every matrix index is a compile-time constant and the block
// stays in registers; partial pivoting by predicated row swaps; log|det| and sign by
// mantissa/exponent tracking.
template <int NN, int C, typename Det>
struct LuStep {
  static __device__ __forceinline__ void run(Det (&a)[NN][NN], Det& sgn, Det& mant, int& expo, bool& singular) {
    auto best = abs_key(a[C][C]);
    int piv = C;
#pragma unroll
    for (int r = C + 1; r < NN; ++r) {
      const auto v = abs_key(a[r][C]);
      if (v > best) { best = v; piv = r; }
    }
    if (best == 0) singular = true;
#pragma unroll
    for (int r = C + 1; r < NN; ++r) {
      const bool sw = r == piv;
#pragma unroll
      for (int j = 0; j < NN; ++j) {
        const Det t = a[C][j];
        a[C][j] = sw ? a[r][j] : t;
        a[r][j] = sw ? t : a[r][j];
      }
    }
    if (piv != C) sgn = -sgn;
    const Det p = a[C][C];
    const Det rp = (Det)1 / p;
    int e;
    mant *= frexp(p, &e);
    expo += e;
    int e2;
    mant = frexp(mant, &e2);
    expo += e2;
#pragma unroll
    for (int r = C + 1; r < NN; ++r) {
      const Det f = a[r][C] * rp;
#pragma unroll
      for (int j = C + 1; j < NN; ++j) a[r][j] -= f * a[C][j];
    }
    LuStep<NN, C + 1, Det>::run(a, sgn, mant, expo, singular);
  }
};
template <int NN, typename Det>
struct LuStep<NN, NN, Det> {
  static __device__ __forceinline__ void run(Det (&)[NN][NN], Det&, Det&, int&, bool&) {}
};

template <int NN, typename Det, typename PhiT>
__device__ __forceinline__ void lu_regs(const PhiT* __restrict__ Ag, Det* mant_out, int* expo_out) {
  Det a[NN][NN];
#pragma unroll
  for (int i = 0; i < NN; ++i)
#pragma unroll
    for (int j = 0; j < NN; ++j) a[i][j] = widen<Det, PhiT>(Ag[i * NN + j]);
  Det sgn = 1, mant = 1;
  int expo = 0;
  bool singular = false;
  LuStep<NN, 0, Det>::run(a, sgn, mant, expo, singular);
  *mant_out = singular ? (Det)0 : sgn * mant;
  *expo_out = singular ? 0 : expo;
}

// det A = mant 2^expo with |mant| in [1/2, 1) (mant = 0 for a singular block)
template <typename Det, typename PhiT>
__device__ __forceinline__ void lu_regs_any(const PhiT* Ag, int n, Det* mant, int* expo) {
  switch (n) {
    case 1: lu_regs<1, Det, PhiT>(Ag, mant, expo); break;
    case 2: lu_regs<2, Det, PhiT>(Ag, mant, expo); break;
    case 3: lu_regs<3, Det, PhiT>(Ag, mant, expo); break;
    case 4: lu_regs<4, Det, PhiT>(Ag, mant, expo); break;
    case 5: lu_regs<5, Det, PhiT>(Ag, mant, expo); break;
    case 6: lu_regs<6, Det, PhiT>(Ag, mant, expo); break;
    case 7: lu_regs<7, Det, PhiT>(Ag, mant, expo); break;
    default: lu_regs<8, Det, PhiT>(Ag, mant, expo); break;
  }
}

}  // namespace fn
