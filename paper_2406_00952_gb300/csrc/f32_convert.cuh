// FP64 <-> FP32 conversions of the FP32 preconditioner passes.
#pragma once
#include <cuda_runtime.h>

namespace pcb {

// FP64 <-> FP32 conversions with integer operations.  The conversion instructions run on the FP64
// pipe, which is narrow on this GPU and became the bottleneck of the passes that read or write
// the FP64 vectors.  IEEE-754 binary64 -> binary32, round to nearest even: for results in the
// normal FP32 range the rounded value is the top 31 bits of (exponent - 896, mantissa >> 29)
// plus one when the dropped 29 bits exceed half, or equal half and the kept value is odd (a
// carry into the exponent gives the right next binade, or infinity).  Zeros keep their sign;
// the rare remaining cases (FP32 subnormals, overflow, infinities, NaN) use the instruction.
__device__ __forceinline__ float d2f(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned ah = hi & 0x7fffffffu, e = ah >> 20;
  if (e - 897u <= 253u) {
    const unsigned m = (ah << 3) | (lo >> 29);
    const unsigned rem = lo & 0x1fffffffu;
    const unsigned rnd = (unsigned)(rem > 0x10000000u) | ((unsigned)(rem == 0x10000000u) & m & 1u);
    return __uint_as_float(((m - (896u << 23)) + rnd) | (hi & 0x80000000u));
  }
  if ((ah | lo) == 0u) return __uint_as_float(hi & 0x80000000u);
  return __double2float_rn(x);
}
// binary32 -> binary64 (exact): exponent rebiased by 896, mantissa moved up by 29 bits
__device__ __forceinline__ double f2d(float f) {
  const unsigned b = __float_as_uint(f), e = (b >> 23) & 0xffu;
  if (e - 1u < 254u) {
    const unsigned hi = (b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20));
    return __hiloint2double((int)hi, (int)(b << 29));
  }
  if ((b & 0x7fffffffu) == 0u) return __hiloint2double((int)(b & 0x80000000u), 0);
  return (double)f;
}
__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(double v) { return d2f(v); }
// Branch-free forms for values held in registers: a branch per value would order the loads that feed
// it one after another.  `rare` collects the inputs the integer route does not cover (see above); the
// caller converts its values again with the instruction when any reports one.
__device__ __forceinline__ float d2f_plain(double x, unsigned& rare) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned ah = hi & 0x7fffffffu;
  const unsigned m = __funnelshift_l(lo, hi, 3) - (896u << 23);
  const unsigned rnd = ((lo & 0x1fffffffu) + 0x0fffffffu + ((lo >> 29) & 1u)) >> 29;
  const bool normal = ah - (897u << 20) < (254u << 20);
  rare |= normal ? 0u : (ah | lo);
  return __uint_as_float(((normal ? m + rnd : 0u) & 0x7fffffffu) | (hi & 0x80000000u));
}
__device__ __forceinline__ double f2d_plain(float f, unsigned& rare) {
  const unsigned b = __float_as_uint(f), a = b & 0x7fffffffu;
  const bool normal = a - 0x00800000u < 0x7f000000u;
  rare |= normal ? 0u : a;                             // subnormal, infinite, NaN
  return __hiloint2double((int)((normal ? (a >> 3) + (896u << 20) : 0u) | (b & 0x80000000u)), (int)(b << 29));
}
// The gather of pass 1 converts every kF2FEvery-th register of a line with the conversion
// instruction and the rest with integer operations: both round to nearest even, and the mix
// shares the work between the FP64 pipe and the integer pipe.
constexpr int kF2FEvery = 2;
__device__ __forceinline__ float to_f32_at(float v, int) { return v; }
__device__ __forceinline__ float to_f32_at(double v, int q) {
  return (kF2FEvery > 0 && q % kF2FEvery == kF2FEvery - 1) ? __double2float_rn(v) : d2f(v);
}
template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ double from_f32<double>(float v) { return f2d(v); }
// pass 5's FP64 results: every kF2DEvery-th register through the conversion instruction
constexpr int kF2DEvery = 2;
template <typename T> __device__ __forceinline__ T from_f32_at(float v, int j) {
  if constexpr (sizeof(T) == 8) {
    if (kF2DEvery > 0 && j % kF2DEvery == kF2DEvery - 1) return (double)v;
  }
  return from_f32<T>(v);
}

}  // namespace pcb
