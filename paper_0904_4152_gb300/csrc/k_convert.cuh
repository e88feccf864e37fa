// FP32 <-> FP64 conversions that leave the FP64 pipe to the arithmetic.
#pragma once

namespace hn {
namespace {

// FP32 to FP64 and back (to nearest, ties to even) by the IEEE 754 bit layout, the operands of the conversion
// instruction in the ranges that need more than a shift: that instruction takes a slot of the FP64 pipe, which bounds
// the kernels that use this, as an FMA does; these few integer operations take a third of it of another pipe.  The steps of
// CG at L = 11: x, r 73 -> 62 us, (r, c) 43 -> 34, p 29 -> 22; the update at L = 10 12.4 -> 10.5 us.
__device__ __forceinline__ double to_f64(float f) {
  const unsigned u = __float_as_uint(f), a = u & 0x7fffffffu;
  if (a - 0x00800000u < 0x7f000000u)              // normal: the exponent's bias from 127 to 1023
    return __hiloint2double((int)((u & 0x80000000u) | ((a >> 3) + (896u << 20))), (int)(u << 29));
  return a == 0u ? __hiloint2double((int)u, 0) : double(f);
}
__device__ __forceinline__ double to_f64(double f) { return f; }
template <class V> __device__ __forceinline__ V from_f64(double d);
template <> __device__ __forceinline__ double from_f64<double>(double d) { return d; }
template <> __device__ __forceinline__ float from_f64<float>(double d) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d), a = hi & 0x7fffffffu;
  if (a - (897u << 20) < (253u << 20)) {          // a normal float, also after rounding up
    const unsigned m = ((a - (896u << 20)) << 3) | (lo >> 29), rest = lo << 3;
    const unsigned up = rest > 0x80000000u || (rest == 0x80000000u && (m & 1u));
    return __uint_as_float((hi & 0x80000000u) | (m + up));
  }
  return (a | lo) == 0u ? __uint_as_float(hi) : float(d);
}

}  // namespace
}  // namespace hn
