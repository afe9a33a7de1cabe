#pragma once
// Conversions between FP32, FP64 and pairs of FP32 values on the integer units.
//
// The conversion instructions that touch a double issue at the rate of the FP64 pipe (two lanes a clock
// on an SM, 1/64 of the FP32 rate), so a pass that does nothing but convert is bound by them and not by
// memory: splitting 17.3 million complex values takes 104 million FP64-pipe operations, 0.26 ms, against
// 0.08 ms for the 550 MB it moves. Both formats differ only in the width of the exponent and the
// mantissa, so in the normal range a few integer operations do it: widening shifts the 31 magnitude bits
// by 3 and adds the difference of the exponent biases (1023 - 127 = 896), narrowing does the reverse and
// rounds the 29 bits shifted out to nearest even. Zeros keep their sign; subnormals, infinities, NaNs
// and magnitudes outside the normal FP32 range go to the conversion instruction, so every result has the
// bits of the plain cast.
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define WDF_CB __host__ __device__ __forceinline__
#else
#define WDF_CB inline
#endif

namespace wdf {

WDF_CB uint32_t cb_bits(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  uint32_t u;
  std::memcpy(&u, &f, 4);
  return u;
#endif
}
WDF_CB float cb_float(uint32_t u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float f;
  std::memcpy(&f, &u, 4);
  return f;
#endif
}
WDF_CB void cb_split(double d, uint32_t &hi, uint32_t &lo) {
#ifdef __CUDA_ARCH__
  hi = (uint32_t)__double2hiint(d);
  lo = (uint32_t)__double2loint(d);
#else
  uint64_t u;
  std::memcpy(&u, &d, 8);
  hi = (uint32_t)(u >> 32);
  lo = (uint32_t)u;
#endif
}
WDF_CB double cb_double(uint32_t hi, uint32_t lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double((int)hi, (int)lo);
#else
  const uint64_t u = ((uint64_t)hi << 32) | lo;
  double d;
  std::memcpy(&d, &u, 8);
  return d;
#endif
}

// (double)f
WDF_CB double widen(float f) {
  const uint32_t u = cb_bits(f), m = u & 0x7fffffffu;
  if (m - 0x00800000u < 0x7f000000u) return cb_double((u & 0x80000000u) | ((m >> 3) + 0x38000000u), u << 29);
  if (m == 0) return cb_double(u, 0u);
  return (double)f;
}

// (float)d, rounded to nearest even
WDF_CB float narrow(double d) {
  uint32_t hi, lo;
  cb_split(d, hi, lo);
  const uint32_t m = hi & 0x7fffffffu, s = hi & 0x80000000u;
  if (m - 0x38100000u < 0x0fe00000u) {
    const uint32_t r = ((m - 0x38000000u) << 3) | (lo >> 29), rest = lo << 3;
    return cb_float(s | (r + (rest + (r & 1u) > 0x80000000u ? 1u : 0u)));
  }
  if ((m | lo) == 0) return cb_float(s);
  return (float)d;
}

}  // namespace wdf
