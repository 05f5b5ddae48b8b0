// unpack_device.cuh -- the unpack step of Sec. 2.4 as device functions: 16
// bytes of samples to operand numbers, and the float windows' digits.  Used by
// the stand-alone unpack kernels (xcorr_unpack.cu) and by the unpack warps of
// the CTA-pair kernel (xcorr_tc_pair.cu).
#pragma once
#include <cuda_bf16.h>

#include <cstdint>

#include "ci4_decode.cuh"
#include "xcorr_internal.h"

namespace xc {

// Sixteen CI4 samples -> sixteen E4M3 real codes and sixteen imaginary codes.
__device__ __forceinline__ void decode_ci4(const uint4& v, uint4& re, uint4& im) {
  ci4_to_e4m3(v.x, re.x, im.x);
  ci4_to_e4m3(v.y, re.y, im.y);
  ci4_to_e4m3(v.z, re.z, im.z);
  ci4_to_e4m3(v.w, re.w, im.w);
}

// Float input, per (channel, window, input): find the window's
// largest magnitude max < 2^(E+1), quantise each component to the integer
// M = rint(x 2^(22-E)) (|M| < 2^23, error <= 2^-23 max), and write the
// balanced base-256 digits of M = d0 2^16 + d1 2^8 + d2 (|d_p| <= 128, exact
// BF16 values) to planes re_p = p and im_p = 3 + p.  E goes to exps.
//
// Edges.  The maximum is taken over the components' bit patterns with the
// sign cleared: for non-negative floats they order as the values do, and the
// patterns of infinities and NaNs lie above every finite one, so one integer
// maximum also finds a non-finite sample.  Such a window gets E =
// kExpNonFinite and zero digits; the X kernel's drain turns every block that
// involves it into NaN.  A window whose maximum is subnormal gets that
// maximum's own exponent (down to -149), so its samples keep 23-bit integers
// like any other window's and no finite input is flushed.  2^(22-E) spans
// 2^-105 .. 2^171, past the float range, so it is applied as two exact
// power-of-two factors.
__device__ __forceinline__ uint32_t abs_bits(float x) { return __float_as_uint(x) & 0x7FFFFFFFu; }

__device__ __forceinline__ int window_exponent(uint32_t max_bits) {
  if (max_bits >= 0x7F800000u) return kExpNonFinite;
  if (max_bits >= 0x00800000u) return static_cast<int>(max_bits >> 23) - 127;  // normal
  if (max_bits == 0u) return kExpMin;
  return (31 - __clz(static_cast<int>(max_bits))) - 149;  // subnormal m 2^-149: floor(log2 m) - 149
}

// The two factors of 2^(22 - e), each in [2^-53, 2^86]; zero for a non-finite window.
__device__ __forceinline__ void window_scale(int e, float& s1, float& s2) {
  if (e == kExpNonFinite) {
    s1 = s2 = 0.f;
    return;
  }
  const int n = 22 - e, a = n >> 1;
  s1 = pow2i(a);
  s2 = pow2i(n - a);
}

// The digits of one component of two inputs, as BF16 pairs: with M + 0x808080 the bytes are d2 + 128
// and d1 + 128 and the upper half-word d0 + 128 (at most 256), each an exact float when put into the
// low mantissa bits of 2^23, and 2^23 + 128 subtracted; the upper half of that float is its BF16
// value.  (The conversion instructions, three of each kind a component, run at an eighth of the ALU's rate.)
__device__ __forceinline__ void digit_pairs(float x0, float s0a, float s0b, float x1, float s1a, float s1b,
                                            uint32_t (&d)[3]) {
  const uint32_t m0 = static_cast<uint32_t>(__float2int_rn((x0 * s0a) * s0b)) + 0x808080u;
  const uint32_t m1 = static_cast<uint32_t>(__float2int_rn((x1 * s1a) * s1b)) + 0x808080u;
  constexpr uint32_t kSel[3] = {0x7432, 0x7441, 0x7440};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float a = __uint_as_float(__byte_perm(m0, 0x4B000000u, kSel[k])) - 8388736.0f;
    const float b = __uint_as_float(__byte_perm(m1, 0x4B000000u, kSel[k])) - 8388736.0f;
    d[k] = __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
  }
}

}  // namespace xc
