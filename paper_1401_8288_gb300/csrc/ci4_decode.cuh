// ci4_decode.cuh -- 4+4-bit complex samples to E4M3 codes, four at a time.
//
// A CI4 byte holds a 4-bit two's-complement real part in its high nibble and
// the imaginary part in its low nibble (the library's reading of the paper's
// four bits for each of the real and imaginary parts, Sec. 2.3).  Every value in [-8, 7] is an
// exact E4M3 number, so these codes feed kind::f8f6f4 MMAs with the true
// integers.  The lookups are byte permutes over two 8-entry tables.
#pragma once
#include <cstdint>

namespace xc {

// E4M3 codes of 0..7 and of -8..-1, four per word, lowest byte first.
constexpr uint32_t kE4m3Pos0 = 0x44403800u;  // 0, 1, 2, 3
constexpr uint32_t kE4m3Pos1 = 0x4E4C4A48u;  // 4, 5, 6, 7
constexpr uint32_t kE4m3Neg0 = 0xCACCCED0u;  // -8, -7, -6, -5
constexpr uint32_t kE4m3Neg1 = 0xB8C0C4C8u;  // -4, -3, -2, -1

// The permute itself: unlike __byte_perm it keeps selector bit 3, which spreads the chosen byte's
// sign bit over the result byte.
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
  return r;
}

// Four CI4 samples (one per byte) -> four E4M3 real parts and four imaginary parts.
// A permute's selector nibbles pick bytes by their low three bits, so the samples' own nibbles
// (their top bits cleared) select from both tables, low half-word and high half-word in turn; the
// four results hold im and re interleaved.  A sign-replicating permute (selector bit 3) spreads
// each sample's sign bit over its byte to choose between the tables.
__device__ __forceinline__ void ci4_to_e4m3(uint32_t v, uint32_t& re, uint32_t& im) {
  const uint32_t lo = v & 0x77777777u, hi = lo >> 16;
  const uint32_t p0 = prmt(kE4m3Pos0, kE4m3Pos1, lo), p1 = prmt(kE4m3Pos0, kE4m3Pos1, hi);
  const uint32_t n0 = prmt(kE4m3Neg0, kE4m3Neg1, lo), n1 = prmt(kE4m3Neg0, kE4m3Neg1, hi);
  const uint32_t re_neg = prmt(v, 0u, 0xBA98), im_neg = prmt(v << 4, 0u, 0xBA98);
  re = (prmt(n0, n1, 0x7531) & re_neg) | (prmt(p0, p1, 0x7531) & ~re_neg);
  im = (prmt(n0, n1, 0x6420) & im_neg) | (prmt(p0, p1, 0x6420) & ~im_neg);
}

}  // namespace xc
