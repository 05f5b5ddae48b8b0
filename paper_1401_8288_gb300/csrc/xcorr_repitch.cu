// xcorr_repitch.cu -- input whose rows do not sit on the 16-byte boundaries the tiled copies of the
// on-chip decoding kernels need (4-bit: inputs not a multiple of 16; int8: not of 8; or a base
// address off 16 bytes) is copied, still packed, to rows that do, and correlated from there.
// Unpacking it to planes instead writes and reads two to four times the bytes and left the X-stage
// to the slower kernels that read planes (4-bit, 338 inputs x 97 channels x 1500 samples: 120 us from
// a ring of planes, 70 so; 122 x 300 x 2048 from planes in memory: 330, now 60; int8, 122 x 300 x 4096:
// 716, now 290; 510 x 300 x 2048: 820, now 725).
//
// Bound by memory: each byte is read once and written once.
#include "sm103_ptx.cuh"
#include "xcorr_internal.h"

namespace xc {
namespace {

constexpr int kUnits = 4;  // 16-byte pieces a thread has in flight

struct RepitchParams {
  const uint8_t* in;       // first byte of the first row's first channel
  const uint8_t* end;      // one past the caller's last byte
  uint4* out;
  int64_t time_bytes;      // bytes from one sample to the next
  uint32_t units;          // 16-byte pieces written for one sample: n_chan * per_row
  uint32_t per_row, row_bytes;
  int n_time;
};

// One thread per piece of 16 bytes: the two aligned words that hold its source bytes, shifted
// together.  (A row's last piece reads on into the next row: those inputs are never used.)  Only
// words that hold bytes of the input are read.
__global__ void __launch_bounds__(256) repitch_kernel(const RepitchParams p) {
  pdl_wait();
  const uint32_t u = blockIdx.x * 256 + threadIdx.x;
  if (u >= p.units) return;
  const uint32_t row = u / p.per_row, piece = u - row * p.per_row;
  const uint8_t* s = p.in + (int64_t)row * p.row_bytes + 16 * piece;
  uint4* d = p.out + u;
  for (int t0 = blockIdx.y * kUnits; t0 < p.n_time; t0 += gridDim.y * kUnits) {
    uint4 lo[kUnits], hi[kUnits];
    uint32_t sh[kUnits];
#pragma unroll
    for (int k = 0; k < kUnits; ++k) {
      lo[k] = hi[k] = make_uint4(0, 0, 0, 0);
      const uintptr_t a = reinterpret_cast<uintptr_t>(s + (int64_t)(t0 + k) * p.time_bytes);
      sh[k] = static_cast<uint32_t>(a & 15);
      const uint4* w = reinterpret_cast<const uint4*>(a - sh[k]);
      if (t0 + k < p.n_time) {
        lo[k] = __ldg(w);
        if (sh[k] && reinterpret_cast<const uint8_t*>(w + 1) < p.end) hi[k] = __ldg(w + 1);
      }
    }
#pragma unroll
    for (int k = 0; k < kUnits; ++k) {
      uint32_t v[7] = {lo[k].x, lo[k].y, lo[k].z, lo[k].w, hi[k].x, hi[k].y, hi[k].z};
      uint32_t last = hi[k].w;
      if (sh[k] & 8) {
#pragma unroll
        for (int q = 0; q < 5; ++q) v[q] = v[q + 2];
        v[5] = last;
      }
      if (sh[k] & 4) {
        last = v[5];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = v[q + 1];
        v[4] = last;
      }
      const uint32_t bits = 8 * (sh[k] & 3);
      if (t0 + k < p.n_time)
        d[(int64_t)(t0 + k) * p.units] =
            make_uint4(__funnelshift_r(v[0], v[1], bits), __funnelshift_r(v[1], v[2], bits),
                       __funnelshift_r(v[2], v[3], bits), __funnelshift_r(v[3], v[4], bits));
    }
  }
}

}  // namespace

cudaError_t launch_repitch(const void* in, const void* end, void* out, int row_bytes, int row_chans, int n_chan,
                           int n_time, int num_sms, cudaStream_t stream) {
  RepitchParams p{};
  p.in = static_cast<const uint8_t*>(in);
  p.end = static_cast<const uint8_t*>(end);
  p.out = static_cast<uint4*>(out);
  p.time_bytes = (int64_t)row_bytes * row_chans;
  p.per_row = static_cast<uint32_t>((row_bytes + 15) / 16);
  p.row_bytes = static_cast<uint32_t>(row_bytes);
  const int64_t units = (int64_t)p.per_row * n_chan;
  if (units > 0x7FFFFFFF - 256) return cudaErrorInvalidValue;
  p.units = static_cast<uint32_t>(units);
  p.n_time = n_time;
  const unsigned bx = static_cast<unsigned>((units + 255) / 256);
  // about four waves of eight CTAs an SM, each thread at least one turn of kUnits samples
  unsigned by = static_cast<unsigned>((n_time + kUnits - 1) / kUnits);
  const unsigned want = (32u * static_cast<unsigned>(num_sms) + bx - 1) / bx;
  if (by > want) by = want;
  return launch_dependent(repitch_kernel, dim3(bx, by), 256, 0, stream, p);
}

}  // namespace xc
