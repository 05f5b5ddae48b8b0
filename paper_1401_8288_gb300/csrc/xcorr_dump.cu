// xcorr_dump.cu -- the cross-dump accumulation: the GPU integrates K samples
// per dump and further integration happens downstream (Sec. 2.4, Sec. 4: 1024
// spectra on the GPU, then 119 more on the CPU).  Here that downstream sum is
// kept exact on the device: each dump's int32 integration is widened and added
// into a caller-owned int64 buffer.
#include "sm103_ptx.cuh"
#include "xcorr_internal.h"

namespace xc {
namespace {

// ADD: into the caller's sums; else into a new buffer, which need not be cleared and read for it (1024
// inputs x 64 channels: 78 us of clearing and 184 of folding, now 120).
template <bool ADD>
__global__ void __launch_bounds__(256) fold_wide_i64_kernel(const int4* __restrict__ acc,
                                                            longlong2* __restrict__ out, int64_t n4) {
  // one int4 of the accumulator = two (re, im) pairs = two longlong2 of the output
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n4;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int4 a = __ldg(acc + q);
    longlong2 o0 = make_longlong2(0, 0), o1 = o0;
    if (ADD) o0 = out[2 * q], o1 = out[2 * q + 1];
    o0.x += a.x;
    o0.y += a.y;
    o1.x += a.z;
    o1.y += a.w;
    out[2 * q] = o0;
    out[2 * q + 1] = o1;
  }
}

template <bool ADD>
__global__ void fold_wide_i64_tail(const int2* __restrict__ acc, longlong2* __restrict__ out, int64_t first,
                                   int64_t n) {
  const int64_t q = first + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (q < n) {
    longlong2 o = make_longlong2(0, 0);
    if (ADD) o = out[q];
    o.x += acc[q].x;
    o.y += acc[q].y;
    out[q] = o;
  }
}

// Float visibilities: widen each dump into a double running sum, the FP64
// cross-dump accumulation for integrations longer than one FP32 dump.
template <bool ADD>
__global__ void __launch_bounds__(256) fold_wide_f64_kernel(const float2* __restrict__ acc,
                                                            double2* __restrict__ out, int64_t n) {
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    const float2 a = __ldg(acc + q);
    double2 o = make_double2(0.0, 0.0);
    if (ADD) o = out[q];
    o.x += a.x;
    o.y += a.y;
    out[q] = o;
  }
}

// A memset of its own, for the time-split launches of the fused kernel, which add into a cleared output:
// behind a memset node the next kernel's launch and set-up wait for its end.  Replayed from a graph, 64
// inputs x 64 channels x 1024 samples 11.1 -> 10.5 us, 10 x 300 x 2000 14.6 -> 13.0.  (The CUDA-core
// kernel's many CTAs only crowd the SMs while they wait: 16 int8 inputs x 16 x 512 11.9 us behind a
// memset, 13.3 behind this.)
__global__ void __launch_bounds__(256) clear_kernel(uint2* __restrict__ out, int64_t pairs) {
  pdl_release();
  pdl_wait();
  const int64_t step = (int64_t)gridDim.x * 256 * 2;
  for (int64_t q = (blockIdx.x * (int64_t)256 + threadIdx.x) * 2; q < pairs; q += step) {
    if (q + 1 < pairs && (reinterpret_cast<uintptr_t>(out) & 8) == 0) {
      *reinterpret_cast<uint4*>(out + q) = make_uint4(0, 0, 0, 0);
    } else {
      out[q] = make_uint2(0, 0);
      if (q + 1 < pairs) out[q + 1] = make_uint2(0, 0);
    }
  }
}

}  // namespace

cudaError_t launch_clear(void* out, int64_t pairs, cudaStream_t stream) {
  // (the adding launch behind it takes any output of aligned integers)
  if (reinterpret_cast<uintptr_t>(out) % sizeof(uint2)) return cudaMemsetAsync(out, 0, pairs * sizeof(uint2), stream);
  int64_t blocks = (pairs + 511) / 512;
  if (blocks > 4096) blocks = 4096;
  return launch_dependent(clear_kernel, static_cast<unsigned>(blocks), 256, 0, stream, static_cast<uint2*>(out), pairs);
}

cudaError_t launch_fold_wide_f64(const float2* acc, double* out, int64_t n_pairs_total, bool add, cudaStream_t stream) {
  int64_t blocks = (n_pairs_total + 255) / 256;
  if (blocks > 65535) blocks = 65535;
  if (blocks < 1) blocks = 1;
  (add ? fold_wide_f64_kernel<true> : fold_wide_f64_kernel<false>)<<<(unsigned)blocks, 256, 0, stream>>>(
      acc, reinterpret_cast<double2*>(out), n_pairs_total);
  return cudaGetLastError();
}

cudaError_t launch_fold_wide_i64(const int2* acc, int64_t* out, int64_t n_pairs_total, bool add, cudaStream_t stream) {
  const int64_t n4 = n_pairs_total / 2;
  if (n4 > 0) {
    int64_t blocks = (n4 + 255) / 256;
    if (blocks > 65535) blocks = 65535;
    (add ? fold_wide_i64_kernel<true> : fold_wide_i64_kernel<false>)<<<(unsigned)blocks, 256, 0, stream>>>(
        reinterpret_cast<const int4*>(acc), reinterpret_cast<longlong2*>(out), n4);
  }
  if (n_pairs_total % 2)
    (add ? fold_wide_i64_tail<true> : fold_wide_i64_tail<false>)<<<1, 32, 0, stream>>>(
        acc, reinterpret_cast<longlong2*>(out), 2 * n4, n_pairs_total);
  return cudaGetLastError();
}

}  // namespace xc
