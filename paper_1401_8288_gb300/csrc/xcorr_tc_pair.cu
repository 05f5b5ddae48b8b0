// xcorr_tc_pair.cu -- the X-stage in one launch on CTA pairs: samples are
// unpacked once into a ring of operand planes, mostly read from L2, and
// pairs of SMs correlate from it with cta_group::2 tcgen05 MMAs.
//
// Same operands, K axis, exact blocks and results as xcorr_unpack.cu followed
// by xcorr_tc.cu (per channel the packed lower triangle of V = sum_t x_t x_t^H;
// Sec. 1, Sec. 2.1, Eq. 1; the unpack and corner turn of Sec. 2.4): 4-bit
// samples as E4M3 planes, float as six BF16 planes of integer digits with one
// exponent per (channel, 384-sample window, input).
// For problems of two or more 128-input tiles that keep every cluster at work for
// long (planes_beat_ring in xcorr_api.cu has the rule).
//
// Why one launch.  Unpacking to planes in HBM writes 2 (4-bit) or 12 (float)
// bytes per sample that the X kernel reads back: as much time as the
// tensor work itself.  Unpacking on chip inside the tile pairs repeats the
// decode for every tile pair that needs an input.  Here four warps of every
// CTA unpack each sample once, a chunk of time ahead of the tile pairs, into a
// ring of slots (one chunk of one channel each).  The ring has 48 MB, or three
// steps of a batch where those are more (512 inputs: 120 MB), and such a ring does
// not stay in the 129 MB L2 beside the samples: a launch of 512 x 24 x 1536 reads
// 151 MB of float samples and writes 25 MB, but moves 325 MB from DRAM and 220 to it.
//
// Why pairs.  An SM's shared memory serves 128 bytes per cycle, to the TMA
// writes and the tensor core's operand reads together.  One MMA step (32 E4M3
// or 16 BF16 samples) of a 128 x 128 complex tile pair is 256 tensor cycles;
// the single-SM planes kernel writes 16 KB and reads 28 KB per step: 344
// cycles of shared memory, its measured rate.  Here each CTA loads its own row
// tile but only half of the column tile, and all MMAs are M = 256, N = 256: 12
// KB written by the TMA, 4 KB moved by the negation below, 16 KB read.
//
// The two CTAs of a cluster run the tile pairs (c, R0, S) and (c, R1, S).  The
// even CTA issues, per step,
//     [Re | X] += A_re [B_re | B_im],   [Re | X] += A_im [B_im | -B_re],
// X = -Im, with A the two row tiles (each CTA's own 128 rows) and B the column
// tile S, 64 columns from each CTA, so a CTA's accumulator holds [Re | X] of
// columns 0-63, then of columns 64-127.  -B_re is made in shared memory by two
// warps that copy the real half-tile with the sign bits flipped as soon as it
// lands (a third plane would cost half as much L2 traffic again, and four
// N = 128 MMAs with the negate bit would read 24 KB per step).
//
// A channel's tile pairs are grouped by their column tile (fused_pairing.h);
// where a column's count is odd its last tile pair is computed TRANSPOSED in
// another column's entry, and the epilogue writes V[b][a] = conj(W[a][b]),
// coalesced as it comes: a warp holds 32 consecutive a of each output row b.
//
// Order and waiting.  Entries run channel-major, one per cluster at a time, so
// all clusters walk a batch of consecutive channels together.  The unpack
// follows that order: (batch, time chunk, channel of the batch).  A chunk's
// slot is ready when its sub-tasks have added up in ready[u]; it may be
// refilled once every CTA that reads it has added to done[u].  An unpack waits
// for the reports of earlier places only, a reader reports what it has read
// before it waits for an unpack, and the launch is cooperative (every CTA is
// resident), so both waits always end, with a ring of any length (ring_order.h;
// tests/test_ring_order.py plays it); like all waits here they are bounded
// (sm103_ptx.cuh).  The last CTA to leave clears the flags.
//
// Measured (one GB300), against unpack + planes kernel: 512 inputs x 256 channels x 4096 samples, float
// 5.2-5.8 ms (7.2-7.3); 338 inputs x 97 channels x 1500, 4-bit, 129 us (252); two tiles: 256 inputs x
// 256 channels x 2048, float, 1.22 ms (1.40), 250 x 300 x 2048, 4-bit, 355 us (670).
// A step takes 272 cycles with the MMAs alone, 307-318 from a ring that nobody refills (about 40
// bytes per cycle and SM from L2, the rate every form of these loads stopped at), 450-470 beside the
// unpack, which alone would take 250-330.  With one tile half of every
// pair's rows are idle, and the planes kernel wins once there are channels for every SM (128 inputs x
// 300 channels x 4096, float: 1.11 ms against 1.29 here).  4-bit input comes here when planes are asked
// for and all of them would be too much, or under a memory limit too tight for padded rows: otherwise it stays with the fused kernel (492
// us against about 600 here at 512 inputs x 512 channels x 2048 samples: its L2 traffic is the raw
// bytes), over padded rows where its own are not aligned (70 against 119 us at 338 x 97 x 1500).  int8
// input goes to xcorr_tc_raw_pair.cu (0.87 ms against 1.00 with BF16 planes here).
//
// Warp roles (512 threads, one CTA per SM): warps 0-7 drain TMEM into running
// sums held in registers (warp w: lane quarter w % 4, columns 64 (w / 4) ..
// + 63) and write finished tiles; warp 8 is the TMA producer; warp 9 owns
// tensor memory and (in the even CTA) issues the MMAs; warps 10-11 negate;
// warps 12-15 unpack.  The odd CTA signals the even one with 16-byte bulk
// copies that complete bytes on its barriers.  Two 256-column accumulators let
// the drain of one block overlap the MMAs of the next.
#include <type_traits>

#include "pair_common.cuh"
#include "ring_order.h"
#include "unpack_device.cuh"
#include "xcorr_internal.h"

namespace xc {
namespace {

using namespace pairs;
using fused::pair_entries;

constexpr int kProducerWarp = 8;
constexpr int kMmaWarp = 9;
constexpr int kNegWarp0 = 10;
constexpr int kNegWarps = 2;
constexpr int kUnpackWarp0 = 12;
constexpr int kUnpackWarps = 4;
constexpr int kThreads = (kUnpackWarp0 + kUnpackWarps) * 32;
constexpr int kFactorBytes = kEpiWarps * kHalf * 4;  // float input: column factors of a window
constexpr int kStages = 6;         // of 28 KB: finer stages cover the copies' latency better than 3 x 56 KB
constexpr int kRowsPerTask = 32;   // an unpack sub-task (integer formats): 32 samples of one channel x
constexpr int kHalfPerTask = 4;    // 4 columns of 128 bytes of raw samples
constexpr int kFetchGroups = 3;    // groups of raw copies in flight per unpack warp
constexpr int kFetchRows = 16;     // samples per group: 4 copies of 16 bytes per lane (4 samples x 8 units a warp)
// raw samples on their way to the unpack warps: per lane and copy 16 bytes, and for the last unit of a
// sample's column (or row) the word after it (rows that are not 16-byte aligned)
constexpr int kFetchSlots = kUnpackWarps * 32 * 4 * kFetchGroups;
constexpr int kFetchBytes = kFetchSlots * 16 + kFetchSlots / 8 * 4;
constexpr int kBarrierBytes = 512;
constexpr int64_t kRingPlaces = int64_t(1) << 24;   // of a launch: 134 MB of flags, far inside an int
constexpr int kSinkSlots = kNegWarps + kEpiWarps;  // one per signalling warp of the odd CTA

// FMT: XCORR_IN_CI4 / CF32
template <int FMT>
struct Geom {
  static constexpr int E = FMT == XCORR_IN_CI4 ? 1 : 2;      // operand bytes
  static constexpr int kRows = 64 / E;                       // samples per stage
  static constexpr int kRowB = kHalf * E;                    // bytes per sample of 64 inputs
  static constexpr int kPlane = kRows * kRowB;               // one component of 64 inputs: the unit of the ring and of a stage
  static constexpr int kOffB = 4 * kPlane;                   // [A: 2 x (re | im) | B re | B im | -B re]
  static constexpr int kStageBytes = 7 * kPlane;
  static constexpr int kMmaK = 32 / E;                       // K of one MMA (samples)
  static constexpr int kSteps = kRows / kMmaK;
  static constexpr uint32_t kSignMask = E == 1 ? 0x80808080u : 0x80008000u;
  static constexpr int kDigits = FMT == XCORR_IN_CF32 ? 3 : 1;  // digit planes per component
  static constexpr int kPairsK = FMT == XCORR_IN_CF32 ? 6 : 1;  // plane pairs on the K axis
  static constexpr int kWindow = FMT == XCORR_IN_CI4 ? kTcWindowCI4 : kTcWindowBF16;
  static constexpr int kMaxChunk = FMT == XCORR_IN_CI4 ? 512 : kTcWindowBF16;
  static constexpr int kSpw = kWindow / kRows;               // stages per window
  static constexpr int kOffStaging = kStages * kStageBytes;
  static constexpr int kOffFactors = kOffStaging + kStagingBytes;
  static constexpr int kOffFetch = kOffFactors + kFactorBytes;
  static constexpr int kOffBarriers = kOffFetch + kFetchBytes;
  static constexpr int kSmem = 1024 + kOffBarriers + kBarrierBytes;
  static_assert(kPlane % 1024 == 0, "swizzle atoms stay aligned");
  static_assert(kRows % kFetchRows == 0 && kRowsPerTask % kFetchRows == 0, "a group of copies lies in one stage");
  // (a float window has at least 2 x 32 / 16 = 4 groups)
  static_assert(kFetchGroups < 4 && kFetchGroups < kHalfPerTask * (kRowsPerTask / kFetchRows),
                "the copies in flight reach at most into the next sub-task");
  static_assert(kPlane % (kNegWarps * 32 * 16) == 0, "the negation's passes are whole");
  static_assert((3 * kStages + 5) * 8 + 8 + 16 + 16 * kSinkSlots + 16 <= kBarrierBytes, "barrier area");
  static_assert(kWindow % kRows == 0 && kMaxChunk % kRows == 0, "windows and chunks are whole stages");
  static_assert(kSmem <= 232448, "shared memory budget");
};

// The digit planes (p, q) of each block of a float window: the products d_p d_q with p + q <= 2.
__device__ __forceinline__ int digit_p(int pk) { return (0x120100 >> (4 * pk)) & 15; }
__device__ __forceinline__ int digit_q(int pk) { return (0x102010 >> (4 * pk)) & 15; }

struct P2Params {
  int n_chan, n_inputs, n_time;
  int nb;                // tiles per side
  ring::Order order;
  int n_kt;              // stages along time
  int chunk;             // samples per ring chunk (a multiple of the stage)
  int subs;              // unpack sub-tasks per chunk
  int halves;            // 64-input halves: two per tile
  int64_t slot_bytes;
  uint8_t* ring;
  int* ready;            // [u]: finished unpack sub-tasks
  int* done;             // [u]: CTAs that have read the chunk (only while slots are reused)
  int* leavers;          // CTAs that have left
  int n_flags;
  int reuse;             // the ring is shorter than the launch's chunks
  int vec;               // 16-byte aligned rows
  int row_bytes;         // one sample of one channel
  int64_t row_step;      // bytes from one sample to the next
  int unit_cols;         // 128-byte columns of a row
  int col_splits;        // sub-tasks a row is cut into (integer formats)
  const uint8_t* in;
  int64_t n_pairs;
  void* out;             // int2 or float2 [C][P]
  int* status;
  int16_t* exps;         // float input: window exponents [C][exp_windows][exp_pitch]
  int exp_windows, exp_pitch;
};

__device__ __forceinline__ int flag_load(const int* f) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(f) : "memory");
  return v;
}
__device__ __forceinline__ void flag_add(int* f) {
  asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(f) : "memory");
}
// The same without a release: for a CTA that has only read (its copies were waited for).  A release
// here would stall the producer for over a thousand cycles per chunk.
__device__ __forceinline__ void flag_add_relaxed(int* f) {
  asm volatile("red.relaxed.gpu.global.add.s32 [%0], 1;" ::"l"(f) : "memory");
}
// Bounded wait for *f >= target.
__device__ __forceinline__ bool flag_wait(const int* f, int target, volatile int* abort_flag, int* status, int code) {
  if (flag_load(f) >= target) return true;
  const uint64_t t0 = global_ns();
  for (uint32_t spin = 0;; ++spin) {
    if (flag_load(f) >= target) return true;
    if ((spin & 15u) == 15u) {
      if (*abort_flag) return false;
      if (global_ns() - t0 > kWaitLimitNs) {
        *abort_flag = 1;
        atomicCAS(status, DEV_OK, code);
        return false;
      }
    }
  }
}

// Contiguous copy of `bytes` from global to this CTA's shared memory, completing on `bar`.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// The ring's layout is the shared-memory image of the operands, so that a stage is two contiguous
// copies (tensor-map copies of the same tiles ran at 353-614 cycles per step, by how many boxes a
// stage took): per slot [stage][digit][half of 64 inputs][re | im][sample][64 inputs], the rows'
// 16-byte units swizzled as the MMA descriptors say (64-byte pattern for E4M3, 128-byte for BF16).
template <int FMT>
__device__ __forceinline__ int64_t plane_at(const P2Params& p, int stage, int digit, int half) {
  using G = Geom<FMT>;
  return (((int64_t)stage * G::kDigits + digit) * p.halves + half) * (2 * G::kPlane);
}

// ------------------------------------------------------------------ unpack --
// An unpack sub-task: 32 samples x 4 columns of a channel (integer formats) or 16 inputs of a float
// window (two passes over it).  They are dealt round robin over every CTA's unpack warps.
struct Task {
  int u, sub;          // place in the unpack order; which part of the chunk
  int chan, k;         // channel, chunk along time
  const uint8_t* src;  // its first sample, the channel's first input
  int live;            // samples before n_time
  int prev;            // the place that had the slot before, or -1
  int done, readers;   // its readers: finished (as last seen), in all
};

// Bring x.u, x.sub to the first sub-task at or after them that has any reader; false at the end.
template <int FMT>
__device__ __forceinline__ bool task_seek(const P2Params& p, Task& x, int n_warps, int n_places) {
  for (;; x.sub += n_warps) {
    x.u += x.sub / p.subs;
    x.sub %= p.subs;
    if (x.u >= n_places) return false;
    if (ring::readers_of(p.order, x.u) > 0) break;
  }
  const int j = x.u % p.order.batch_chans, bk = x.u / p.order.batch_chans;
  const int batch = bk / p.order.n_chunks;
  x.k = bk - batch * p.order.n_chunks;
  x.chan = ring::first_chan(p.order, batch) + j;
  const int t = x.k * p.chunk + (FMT == XCORR_IN_CF32 ? 0 : x.sub / p.col_splits * kRowsPerTask);
  x.src = p.in + ((int64_t)t * p.n_chan + x.chan) * p.row_bytes;
  x.live = p.n_time - t;
  x.done = x.readers = 0;
  x.prev = ring::slot_user(p.order, x.u);
  if (x.prev >= 0) {  // looked up when the sub-task's first copies start, used when they have arrived
    x.readers = ring::readers_of(p.order, x.prev);
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(x.done) : "l"(p.done + x.prev) : "memory");
  }
  return true;
}

// Group g of a sub-task: its first row and 8-unit column.
template <int FMT>
__device__ __forceinline__ void group_at(const P2Params& p, int sub, int g, int& row, int& col) {
  if (FMT == XCORR_IN_CF32) {
    const int n = p.chunk / kFetchRows;
    row = (g >= n ? g - n : g) * kFetchRows;
    col = sub;
  } else {
    constexpr int kPer = kRowsPerTask / kFetchRows;
    row = g % kPer * kFetchRows;
    col = sub % p.col_splits * kHalfPerTask + g / kPer;
  }
}

// Whether no lane copies the unit after the one at `off`: the last of a column, or of the row.
__device__ __forceinline__ bool last_unit(const P2Params& p, int off, int lane) {
  return (lane & 7) == 7 || off + 16 >= p.row_bytes;
}

// Start the copies of a group: lane l takes unit l % 8 of samples l / 8 + 4 i.  Units past the row
// and samples past n_time arrive as zeros (or, unaligned, are not copied).
template <int FMT, bool VEC>
__device__ __forceinline__ void fetch_group(const P2Params& p, const Task& c, int group, uint32_t dst, uint32_t dst_w,
                                            int lane) {
  int row, col;
  group_at<FMT>(p, c.sub, group, row, col);
  const int off = (8 * col + (lane & 7)) * 16;
  const uint8_t* s = c.src + (int64_t)(row + (lane >> 3)) * p.row_step + off;
  const bool have = off < p.row_bytes;
#pragma unroll
  for (int i = 0; i < 4; ++i, s += 4 * p.row_step) {
    const bool in = have && row + (lane >> 3) + 4 * i < c.live;
    if (VEC) {
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + i * 512), "l"(in ? s : p.in),
                   "r"(in ? 16 : 0)
                   : "memory");
    } else {
      // the five 4-byte words around the unit that hold bytes of the row
      const uintptr_t w = reinterpret_cast<uintptr_t>(s) & ~uintptr_t(3);
      const uintptr_t end = reinterpret_cast<uintptr_t>(s) + (p.row_bytes - off);
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        if (k == 4 && !(have && last_unit(p, off, lane))) break;  // the next lane's first word
        const bool ok = in && w + 4 * k < end;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(k < 4 ? dst + i * 512 + 4 * k : dst_w + i * 16),
                     "l"(ok ? reinterpret_cast<const uint8_t*>(w + 4 * k)
                            : reinterpret_cast<const uint8_t*>(reinterpret_cast<uintptr_t>(p.in) & ~uintptr_t(3))),
                     "r"(ok ? 4 : 0)
                     : "memory");
      }
    }
  }
}

// The unit copied by fetch_group's copy i (its bytes shifted into place when the row is unaligned).
template <bool VEC>
__device__ __forceinline__ uint4 fetched(const P2Params& p, const Task& c, int row, int col, int lane, const uint4* buf,
                                         const uint32_t* buf_w, int i) {
  const uint4 v = buf[i * 32];
  if (VEC) return v;
  uint32_t w = __shfl_down_sync(0xFFFFFFFFu, v.x, 1);
  if (last_unit(p, (8 * col + (lane & 7)) * 16, lane)) w = buf_w[i * 4];
  const uint32_t sh =
      static_cast<uint32_t>((reinterpret_cast<uintptr_t>(c.src) + (int64_t)(row + (lane >> 3) + 4 * i) * p.row_step) & 3) * 8;
  return make_uint4(__funnelshift_r(v.x, v.y, sh), __funnelshift_r(v.y, v.z, sh), __funnelshift_r(v.z, v.w, sh),
                    __funnelshift_r(v.w, w, sh));
}

// The unpack warps: raw samples stream through shared memory by asynchronous copies that run three
// groups ahead (24 KB per SM in flight) across sub-tasks, so that HBM's latency is not waited for.
template <int FMT, bool VEC>
__device__ __forceinline__ void unpack_role(const P2Params& p, uint8_t* fetch, int uw, int lane,
                                            volatile int* abort_flag) {
  using G = Geom<FMT>;
  constexpr bool FLOAT = FMT == XCORR_IN_CF32;
  const int n_places = ring::places(p.order);
  const int n_warps = static_cast<int>(gridDim.x) * kUnpackWarps;
  const int n_groups = FLOAT ? 2 * (p.chunk / kFetchRows) : kHalfPerTask * (kRowsPerTask / kFetchRows);
  uint4* buf = reinterpret_cast<uint4*>(fetch) + uw * (kFetchGroups * 128) + lane;
  uint32_t* buf_w = reinterpret_cast<uint32_t*>(fetch + kFetchSlots * 16) + uw * (kFetchGroups * 16) + (lane >> 3);
  const int row_lane = lane >> 3, unit_lane = lane & 7;
  // f: the sub-task being copied; c: the one being unpacked, the same or the one before (a sub-task
  // has more groups than are in flight)
  Task f{};
  f.sub = static_cast<int>(blockIdx.x) * kUnpackWarps + uw;
  bool more = task_seek<FMT>(p, f, n_warps, n_places);
  int fg = 0, cg = 0;  // their next groups
  Task c = f;
  bool run = more;
  auto fetch_next = [&](int d) {
    if (!more) return;
    fetch_group<FMT, VEC>(p, f, fg, smem_u32(buf + d * 128), smem_u32(buf_w + d * 16), lane);
    if (++fg == n_groups) {
      fg = 0;
      f.sub += n_warps;
      more = task_seek<FMT>(p, f, n_warps, n_places);
    }
  };
#pragma unroll
  for (int d = 0; d < kFetchGroups; ++d) {
    fetch_next(d);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  int d = 0;
  uint8_t* slot = nullptr;
  uint32_t m0 = 0u, m1 = 0u;  // float: largest magnitudes of this lane's two inputs
  float s0a = 0.f, s0b = 0.f, s1a = 0.f, s1b = 0.f;
  while (run) {
    if (cg == 0) {
      // the slot's previous chunk is still being read (every lane looked for itself, at its own time)
      if (__any_sync(0xFFFFFFFFu, c.done < c.readers)) {
        bool ok = true;
        if (lane == 0)
          ok = flag_wait(p.done + c.prev, c.readers, abort_flag, p.status, DEV_TIMEOUT_EMPTY);
        if (!__all_sync(0xFFFFFFFFu, ok)) break;
      }
      asm volatile("fence.proxy.async;" ::: "memory");  // the slot's TMA reads before these writes
      slot = p.ring + (int64_t)(c.u % p.order.slots) * p.slot_bytes;
      m0 = m1 = 0u;
    }
    int row, col;
    group_at<FMT>(p, c.sub, cg, row, col);
    asm volatile("cp.async.wait_group %0;" ::"n"(kFetchGroups - 1) : "memory");
    const uint4* b = buf + d * 128;
    const uint32_t* bw = buf_w + d * 16;
    uint4 v[4];  // all four before any store, so that they do not wait for one another
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = fetched<VEC || FLOAT>(p, c, row, col, lane, b, bw, i);
    if (!FLOAT) {
      const int unit = 8 * col + unit_lane, s0 = c.sub / p.col_splits * kRowsPerTask + row;  // first sample within the chunk
      const int half = unit / (G::kRowB / 16), pos = unit % (G::kRowB / 16);
      const int stage = s0 / G::kRows, r0 = s0 - stage * G::kRows + row_lane;
      uint8_t* dst = slot + plane_at<FMT>(p, stage, 0, half) + r0 * G::kRowB;
      const bool have = unit * 16 < p.row_bytes;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        uint4 re, im;
        decode_ci4(v[i], re, im);
        const int r = r0 + 4 * i;
        uint8_t* q = dst + 4 * i * G::kRowB + ((pos ^ ((r >> 1) & 3)) << 4);
        if (have) {
          *reinterpret_cast<uint4*>(q) = re;
          *reinterpret_cast<uint4*>(q + G::kPlane) = im;
        }
      }
    } else if (cg < n_groups / 2) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        m0 = max(m0, max(v[i].x & 0x7FFFFFFFu, v[i].y & 0x7FFFFFFFu));
        m1 = max(m1, max(v[i].z & 0x7FFFFFFFu, v[i].w & 0x7FFFFFFFu));
      }
      if (cg == n_groups / 2 - 1) {  // the window's exponents
#pragma unroll
        for (int x = 8; x <= 16; x <<= 1) {
          m0 = max(m0, __shfl_xor_sync(0xFFFFFFFFu, m0, x));
          m1 = max(m1, __shfl_xor_sync(0xFFFFFFFFu, m1, x));
        }
        const int e0 = window_exponent(m0), e1 = window_exponent(m1);
        const int in = 16 * col + 2 * unit_lane;
        if (row_lane == 0 && in < p.n_inputs) {
          *reinterpret_cast<uint32_t*>(p.exps + ((int64_t)c.chan * p.exp_windows + c.k) * p.exp_pitch + in) =
              (static_cast<uint32_t>(e0) & 0xFFFFu) | (static_cast<uint32_t>(e1) << 16);
        }
        window_scale(e0, s0a, s0b);
        window_scale(e1, s1a, s1b);
      }
    } else {
      const int in = 16 * col + 2 * unit_lane;
      const int half = in >> 6, pos = (in & 63) >> 3, byte = (in & 7) * 2;
      const int stage = row / G::kRows, r0 = row - stage * G::kRows + row_lane;
      uint8_t* dst = slot + plane_at<FMT>(p, stage, 0, half) + r0 * G::kRowB + byte;
      const int64_t digit = plane_at<FMT>(p, 0, 1, 0);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        uint32_t re[3], im[3];
        digit_pairs(__uint_as_float(v[i].x), s0a, s0b, __uint_as_float(v[i].z), s1a, s1b, re);
        digit_pairs(__uint_as_float(v[i].y), s0a, s0b, __uint_as_float(v[i].w), s1a, s1b, im);
        const int r = r0 + 4 * i;
        uint8_t* q = dst + 4 * i * G::kRowB + ((pos ^ (r & 7)) << 4);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          *reinterpret_cast<uint32_t*>(q + k * digit) = re[k];
          *reinterpret_cast<uint32_t*>(q + k * digit + G::kPlane) = im[k];
        }
      }
    }
    fetch_next(d);
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (++d == kFetchGroups) d = 0;
    if (++cg == n_groups) {
      // generic writes, read by other SMs' copies: every lane's are ordered before lane 0's release
      asm volatile("fence.proxy.async.global;" ::: "memory");
      __syncwarp();
      if (lane == 0) flag_add(p.ready + c.u);
      __syncwarp();
      run = f.u < n_places;  // the next sub-task, if there is one: its first copies are in flight
      c = f;
      cg = 0;
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// ADD: the launch adds into out (else it stores).
template <int FMT, bool ADD>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    xcorr_tc_pair_kernel(const __grid_constant__ P2Params p) {
  using G = Geom<FMT>;
  constexpr bool FLOAT_OUT = FMT == XCORR_IN_CF32;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* stages = smem;
  uint2* staging = reinterpret_cast<uint2*>(smem + G::kOffStaging);
  float* factors = reinterpret_cast<float*>(smem + G::kOffFactors);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + G::kOffBarriers);  // this CTA's copies have landed
  uint64_t* ready = full + kStages;   // even CTA: both CTAs' stages are complete, negated half included
  uint64_t* empty = ready + kStages;  // both CTAs: the pair's MMAs are done with the stage
  uint64_t* tfull = empty + kStages;  // [2] both CTAs: an accumulator holds a block
  uint64_t* tempty = tfull + 2;       // [2] even CTA: both epilogues have it out
  uint64_t* mma_done = tempty + 2;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(mma_done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
  uint8_t* token = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(tslot + 2) + 15) & ~uintptr_t(15));
  uint8_t* sink = token + kSignalBytes;  // [kSinkSlots][16], written by the odd CTA's signals

  const uint32_t rank = cluster_ctarank();
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&ready[s], kNegWarps);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], kEpiWarps);
    }
    mbar_init(mma_done, 1);
    for (int k = 0; k < 4; ++k) reinterpret_cast<uint32_t*>(token)[k] = 0u;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the token is read by the async proxy
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == kMmaWarp) tmem_alloc_pair(tslot, kTmemCols);
  tc_fence_before();
  cluster_sync();  // both CTAs' barriers and tensor memory exist before either touches the other's
  tc_fence_after();
  const uint32_t tmem = *tslot;
  const int n_items = p.order.n_items, n_entries = p.order.n_entries;
  const int cl = static_cast<int>(blockIdx.x >> 1), n_cl = static_cast<int>(gridDim.x >> 1);
  const int n_tw = (p.n_kt + G::kSpw - 1) / G::kSpw;
  const int n_blocks = n_tw * G::kPairsK;  // drained blocks per item: (window, plane pair)

  // registers: launched with 128 a thread; the two epilogue warpgroups hold 128 running sums a
  // thread and take 184, the other two give up the difference (184 + 184 + 72 + 72 = 4 x 128)
  if (warp < kEpiWarps) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 184;");
    using Acc = typename std::conditional<FLOAT_OUT, float, int>::type;
    uint2* stage_rows = staging + warp * 32 * kOutPitch;
    float* col_f = factors + warp * kHalf;
    const int quarter = warp & 3, colh = warp >> 2;
    const uint32_t tempty_even = smem_cluster(tempty, 0);
    const uint32_t sink_even = smem_cluster(sink + kSignalBytes * (kNegWarps + warp), 0);
    const int n_inputs = p.n_inputs;
    int g = 0;
    bool ok = true;
    for (int q = cl; ok && q < n_items; q += n_cl) {
      const Item it = item_of(p.nb, n_entries, q, rank);
      uint2* out_c = static_cast<uint2*>(p.out) + (int64_t)it.chan * p.n_pairs;
      const int row0 = it.R * kBlk + quarter * 32;  // first global row of this warp
      const int col0 = it.S * kBlk + colh * kHalf;  // first global column of this warp
      const bool live = it.has_row && row0 < n_inputs && col0 < n_inputs && (it.transposed || col0 <= row0 + 31);
      Acc acc_re[kHalf], acc_im[kHalf];
#pragma unroll
      for (int k = 0; k < kHalf; ++k) acc_re[k] = acc_im[k] = Acc(0);
      // float input: the window's exponents of this lane's row and, for the slow path, its columns
      const int16_t* exps_w = nullptr;
      int e_row = 0;
      bool fast = true;
      for (int blk = 0; blk < n_blocks; ++blk, ++g) {
        const int buf = g & 1;
        if (!mbar_wait_warp(&tfull[buf], (g >> 1) & 1, abort_flag, p.status, DEV_TIMEOUT_TMEM_FULL)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t taddr =
            tmem + (static_cast<uint32_t>(quarter * 32) << 16) + buf * kAccCols + colh * 2 * kHalf;
        if (FLOAT_OUT) {
          // a block's exact integer sums times 2^k, k = E_i + E_j - 12 - 8(p + q).  While every
          // exponent of the window's rows and columns lies in [-45, 45] (kept per window), 2^k is a
          // normal float and the product exact, so one multiply-add by the product of a row and a
          // column factor gives the bits of the general form; it halves the drain.  The general
          // form applies 2^k in two factors (k in [-342, 242]): see xcorr_tc.cu.
          const int w = blk / G::kPairsK, pk = blk - w * G::kPairsK;
          if (pk == 0) {
            exps_w = p.exps + ((int64_t)it.chan * p.exp_windows + w) * p.exp_pitch;
            const int ir = max(0, min(row0 + lane, n_inputs - 1));
            const int c_lo = min(col0 + lane, n_inputs - 1), c_hi = min(col0 + 32 + lane, n_inputs - 1);
            e_row = __ldcg(exps_w + ir);
            const int ea = __ldcg(exps_w + c_lo), eb = __ldcg(exps_w + c_hi);
            fast = __all_sync(0xFFFFFFFFu, abs(e_row) <= 45 && abs(ea) <= 45 && abs(eb) <= 45);
            __syncwarp();
            col_f[lane] = fast ? pow2i(ea) : __int_as_float(ea);
            col_f[lane + 32] = fast ? pow2i(eb) : __int_as_float(eb);
            __syncwarp();
          }
          const int row_k = e_row - 12 - 8 * (digit_p(pk) + digit_q(pk));
          if (fast) {
            const float rf = pow2i(row_k);
#pragma unroll
            for (int k = 0; k < kHalf / 8; ++k) {
              uint32_t re[8], nim[8];
              tmem_ld8(taddr + 8 * k, re);
              tmem_ld8(taddr + kHalf + 8 * k, nim);
              const float4 f0 = *reinterpret_cast<const float4*>(col_f + 8 * k);
              const float4 f1 = *reinterpret_cast<const float4*>(col_f + 8 * k + 4);
              const float f[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
              tmem_ld_wait();
              if (!live) continue;
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const float s = rf * f[j];
                acc_re[8 * k + j] = fmaf(__uint_as_float(re[j]), s, acc_re[8 * k + j]);
                acc_im[8 * k + j] = fmaf(-__uint_as_float(nim[j]), s, acc_im[8 * k + j]);
              }
            }
          } else {
            const bool row_bad = e_row == kExpNonFinite;
#pragma unroll
            for (int k = 0; k < kHalf / 8; ++k) {
              uint32_t re[8], nim[8];
              tmem_ld8(taddr + 8 * k, re);
              tmem_ld8(taddr + kHalf + 8 * k, nim);
              tmem_ld_wait();
              if (!live) continue;
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const int ej = __float_as_int(col_f[8 * k + j]);
                // below -298 a block's contribution rounds to zero either way
                const int kk = max(row_k + ej, -298);
                const float f1 = (row_bad || ej == kExpNonFinite) ? __int_as_float(0x7FC00000) : pow2i(kk >> 1);
                const float f2 = pow2i(kk - (kk >> 1));
                acc_re[8 * k + j] += (__uint_as_float(re[j]) * f1) * f2;
                acc_im[8 * k + j] -= (__uint_as_float(nim[j]) * f1) * f2;
              }
            }
          }
        } else {
#pragma unroll
          for (int k = 0; k < kHalf / 8; ++k) {
            uint32_t re[8], nim[8];
            tmem_ld8(taddr + 8 * k, re);
            tmem_ld8(taddr + kHalf + 8 * k, nim);
            tmem_ld_wait();
            if (!live) continue;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              acc_re[8 * k + j] += __float2int_rn(__uint_as_float(re[j]));
              acc_im[8 * k + j] -= __float2int_rn(__uint_as_float(nim[j]));
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (rank != 0)
            bulk_copy_to_cluster(sink_even, token, kSignalBytes, tempty_even + 8u * static_cast<uint32_t>(buf));
          else if (warp == 0)
            mbar_expect_tx(&tempty[buf], kEpiWarps * kSignalBytes);
          else
            mbar_arrive(&tempty[buf]);
        }
      }
      if (!ok || !live) continue;
      RowsOut ro;
      ColsOut co;
      if (it.transposed)
        cols_out(co, out_c, row0, col0, n_inputs, lane);
      else
        rows_out(ro, out_c, row0, col0, n_inputs, lane);
#pragma unroll
      for (int ch = 0; ch < kHalf; ch += 8) {
        uint2 v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const Acc vr = acc_re[ch + k], vi = it.transposed ? -acc_im[ch + k] : acc_im[ch + k];
          v[k] = FLOAT_OUT ? make_uint2(__float_as_uint(vr), __float_as_uint(vi))
                           : make_uint2(static_cast<uint32_t>(vr), static_cast<uint32_t>(vi));
        }
        if (it.transposed)
          put_cols<FLOAT_OUT, ADD>(co, v);
        else
          put_rows<FLOAT_OUT, ADD>(ro, stage_rows, v, ch, lane);
      }
    }
  } else if (warp < kUnpackWarp0) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    if (warp == kProducerWarp) {
      if (lane == 0) {
        // one thread feeds a stage every 512 cycles: all index arithmetic is per chunk or plane pair
        const int spc = p.chunk / G::kRows;  // stages per ring chunk
        const int64_t stage_step = plane_at<FMT>(p, 1, 0, 0);
        int s = 0;
        uint32_t ph = 0, filled = 0, fill_parity = 0;  // bit s: the stage was filled, and with which parity
        ring::Reads reads;  // (kept only while slots are reused)
        // tell the unpack warps that a chunk is read; landed: its copies are known to have landed
        auto report = [&](bool landed) {
          const int ps = (reads.end - 1) % kStages;
          if (!landed && !mbar_wait(&full[ps], (fill_parity >> ps) & 1u, abort_flag, p.status, DEV_TIMEOUT_FULL))
            return false;
          flag_add_relaxed(p.done + reads.place);
          reads.reported();
          return true;
        };
        bool ok = true;
        for (int q = cl, batch = 0; ok && q < n_items; q += n_cl, ++batch) {
          const Item it = item_of(p.nb, n_entries, q, rank);
          const int j = it.chan - ring::first_chan(p.order, batch);
          const uint32_t bytes = (it.has_row ? 4 * G::kPlane : 0) + 2 * G::kPlane;
          for (int k = 0; ok && k < p.order.n_chunks; ++k) {
            const int u = ring::place_of(p.order, batch, k, j);
            if (flag_load(p.ready + u) < p.subs) {  // it has not been unpacked
              if ((reads.due_before_wait(false) && !report(false)) ||
                  !flag_wait(p.ready + u, p.subs, abort_flag, p.status, DEV_TIMEOUT_FULL)) {
                ok = false;
                break;
              }
            }
            asm volatile("fence.proxy.async;" ::: "memory");  // generic writes, read by the copies
            const uint8_t* sl = p.ring + (int64_t)(u % p.order.slots) * p.slot_bytes;
            const int n_st = min(spc, p.n_kt - k * spc);
            for (int pk = 0; ok && pk < G::kPairsK; ++pk) {
              const uint8_t* a = sl + plane_at<FMT>(p, 0, FLOAT_OUT ? digit_p(pk) : 0, 2 * it.R);
              const uint8_t* b = sl + plane_at<FMT>(p, 0, FLOAT_OUT ? digit_q(pk) : 0, 2 * it.S + static_cast<int>(rank));
              for (int st = 0; st < n_st; ++st, a += stage_step, b += stage_step) {
                if (!mbar_wait(&empty[s], ph ^ 1u, abort_flag, p.status, DEV_TIMEOUT_EMPTY)) {
                  ok = false;
                  break;
                }
                uint8_t* dst = stages + s * G::kStageBytes;
                mbar_expect_tx(&full[s], bytes);
                bulk_load(dst + G::kOffB, b, 2 * G::kPlane, &full[s]);
                if (it.has_row) bulk_load(dst, a, 4 * G::kPlane, &full[s]);
                fill_parity = (fill_parity & ~(1u << s)) | (ph << s);
                filled |= 1u << s;
                if (++s == kStages) {
                  s = 0;
                  ph ^= 1u;
                }
                if (reads.due_after_stage(kStages)) report(true);  // its last stage's buffer has come round
              }
            }
            if (ok && p.reuse) {
              if (reads.due_after_chunk() && !report(false)) {  // a chunk shorter than the stage ring
                ok = false;
                break;
              }
              reads.chunk_read(u);
            }
          }
        }
        // Let every copy this CTA issued land before the CTA can exit.
        volatile int never = 0;
        for (int k = 0; k < kStages; ++k)
          if (filled & (1u << k)) mbar_wait(&full[k], (fill_parity >> k) & 1u, &never, p.status, DEV_TIMEOUT_DRAIN);
        if (reads.due_after_chunk()) report(true);
      }
    } else if (warp >= kNegWarp0) {
      // -B_re: the real half-tile with the sign bits flipped, at the same swizzled offsets
      const int nw = warp - kNegWarp0, tid = nw * 32 + lane;
      constexpr int kPasses = G::kPlane / (kNegWarps * 32 * 16);
      const uint32_t ready_even = smem_cluster(ready, 0);
      const uint32_t sink_even = smem_cluster(sink + kSignalBytes * nw, 0);
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int q = cl; ok && q < n_items; q += n_cl) {
        for (int n = 0; n < p.n_kt * G::kPairsK; ++n) {  // the item's stages
          if (!mbar_wait_warp(&full[s], ph, abort_flag, p.status, DEV_TIMEOUT_FULL)) {
            ok = false;
            break;
          }
          const uint4* src = reinterpret_cast<const uint4*>(stages + s * G::kStageBytes + G::kOffB);
          uint4* dst = reinterpret_cast<uint4*>(stages + s * G::kStageBytes + G::kOffB + 2 * G::kPlane);
          uint4 v[kPasses];
#pragma unroll
          for (int k = 0; k < kPasses; ++k) v[k] = src[tid + k * kNegWarps * 32];
#pragma unroll
          for (int k = 0; k < kPasses; ++k)
            dst[tid + k * kNegWarps * 32] = make_uint4(v[k].x ^ G::kSignMask, v[k].y ^ G::kSignMask,
                                                       v[k].z ^ G::kSignMask, v[k].w ^ G::kSignMask);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) {
            if (rank != 0)
              bulk_copy_to_cluster(sink_even, token, kSignalBytes, ready_even + 8u * static_cast<uint32_t>(s));
            else if (nw == 0)
              mbar_expect_tx(&ready[s], kNegWarps * kSignalBytes);
            else
              mbar_arrive(&ready[s]);
          }
          if (++s == kStages) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
    } else if (rank == 0 && lane == 0) {
      const uint32_t idesc = instr_desc(G::E == 1 ? kTypeE4M3 : kTypeBF16, true, 256, 256, false);
      int s = 0;
      uint32_t ph = 0;
      int g = 0;  // blocks started by this pair
      bool ok = true;
      for (int q = cl; ok && q < n_items; q += n_cl) {
        for (int blk = 0; ok && blk < n_blocks; ++blk, ++g) {
          const int w = blk / G::kPairsK;
          const int buf = g & 1;
          if (!mbar_wait(&tempty[buf], ((g >> 1) & 1) ^ 1, abort_flag, p.status, DEV_TIMEOUT_TMEM_EMPTY)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d = tmem + static_cast<uint32_t>(buf * kAccCols);
          const int kb0 = w * G::kSpw, kb1 = min(p.n_kt, kb0 + G::kSpw);
          for (int kb = kb0; kb < kb1; ++kb) {
            if (!mbar_wait(&ready[s], ph, abort_flag, p.status, DEV_TIMEOUT_FULL)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t a_r = smem_u32(stages + s * G::kStageBytes);
            const uint32_t b_r = a_r + G::kOffB;
            // the start address fields count 16 bytes
            const uint64_t da_r = G::E == 1 ? smem_desc_sw64(a_r, 2 * G::kPlane, 8 * G::kRowB)
                                            : smem_desc_sw128(a_r, 2 * G::kPlane, 8 * G::kRowB);
            const uint64_t da_i = da_r + (G::kPlane >> 4);
            const uint64_t db_r = G::E == 1 ? smem_desc_sw64(b_r, G::kPlane, 8 * G::kRowB)
                                            : smem_desc_sw128(b_r, G::kPlane, 8 * G::kRowB);
            const uint64_t db_i = db_r + (G::kPlane >> 4);
#pragma unroll
            for (int k = 0; k < G::kSteps; ++k) {
              const uint64_t o = static_cast<uint64_t>((k * G::kMmaK * G::kRowB) >> 4);
              mma_pair<G::E>(d, da_r + o, db_r + o, idesc, (kb == kb0 && k == 0) ? 0u : 1u);
              mma_pair<G::E>(d, da_i + o, db_i + o, idesc, 1u);
            }
            mma_pair_commit_both(&empty[s]);
            if (++s == kStages) {
              s = 0;
              ph ^= 1u;
            }
          }
          if (ok) mma_pair_commit_both(&tfull[buf]);
        }
      }
      // the odd CTA's last signals land here once both epilogues have drained the last blocks
      for (int k = g > 2 ? g - 2 : 0; ok && k < g; ++k)
        ok = mbar_wait(&tempty[k & 1], (k >> 1) & 1, abort_flag, p.status, DEV_TIMEOUT_TMEM_EMPTY);
      // the pair's MMAs write both CTAs' tensor memory: let them finish before the cluster barrier
      volatile int never = 0;
      mma_pair_commit_both(mma_done);
      mbar_wait(mma_done, 0, &never, p.status, DEV_TIMEOUT_DRAIN);
    }
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    if (p.vec)
      unpack_role<FMT, true>(p, smem + G::kOffFetch, warp - kUnpackWarp0, lane, abort_flag);
    else
      unpack_role<FMT, false>(p, smem + G::kOffFetch, warp - kUnpackWarp0, lane, abort_flag);
  }

  tc_fence_before();
  cluster_sync();  // no remote signal or MMA of either CTA is still in flight
  if (*abort_flag) {
    // a pipeline that gave up may leave signal copies between the CTAs in flight: let them land
    const uint64_t t_end = global_ns() + 20000;
    while (global_ns() < t_end) {
    }
  }
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, kTmemCols);
  }
  // the last CTA to leave clears the flags for the next launch
  if (threadIdx.x == 0) {
    __threadfence();
    *tslot = atomicAdd(p.leavers, 1) == static_cast<int>(gridDim.x) - 1 ? 1u : 0u;
  }
  __syncthreads();
  if (*reinterpret_cast<volatile uint32_t*>(tslot)) {
    __threadfence();
    for (int k = threadIdx.x; k < p.n_flags; k += kThreads) p.ready[k] = p.done[k] = 0;
    if (threadIdx.x == 0) *p.leavers = 0;
  }
}

template <int FMT, bool ADD>
cudaError_t pair_clusters(int* n) {
  using G = Geom<FMT>;
  auto kern = xcorr_tc_pair_kernel<FMT, ADD>;
  static PerDevice<1> most;
  std::array<int, 1> clusters{};
  const cudaError_t e = most.get(&clusters, [kern](std::array<int, 1>& m) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, G::kSmem);
    if (e != cudaSuccess) return e;
    // pairs of SMs that can hold one CTA each at the same time
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(2 * 1024);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = G::kSmem;
    e = cudaOccupancyMaxActiveClusters(&m[0], kern, &cfg);
    return e == cudaSuccess && m[0] < 1 ? cudaErrorLaunchOutOfResources : e;
  });
  *n = clusters[0];
  return e;
}

template <int FMT, bool ADD>
cudaError_t launch_pair(const P2Params& p, int n_cl, cudaStream_t stream) {
  int most = 0;
  cudaError_t e = pair_clusters<FMT, ADD>(&most);
  if (e != cudaSuccess) return e;
  if (n_cl > most) return cudaErrorCooperativeLaunchTooLarge;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(2 * n_cl));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = Geom<FMT>::kSmem;
  cfg.stream = stream;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeCooperative;
  attr.val.cooperative = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, xcorr_tc_pair_kernel<FMT, ADD>, p);
}

}  // namespace

cudaError_t pair_ring_layout(int fmt, int n_inputs, int n_chan, int max_time, size_t most_bytes, PairRing* r) {
  int n_cl = 0, n_add = 0;
  cudaError_t e;
  if (fmt == XCORR_IN_CI4) {
    e = pair_clusters<XCORR_IN_CI4, false>(&n_cl);
    if (e == cudaSuccess) e = pair_clusters<XCORR_IN_CI4, true>(&n_add);
  } else {
    e = pair_clusters<XCORR_IN_CF32, false>(&n_cl);
    if (e == cudaSuccess) e = pair_clusters<XCORR_IN_CF32, true>(&n_add);
  }
  if (e != cudaSuccess) return e;
  if (n_add < n_cl) n_cl = n_add;
  const int elem = fmt == XCORR_IN_CI4 ? 1 : 2, rows = 64 / elem, planes = fmt == XCORR_IN_CF32 ? 6 : 2;
  const int most_chunk = fmt == XCORR_IN_CI4 ? Geom<XCORR_IN_CI4>::kMaxChunk : Geom<XCORR_IN_CF32>::kMaxChunk;
  const int nb = (n_inputs + kBlk - 1) / kBlk, ne = pair_entries(nb);
  const int64_t items = (int64_t)n_chan * ne;
  if (items > 0x7FFFFFFF / 2) return cudaErrorNotSupported;
  r->clusters = static_cast<int>(items < n_cl ? items : n_cl);
  r->halves = 2 * nb;
  const int t_rows = (max_time + rows - 1) / rows * rows;
  r->chunk = t_rows < most_chunk ? t_rows : most_chunk;
  const int64_t chunks = (max_time + r->chunk - 1) / r->chunk;
  const ring::Order one = ring::make_order(n_chan, ne, r->clusters, 1, 1);  // (of one chunk along time)
  r->batch_chans = one.batch_chans;
  const int64_t places = chunks * ring::places(one);
  if (places > kRingPlaces) return cudaErrorNotSupported;
  r->places = static_cast<int>(places);
  r->slot_bytes = (size_t)planes * r->chunk * r->halves * kHalf * elem;
  // at least three batch-wide steps of chunks, and as many as fit kRingBytes (L2 holds them)
  int64_t slots = (int64_t)(kRingBytes / r->slot_bytes);
  if (slots < 3 * (int64_t)r->batch_chans) slots = 3 * (int64_t)r->batch_chans;
  if (slots > places) slots = places;
  const size_t flag_bytes = (2 * (size_t)places + 64) * sizeof(int);
  // a memory budget may shorten the ring, down to one step
  while (slots > r->batch_chans && most_bytes && (size_t)slots * r->slot_bytes + flag_bytes > most_bytes) --slots;
  r->slots = static_cast<int>(slots);
  r->bytes = (size_t)slots * r->slot_bytes;
  r->flag_bytes = flag_bytes;
  return cudaSuccess;
}

cudaError_t launch_xcorr_tc_pair(const PairLaunch& L, cudaStream_t stream) {
  const PairRing& r = *L.ring;
  const int elem = L.fmt == XCORR_IN_CI4 ? 1 : 2, rows = 64 / elem;
  const int in_bytes = L.fmt == XCORR_IN_CI4 ? 1 : 8;
  P2Params p{};
  p.n_chan = L.n_chan;
  p.n_inputs = L.n_inputs;
  p.n_time = L.n_time;
  p.nb = (L.n_inputs + kBlk - 1) / kBlk;
  p.order = ring::make_order(L.n_chan, pair_entries(p.nb), r.clusters, (L.n_time + r.chunk - 1) / r.chunk, r.slots);
  p.n_kt = (L.n_time + rows - 1) / rows;
  p.chunk = r.chunk;
  p.halves = r.halves;
  p.slot_bytes = static_cast<int64_t>(r.slot_bytes);
  p.row_bytes = L.n_inputs * in_bytes;
  p.row_step = static_cast<int64_t>(L.n_chan) * p.row_bytes;
  p.unit_cols = (p.row_bytes + 127) / 128;
  p.col_splits = (p.unit_cols + kHalfPerTask - 1) / kHalfPerTask;
  p.subs = L.fmt == XCORR_IN_CF32 ? p.unit_cols : (r.chunk + kRowsPerTask - 1) / kRowsPerTask * p.col_splits;
  p.ring = static_cast<uint8_t*>(L.ring_mem);
  p.ready = L.flags;
  p.done = L.flags + r.places;
  p.leavers = L.flags + 2 * r.places;
  p.n_flags = ring::places(p.order);
  if (p.n_flags > r.places) return cudaErrorInvalidValue;
  p.reuse = p.n_flags > r.slots ? 1 : 0;
  p.vec = (int64_t)L.n_inputs * in_bytes % 16 == 0 && reinterpret_cast<uintptr_t>(L.in) % 16 == 0;
  p.in = static_cast<const uint8_t*>(L.in);
  p.n_pairs = (int64_t)L.n_inputs * (L.n_inputs + 1) / 2;
  p.out = L.out;
  p.status = L.status;
  p.exps = L.exps;
  p.exp_windows = L.exp_windows;
  p.exp_pitch = L.exp_pitch;
  if (L.fmt == XCORR_IN_CF32 && !L.exps) return cudaErrorInvalidValue;
  switch (L.fmt) {
    case XCORR_IN_CI4:
      return L.accumulate ? launch_pair<XCORR_IN_CI4, true>(p, r.clusters, stream)
                          : launch_pair<XCORR_IN_CI4, false>(p, r.clusters, stream);
    default:
      return L.accumulate ? launch_pair<XCORR_IN_CF32, true>(p, r.clusters, stream)
                          : launch_pair<XCORR_IN_CF32, false>(p, r.clusters, stream);
  }
}

}  // namespace xc
