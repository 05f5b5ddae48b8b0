// xcorr_tc_raw_pair.cu -- the X-stage on CTA pairs with int8 samples unpacked on
// chip, for 16-byte aligned input whose rows are a multiple of 16 bytes.
//
// Same results as the other tensor paths (per channel the packed lower triangle
// of V = sum_t x_t x_t^H; Sec. 1, Sec. 2.1, Eq. 1; the unpack of Sec. 2.4).  The
// MMA scheme is that of xcorr_tc_pair.cu: the two CTAs of a cluster run the tile
// pairs (c, R0, S) and (c, R1, S), the even CTA issues M = 256, N = 256
// cta_group::2 MMAs [Re | X] += A_re [B_re | B_im], [Re | X] += A_im [B_im |
// -B_re] (X = -Im), each CTA provides its own row tile and half of the column
// tile, and two 256-column accumulators let a window's drain overlap the next
// window's MMAs.  Here the operands are decoded from raw samples inside the SM.
//
// What bounds it.  Per MMA step (16 samples; 256 tensor cycles) a CTA's shared
// memory moves 6 KB of raw samples in, 6 KB to the decoders, 14 KB of operands
// back and 16 KB to the tensor core: 42 KB, 328 cycles at 128 bytes per cycle;
// measured 415-420.  Planes from L2 (xcorr_tc_pair.cu) stop at 12 KB per step and
// SM and have to be written first: 480.  One GB300, against unpack + planes kernel
// (us): 512 inputs x 256 channels x 4096 samples 870 (1310), 256 x 256 x 1024 116
// (159), 128 x 300 x 1024 66 (83), 128 x 64 x 1024 23 (29): no unpack launch, no plane
// in memory.  With one tile half of every pair's rows are idle and only half as
// many channels run side by side, so few inputs on many channels go through planes
// (64 x 152 x 4096 105 here, 97 so; ci8_from_planes in xcorr_api.cu has the rule).
//
// Layout.  Everything is cut into half-tiles of 64 inputs, 4 KB of raw samples a
// stage of 32 samples.  TMA lands a raw half-tile with the 128-byte swizzle of
// its operand planes, so 16 raw bytes at some offset (8 inputs' re and im)
// decode into 16 bytes of the real and 16 bytes of the imaginary F16 plane at
// that same offset: a decoder lane owns fixed offsets of every half-tile, and
// loads and stores are contiguous over a warp.  The decode puts v + 128 into the
// low mantissa bits of 1024 and subtracts 1152: exact, two values in two
// instructions.  512-sample windows stay exact in FP32 (2 * 128^2 * 512 = 2^24)
// and are added into int32 running sums in registers.
//
// Two groups of four decoder warps take alternate stages: a stage's waits, fence
// and signals cost a warp as much as several units' decode (one group 543 cycles
// per step, two 420, four 412 with twice the latency per stage).
//
// Warp roles (640 threads, one CTA per SM): warps 0-7 epilogue; warps 8-15
// decode; warp 16 is the TMA producer; warp 17 owns tensor memory and (in the
// even CTA) issues the MMAs.  The odd CTA signals the even one with 16-byte bulk
// copies that complete bytes on its barriers.  Every wait is bounded.
#include "pair_common.cuh"
#include "xcorr_internal.h"

namespace xc {
namespace {

using namespace pairs;
using fused::pair_entries;

constexpr int kDecWarp0 = kEpiWarps;
constexpr int kDecWarps = 8;
constexpr int kDecGroups = 2;      // groups of decoder warps that take alternate stages
constexpr int kGroupWarps = kDecWarps / kDecGroups;
constexpr int kUnits = 4096 / (kGroupWarps * 32 * 16);  // 16-byte units of a half-tile per lane and stage
constexpr int kProducerWarp = kDecWarp0 + kDecWarps;
constexpr int kMmaWarp = kProducerWarp + 1;
constexpr int kThreads = (kProducerWarp + 4) * 32;  // whole warpgroups (setmaxnreg)
constexpr int kPlane = 4096;       // a half-tile's raw samples, and each of its operand planes, per stage
constexpr int kOffB = 4 * kPlane;  // operand stage: [A: 2 x (re | im) | B re | B im | -B re]
constexpr int kOpStage = 7 * kPlane;
constexpr int kRawStage = 3 * kPlane;  // [row tile halves 0, 1 | this CTA's half of the column tile]
constexpr int kRaw = 5, kOps = 4;      // stages of each ring
constexpr int kBarrierBytes = 768;
constexpr int kSinkSlots = kDecWarps + kEpiWarps;
constexpr int kOffOps = kRaw * kRawStage;
constexpr int kOffStaging = kOffOps + kOps * kOpStage;
constexpr int kOffBarriers = kOffStaging + kStagingBytes;
constexpr int kSmem = 1024 + kOffBarriers + kBarrierBytes;
static_assert(kUnits * kGroupWarps * 32 * 16 == kPlane, "a group's lanes cover a half-tile");
static_assert(kOffStaging % 1024 == 0, "buffer alignment");
static_assert((2 * kRaw + 2 * kOps + 5) * 8 + 8 + 32 + 16 * kSinkSlots <= kBarrierBytes, "barrier area");
static_assert(kSmem <= 232448, "shared memory budget");

constexpr int kWindowCI8 = 512;   // samples of one exactly-summed window
constexpr int kRows = 32;         // samples per stage
constexpr int kRowB = kHalf * 2;  // bytes per sample of a half-tile, raw and operand
constexpr int kMmaK = 16;
constexpr int kSpw = kWindowCI8 / kRows;  // stages per window
// registers (5 warpgroups launched with 96 a thread): the epilogue holds 128 running sums a thread
constexpr int kRegsEpi = 168, kRegsDec = 48, kRegsRest = 48;
static_assert(2 * kRegsEpi + 2 * kRegsDec + kRegsRest == 5 * 96, "register split");

struct RParams {
  int n_inputs, nb, n_entries, n_items;
  int n_kt;      // stages per item
  int n_blocks;  // windows per item
  int64_t n_pairs;
  int2* out;     // [C][P]
  int* status;
};

// Int8 samples (re, im interleaved) -> F16 real parts and imaginary parts: two of each per word.
__device__ __forceinline__ uint32_t sub_1152(uint32_t h) {
  uint32_t r;
  asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(h), "r"(0x64806480u));  // 1152 = 0x6480
  return r;
}
__device__ __forceinline__ void ci8_to_f16(uint32_t w, uint32_t& re, uint32_t& im) {
  const uint32_t u = w ^ 0x80808080u;
  re = sub_1152(__byte_perm(u, 0x64646464u, 0x4240));
  im = sub_1152(__byte_perm(u, 0x64646464u, 0x4341));
}

__device__ __forceinline__ void decode16(const uint4& v, uint4& re, uint4& im) {
  ci8_to_f16(v.x, re.x, im.x);
  ci8_to_f16(v.y, re.y, im.y);
  ci8_to_f16(v.z, re.z, im.z);
  ci8_to_f16(v.w, re.w, im.w);
}

// ADD: the launch adds into out (else it stores).
template <bool ADD>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    xcorr_tc_raw_pair_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ RParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* raw = smem;
  uint8_t* ops = smem + kOffOps;
  uint2* staging = reinterpret_cast<uint2*>(smem + kOffStaging);
  uint64_t* raw_full = reinterpret_cast<uint64_t*>(smem + kOffBarriers);
  uint64_t* raw_empty = raw_full + kRaw;
  uint64_t* ready = raw_empty + kRaw;  // even CTA: both CTAs' decoders filled the operand stage
  uint64_t* empty = ready + kOps;      // both CTAs: the pair's MMAs are done with it
  uint64_t* tfull = empty + kOps;      // [2] both CTAs: an accumulator holds a block
  uint64_t* tempty = tfull + 2;        // [2] even CTA: both epilogues have it out
  uint64_t* mma_done = tempty + 2;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(mma_done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
  uint8_t* token = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(tslot + 2) + 15) & ~uintptr_t(15));
  uint8_t* sink = token + kSignalBytes;  // [kSinkSlots][16], written by the odd CTA's signals

  const uint32_t rank = cluster_ctarank();
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kRaw; ++s) {
      mbar_init(&raw_full[s], 1);
      mbar_init(&raw_empty[s], kGroupWarps);
    }
    for (int s = 0; s < kOps; ++s) {
      mbar_init(&ready[s], kGroupWarps);
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
  const int n_items = p.n_items;
  const int cl = static_cast<int>(blockIdx.x >> 1), n_cl = static_cast<int>(gridDim.x >> 1);
  // (The start overlaps the previous kernel's end: 128 inputs x 64 channels x 1024 samples, call after
  // call, 22.5 -> 20.3 us.)
  pdl_wait();

  if (warp < kEpiWarps) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpi));
    uint2* stage_rows = staging + warp * 32 * kOutPitch;
    const int quarter = warp & 3, colh = warp >> 2;
    const uint32_t tempty_even = smem_cluster(tempty, 0);
    const uint32_t sink_even = smem_cluster(sink + kSignalBytes * (kDecWarps + warp), 0);
    const int n_inputs = p.n_inputs;
    const uint32_t lanes = static_cast<uint32_t>(quarter * 32) << 16;
    // one block's accumulator is out: tell the MMA thread
    auto drained = [&](int buf) {
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
    };
    int g = 0;
    bool ok = true;
    for (int q = cl; ok && q < n_items; q += n_cl) {
      const Item it = item_of(p.nb, p.n_entries, q, rank);
      uint2* out_c = reinterpret_cast<uint2*>(p.out) + (int64_t)it.chan * p.n_pairs;
      const int row0 = it.R * kBlk + quarter * 32;  // first global row of this warp
      const int col0 = it.S * kBlk + colh * kHalf;  // first global column of this warp
      const bool live = it.has_row && row0 < n_inputs && col0 < n_inputs && (it.transposed || col0 <= row0 + 31);
      if (ADD && live) {
        // the sums this part adds to, pulled into L2 while its MMAs run: one row (or column) a lane
        const int i = it.transposed ? col0 + 2 * lane : row0 + lane;
        const int j = it.transposed ? row0 : col0;
        for (int k = 0; k < (it.transposed ? 2 : 1); ++k) {
          if (i + k < n_inputs) {
            const char* a = reinterpret_cast<const char*>(out_c + (int64_t)(i + k) * (i + k + 1) / 2 + j);
            const int bytes = 8 * (it.transposed ? 32 : min(kHalf, i - j + 1));
            for (int o = 0; o < bytes; o += 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(a + o));
          }
        }
      }
      int acc_re[kHalf], acc_im[kHalf];
#pragma unroll
      for (int k = 0; k < kHalf; ++k) acc_re[k] = acc_im[k] = 0;
      for (int blk = 0; blk < p.n_blocks; ++blk, ++g) {
        const int buf = g & 1;
        if (!mbar_wait_warp(&tfull[buf], (g >> 1) & 1, abort_flag, p.status, DEV_TIMEOUT_TMEM_FULL)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t taddr = tmem + lanes + buf * kAccCols + colh * 2 * kHalf;
#pragma unroll
        for (int k = 0; k < kHalf / 8; ++k) {
          uint32_t re[8], x[8];
          tmem_ld8(taddr + 8 * k, re);
          tmem_ld8(taddr + kHalf + 8 * k, x);
          tmem_ld_wait();
          if (!live) continue;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            acc_re[8 * k + j] += __float2int_rn(__uint_as_float(re[j]));
            acc_im[8 * k + j] -= __float2int_rn(__uint_as_float(x[j]));
          }
        }
        drained(buf);
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
        for (int k = 0; k < 8; ++k)
          v[k] = make_uint2(static_cast<uint32_t>(acc_re[ch + k]),
                            static_cast<uint32_t>(it.transposed ? -acc_im[ch + k] : acc_im[ch + k]));
        if (it.transposed)
          put_cols<false, ADD>(co, v);
        else
          put_rows<false, ADD>(ro, stage_rows, v, ch, lane);
      }
    }
  } else if (warp < kProducerWarp) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsDec));
    const int dw = warp - kDecWarp0, tid = dw * 32 + lane;
    const int grp = dw / kGroupWarps, gtid = tid - grp * kGroupWarps * 32;
    const uint32_t ready_even = smem_cluster(ready, 0);
    const uint32_t sink_even = smem_cluster(sink + kSignalBytes * dw, 0);
    const uint8_t* src0 = raw + gtid * 16;
    uint8_t* dst0 = ops + gtid * 16;
    constexpr int kStep = kGroupWarps * 32;  // 16-byte units from one of a lane's units to the next
    uint32_t gs = 0;  // the CTA's stages before the current item
    bool ok = true;
    for (int q = cl; ok && q < n_items; q += n_cl) {
      const Item it = item_of(p.nb, p.n_entries, q, rank);
      for (int tb = (grp ^ static_cast<int>(gs)) & 1; tb < p.n_kt; tb += kDecGroups) {
        const uint32_t st = gs + static_cast<uint32_t>(tb);
        const uint32_t r = st % kRaw, d = st % kOps;
        if (!mbar_wait_warp(&raw_full[r], (st / kRaw) & 1u, abort_flag, p.status, DEV_TIMEOUT_FULL)) {
          ok = false;
          break;
        }
        if (!mbar_wait_warp(&empty[d], ((st / kOps) & 1u) ^ 1u, abort_flag, p.status, DEV_TIMEOUT_EMPTY)) {
          ok = false;
          break;
        }
        const uint4* src = reinterpret_cast<const uint4*>(src0 + r * kRawStage);
        uint4* dst = reinterpret_cast<uint4*>(dst0 + d * kOpStage);
#pragma unroll
        for (int u = 0; u < kUnits; ++u, src += kStep, dst += kStep) {
          uint4 va0, va1, re, im;
          if (it.has_row) {
            va0 = src[0];
            va1 = src[kPlane / 16];
          }
          const uint4 vb = src[2 * kPlane / 16];
          if (it.has_row) {
            decode16(va0, re, im);
            dst[0] = re;
            dst[kPlane / 16] = im;
            decode16(va1, re, im);
            dst[2 * kPlane / 16] = re;
            dst[3 * kPlane / 16] = im;
          }
          decode16(vb, re, im);
          dst[4 * kPlane / 16] = re;
          dst[5 * kPlane / 16] = im;
          constexpr uint32_t sign = 0x80008000u;
          dst[6 * kPlane / 16] = make_uint4(re.x ^ sign, re.y ^ sign, re.z ^ sign, re.w ^ sign);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the operands, for the tensor core
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&raw_empty[r]);
          if (rank != 0)
            bulk_copy_to_cluster(sink_even, token, kSignalBytes, ready_even + 8u * d);
          else if (dw % kGroupWarps == 0)
            mbar_expect_tx(&ready[d], kGroupWarps * kSignalBytes);
          else
            mbar_arrive(&ready[d]);
        }
      }
      gs += static_cast<uint32_t>(p.n_kt);
    }
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsRest));
    if (warp == kProducerWarp) {
      if (lane == 0) {
        prefetch_tmap(&map);
        int s = 0;
        uint32_t ph = 0, filled = 0, fill_parity = 0;
        bool ok = true;
        for (int q = cl; ok && q < n_items; q += n_cl) {
          const Item it = item_of(p.nb, p.n_entries, q, rank);
          const int xa = it.R * kBlk, xb = it.S * kBlk + kHalf * static_cast<int>(rank);
          const uint32_t bytes = (it.has_row ? 3 : 1) * kPlane;
          for (int tb = 0, t = 0; tb < p.n_kt; ++tb, t += kRows) {
            if (!mbar_wait(&raw_empty[s], ph ^ 1u, abort_flag, p.status, DEV_TIMEOUT_EMPTY)) {
              ok = false;
              break;
            }
            uint8_t* st = raw + s * kRawStage;
            mbar_expect_tx(&raw_full[s], bytes);
            if (it.has_row) {
              tma_load_3d(st, &map, &raw_full[s], xa, it.chan, t);
              tma_load_3d(st + kPlane, &map, &raw_full[s], xa + kHalf, it.chan, t);
            }
            tma_load_3d(st + 2 * kPlane, &map, &raw_full[s], xb, it.chan, t);
            fill_parity = (fill_parity & ~(1u << s)) | (ph << s);
            filled |= 1u << s;
            if (++s == kRaw) {
              s = 0;
              ph ^= 1u;
            }
          }
        }
        // Let every copy this CTA issued land before the CTA can exit.
        volatile int never = 0;
        for (int k = 0; k < kRaw; ++k)
          if (filled & (1u << k)) mbar_wait(&raw_full[k], (fill_parity >> k) & 1u, &never, p.status, DEV_TIMEOUT_DRAIN);
      }
    } else if (warp == kMmaWarp && rank == 0 && lane == 0) {
      const uint32_t idesc = instr_desc(kTypeF16, true, 256, 256, false);
      int s = 0, g = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int q = cl; ok && q < n_items; q += n_cl) {
        for (int blk = 0; ok && blk < p.n_blocks; ++blk, ++g) {
          const int buf = g & 1;
          if (!mbar_wait(&tempty[buf], ((g >> 1) & 1) ^ 1, abort_flag, p.status, DEV_TIMEOUT_TMEM_EMPTY)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d = tmem + static_cast<uint32_t>(buf * kAccCols);
          const int kb0 = blk * kSpw, kb1 = min(p.n_kt, kb0 + kSpw);
          for (int kb = kb0; kb < kb1; ++kb) {
            if (!mbar_wait(&ready[s], ph, abort_flag, p.status, DEV_TIMEOUT_FULL)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t a = smem_u32(ops + s * kOpStage), b = a + kOffB;
            // the start address fields count 16 bytes; A's two half-tiles are two planes apart, B's
            // [re | im] and [im | -re] one plane
            const uint64_t da_r = smem_desc_sw128(a, 2 * kPlane, 8 * kRowB), da_i = da_r + (kPlane >> 4);
            const uint64_t db_r = smem_desc_sw128(b, kPlane, 8 * kRowB);
            const uint64_t db_i = db_r + (kPlane >> 4);
#pragma unroll
            for (int k = 0; k < kRows / kMmaK; ++k) {
              const uint64_t o = static_cast<uint64_t>((k * kMmaK * kRowB) >> 4);
              mma_pair<2>(d, da_r + o, db_r + o, idesc, (kb == kb0 && k == 0) ? 0u : 1u);
              mma_pair<2>(d, da_i + o, db_i + o, idesc, 1u);
            }
            mma_pair_commit_both(&empty[s]);
            if (++s == kOps) {
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
  }

  tc_fence_before();
  cluster_sync();  // no remote signal, sum or MMA of either CTA is still in flight
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
}

template <bool ADD>
cudaError_t launch_raw_pair(const CUtensorMap& map, const RParams& p, int num_sms, cudaStream_t stream) {
  auto kern = xcorr_tc_raw_pair_kernel<ADD>;
  static PerDevice<1> most;
  std::array<int, 1> clusters{};
  const cudaError_t e = most.get(&clusters, [kern](std::array<int, 1>& m) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
    if (e != cudaSuccess) return e;
    // pairs of SMs that can hold one CTA each at the same time
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(2 * 1024);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmem;
    e = cudaOccupancyMaxActiveClusters(&m[0], kern, &cfg);
    return e == cudaSuccess && m[0] < 1 ? cudaErrorLaunchOutOfResources : e;
  });
  if (e != cudaSuccess) return e;
  int n_cl = clusters[0] < num_sms / 2 ? clusters[0] : num_sms / 2;
  if (n_cl < 1) n_cl = 1;
  if (p.n_items < n_cl) n_cl = p.n_items;
  return launch_dependent(kern, 2 * n_cl, kThreads, kSmem, stream, map, p);
}

}  // namespace

int raw_pair_items(int n_tiles) { return pair_entries(n_tiles); }

bool raw_pair_takes(int pitch, const void* in) {
  return pitch % 8 == 0 && reinterpret_cast<uintptr_t>(in) % 16 == 0;
}

cudaError_t launch_xcorr_tc_raw_pair(const int8_t* in, int row_chans, int n_time, int n_chan, int n_inputs, int pitch,
                                     int2* out, bool accumulate, int* status, int num_sms, cudaStream_t stream) {
  if (!raw_pair_takes(pitch, in) || pitch < n_inputs || row_chans < n_chan || n_time < 1) return cudaErrorInvalidValue;
  RParams p{};
  p.n_inputs = n_inputs;
  p.nb = (n_inputs + kBlk - 1) / kBlk;
  p.n_entries = pair_entries(p.nb);
  const int64_t items = (int64_t)n_chan * p.n_entries;
  if (items > 0x7FFFFFFF) return cudaErrorInvalidValue;
  p.n_items = static_cast<int>(items);
  p.n_kt = (n_time + kRows - 1) / kRows;
  p.n_blocks = (p.n_kt + kSpw - 1) / kSpw;
  p.n_pairs = (int64_t)n_inputs * (n_inputs + 1) / 2;
  p.out = out;
  p.status = status;
  CUtensorMap map;
  if (!encode_raw_ci8_tmap(&map, in, pitch, n_chan, row_chans, n_time, kRows, nullptr)) return cudaErrorInvalidValue;
  return accumulate ? launch_raw_pair<true>(map, p, num_sms, stream) : launch_raw_pair<false>(map, p, num_sms, stream);
}

}  // namespace xc
