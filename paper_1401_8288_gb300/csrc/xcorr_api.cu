// xcorr_api.cu -- the C ABI (xcorr.h): plan validation, device memory owned
// by the plan, kernel selection, tuning and stream-ordered launches.
#include <cstdio>
#include <cstring>
#include <new>
#include <string>

#include "xcorr_internal.h"
#include "xcorr_nvtx.h"

namespace {

thread_local std::string g_last_error;

xcorr_status fail(xcorr_status st, const std::string& msg) {
  g_last_error = msg;
  return st;
}

xcorr_status cuda_fail(cudaError_t e, const char* what) {
  return fail(XCORR_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

int64_t n_pairs_of(int n_inputs) { return (int64_t)n_inputs * (n_inputs + 1) / 2; }

// Checks common to every call on a live plan.
xcorr_status plan_ok(xcorr_plan plan) {
  if (!plan) return fail(XCORR_ERR_INVALID_ARG, "plan is NULL");
  if (!plan->sticky && plan->status_host && *const_cast<volatile int*>(plan->status_host) != 0)
    plan->sticky = *plan->status_host;
  if (plan->sticky)
    return fail(XCORR_ERR_DEVICE, "a kernel of this plan reported failure code " + std::to_string(plan->sticky) +
                                      " (a bounded wait ran out); destroy the plan");
  cudaError_t e = cudaSetDevice(plan->device);
  if (e != cudaSuccess) return cuda_fail(e, "cudaSetDevice");
  return XCORR_OK;
}

void free_profile(xcorr_plan plan) {
  if (plan->prof_events) {
    for (int64_t k = 0; k < (int64_t)xc::kProfileEvents * plan->prof_cap; ++k)
      if (plan->prof_events[k]) cudaEventDestroy(plan->prof_events[k]);
    delete[] plan->prof_events;
  }
  delete[] plan->prof_ngroups;
  plan->prof_events = nullptr;
  plan->prof_ngroups = nullptr;
  plan->prof_cap = 0;
  plan->prof_count = 0;
}

void release(xcorr_plan plan) {
  free_profile(plan);
  if (plan->s_unpack) cudaStreamDestroy(plan->s_unpack);
  for (auto& sx : plan->s_x)
    if (sx) cudaStreamDestroy(sx);
  if (plan->ev_fork) cudaEventDestroy(plan->ev_fork);
  for (auto& ev : plan->ev_unpacked)
    if (ev) cudaEventDestroy(ev);
  for (auto& ev : plan->ev_x_done)
    if (ev) cudaEventDestroy(ev);
  plan->s_unpack = nullptr;
  plan->s_x[0] = plan->s_x[1] = nullptr;
  if (plan->s_down) cudaStreamDestroy(plan->s_down);
  plan->s_down = nullptr;
  for (auto* evs : {plan->ev_up, plan->ev_group_done})
    for (int g = 0; g < xc::kMaxGroups; ++g)
      if (evs[g]) cudaEventDestroy(evs[g]);
  if (plan->ev_down) cudaEventDestroy(plan->ev_down);
  plan->ev_down = nullptr;
  if (plan->host_stage) cudaFree(plan->host_stage);
  plan->host_stage = nullptr;
  if (plan->acc) cudaFree(plan->acc);
  if (plan->planes) cudaFree(plan->planes);
  if (plan->exps) cudaFree(plan->exps);
  plan->exps = nullptr;
  if (plan->ring_flags) cudaFree(plan->ring_flags);
  plan->ring_flags = nullptr;
  if (plan->status) cudaFree(plan->status);
  if (plan->status_host) cudaFreeHost(plan->status_host);
  plan->acc = nullptr;
  plan->planes = nullptr;
  plan->status = nullptr;
  plan->status_host = nullptr;
}

xcorr_status check_execute(xcorr_plan plan, const void* d_in, int n_time) {
  xcorr_status st = plan_ok(plan);
  if (st != XCORR_OK) return st;
  if (!d_in) return fail(XCORR_ERR_INVALID_ARG, "d_in is NULL");
  if (plan->cfg.fmt == XCORR_IN_CF32 && reinterpret_cast<uintptr_t>(d_in) % 4)
    return fail(XCORR_ERR_INVALID_ARG, "float input must be 4-byte aligned");
  if (n_time < 1 || n_time > plan->cfg.max_time_per_exec)
    return fail(XCORR_ERR_INVALID_ARG, "n_time must be in [1, max_time_per_exec]");
  if (plan->samples + n_time > plan->max_integration)
    return fail(XCORR_ERR_OVERFLOW, "the integration would exceed " + std::to_string(plan->max_integration) +
                                        " samples (the exact range of one dump); dump with reset first");
  return XCORR_OK;
}

int packed_channels(xcorr_plan plan) { return (plan->cfg.n_channels + plan->pack - 1) / plan->pack; }

// Channel groups of the tensor path: the tuned count, else enough tile pairs
// per group for about four waves of the persistent X kernel.
int tensor_groups(xcorr_plan plan) {
  int64_t g;
  if (plan->tune_groups > 0) {
    g = plan->tune_groups;
  } else {
    const int nb = (plan->n_inputs + 127) / 128;
    const int64_t items = (int64_t)packed_channels(plan) * nb * (nb + 1) / 2;
    g = items / (4LL * plan->num_sms);
  }
  if (g > xc::kMaxGroups) g = xc::kMaxGroups;
  if (g > packed_channels(plan)) g = packed_channels(plan);
  return g < 1 ? 1 : static_cast<int>(g);
}

// The 4-bit tensor path can unpack on chip: inputs a multiple of 16 and a
// 16-byte aligned pointer (the decoders read whole 16-sample chunks).
bool fused_applies(xcorr_plan plan, const void* d_in) {
  return plan->cfg.fmt == XCORR_IN_CI4 && !plan->tune_unfused && plan->n_inputs % 16 == 0 &&
         reinterpret_cast<uintptr_t>(d_in) % 16 == 0;
}

// int8 input that is decoded on chip: one launch, no planes.
bool raw_ci8_applies(xcorr_plan plan, const void* d_in) {
  return plan->cfg.fmt == XCORR_IN_CI8 && plan->engine == XCORR_ENGINE_TENSOR && xc::raw_pair_takes(plan->n_inputs, d_in);
}

// Whether int8 input is decoded on chip (xcorr_tc_raw_pair.cu) or goes through planes in memory
// (xcorr_unpack.cu and xcorr_tc.cu), by the time of an execute: a set-up, rounds of the persistent kernel
// (so many us, and so many a sample), the MB that the unpack or the padding copy moves, and the MB of
// visibilities.  On chip a CTA pair takes an entry of a channel, and with one tile its second CTA has no
// rows; from planes every SM takes a tile and a step is shorter, but the planes are written and read.
// The figures are least squares over 1500 sizes (2 to 1024 inputs, 1 to 512 channels, 32 to 4096 samples;
// within 17 % of the times of all but 4 % of them); the margin of 5 % goes to the planes, whose time varies
// less.  us, planes / on chip: 16 inputs x 152 channels x 4096 samples 58 / 103, 64 x 512 x 1024 90 / 97, 128 x
// 64 x 1024 29 / 23, 128 x 4 x 4096 51 / 58, 136 x 48 x 256 17 / 21, 256 x 152 x 4096 310 / 214, 62 x 304 x 1024
// 110 / 68.
bool ci8_from_planes(int n_inputs, int n_chan, int n_time, int num_sms, bool aligned) {
  const int nb = (n_inputs + 127) / 128;
  const double t = n_time, mb = 1e-6 * n_chan * t, out = 4e-6 * n_chan * n_inputs * (n_inputs + 1.0);
  const int64_t tiles = (int64_t)n_chan * nb * (nb + 1) / 2, entries = (int64_t)n_chan * xc::raw_pair_items(nb);
  const double rt = static_cast<double>((tiles + num_sms - 1) / num_sms);
  const double re = static_cast<double>((entries + num_sms / 2 - 1) / (num_sms / 2));
  const int padded = (n_inputs + 15) / 16 * 16;
  const double planes = aligned ? 7.9 + rt * (3.3 + 0.0087 * t) + 0.183 * 6 * padded * mb + 0.10 * out
                                : 7.7 + rt * (3.8 + 0.0092 * t) + 0.632 * 6 * n_inputs * mb + 0.13 * out;  // by elements
  const double chip = aligned ? 8.7 + re * (2.3 + 0.0106 * t) + 0.19 * out
                              : 9.8 + re * (2.3 + 0.0106 * t) + 0.116 * 4 * n_inputs * mb + 0.27 * out;  // with the copy
  return planes < 1.05 * chip;
}

// Whether two or more tiles a side of float input, or of 4-bit input that is not decoded on chip, go
// through planes in memory rather than through the ring (xcorr_tc_pair.cu), by the same kind of model.  The
// ring's single launch starts on clusters one at a time and unpacks on the CTAs that it runs, so it wins
// where the rounds are long and many: float, us, planes / ring (1800 sizes; the route so chosen costs 30 % less
// than the ring alone on average): 256 inputs x 16 channels x 256 samples 27 / 44, 256 x 16 x 1024 64 / 106, 512 x 64
// x 1024 439 / 414, 192 x 64 x 4096 670 / 591, 130 x 100 x 10000 2530 / 2010, 512 x 256 x 4096 7200 / 5800.
// 4-bit: where rows are whole 16-byte units the planes take less time at 158 of 170 sizes (256 x 200 x 1024
// 64 / 124); off them they are unpacked byte by byte (338 x 200 x 4096 1226 / 506, 130 x 32 x 1024 33 / 36).
bool planes_beat_ring(int fmt, int n_inputs, int n_chan, int n_time, int num_sms) {
  const int nb = (n_inputs + 127) / 128;
  const double t = n_time, mb = 1e-6 * n_chan * t, out = 4e-6 * n_chan * n_inputs * (n_inputs + 1.0);
  const int64_t tiles = (int64_t)n_chan * nb * (nb + 1) / 2, entries = (int64_t)n_chan * xc::raw_pair_items(nb);
  const double rt = static_cast<double>((tiles + num_sms - 1) / num_sms);
  const double re = static_cast<double>((entries + num_sms / 2 - 1) / (num_sms / 2));
  if (fmt == XCORR_IN_CI4) {
    if (n_inputs % 16 == 0) return true;
    return 7.6 + rt * (4.6 + 0.0056 * t) + 1.196 * 3 * n_inputs * mb + 0.064 * out < 17.8 + re * (3.9 + 0.014 * t) + 0.033 * out;
  }
  const int blocks = 6 * ((n_time + xc::kTcWindowBF16 - 1) / xc::kTcWindowBF16);  // drained one by one, shared by a cluster
  const int split = xc::tc_float_split(tiles, blocks, num_sms);
  const double steps = 6 * t * ((blocks + split - 1) / split) / blocks;
  const int units = (n_inputs + 15) / 16;  // of the unpack, which takes longer over an odd number of them
  const double planes = 11 + rt * (6.2 + 0.0091 * steps) + (units % 2 ? 0.394 : 0.194) * 20 * 16 * units * mb + 0.006 * out;
  const double ring = 20 + re * (3.1 + 0.01165 * 6 * t) + 0.054 * 12 * 128 * nb * mb + 0.27 * out;
  return 1.03 * planes < ring;
}

// An execute of a plan that has the planes still takes the faster route for its own samples and address.
bool staged_execute(xcorr_plan plan, const void* d_in, int n_time) {
  return plan->staged_ci8 && ci8_from_planes(plan->n_inputs, plan->cfg.n_channels, n_time, plan->num_sms,
                                             xc::raw_pair_takes(plan->n_inputs, d_in));
}

// Input that would be decoded on chip but for its rows' or its address's alignment is copied piece by
// piece to padded rows in the plan's planes memory and correlated from there (xcorr_repitch.cu).
// A piece: `nc` channels x `nt` samples.
struct Pieces {
  int pitch = 0;  // inputs from one row to the next; 0: does not apply
  int nc = 0, nt = 0;
};
// At most a GB at a time.  A piece that stays in the L2 saves less than it costs in waves of the X
// kernel that are not full and in launches (510 inputs x 400 channels x 2048 4-bit samples with pieces
// of 64 / 96 / 256 MB / 1 GB: 605 / 556 / 522 / 510 us; 510 x 300 x 2048 int8: 807 / 771 / 740 / 725).
constexpr size_t kPieceBytes = size_t(1) << 30;
// (338 inputs x 20 channels x 1,500,000 4-bit samples in pieces of all samples of one channel or two 96 ms, of a
// wave's channels 13; 512 x 97 x 100,000 at an odd address 49 and 7.6; int8 512 x 40 x 40,000 at one 19 and 2.4.)
constexpr size_t kPieceSamples = 1024;
constexpr size_t kOddAddressPieceBytes = size_t(64) << 20;  // kept by plans that need it at odd addresses only
size_t padded_row_bytes(int fmt, int n_inputs) {
  return static_cast<size_t>((n_inputs * (fmt == XCORR_IN_CI4 ? 1 : 2) + 15) / 16) * 16;
}
Pieces repitch_pieces(xcorr_plan plan, int n_time) {
  Pieces r;
  const int fmt = plan->cfg.fmt;
  if (plan->engine != XCORR_ENGINE_TENSOR || fmt == XCORR_IN_CF32 || (fmt == XCORR_IN_CI4 && plan->tune_unfused))
    return r;
  const int C = plan->cfg.n_channels;
  const size_t row = padded_row_bytes(fmt, plan->n_inputs);
  const size_t room = plan->planes_bytes < kPieceBytes ? plan->planes_bytes : kPieceBytes;
  const size_t rows = room / row;  // of one channel and sample each
  const int nb = (plan->n_inputs + 127) / 128;
  const int per_chan = fmt == XCORR_IN_CI4 ? nb * (nb + 1) / 2 : xc::raw_pair_items(nb);
  const int wave = fmt == XCORR_IN_CI4 ? plan->num_sms : plan->num_sms / 2;
  const int full = wave / per_chan < 1 ? 1 : wave / per_chan < C ? wave / per_chan : C;  // channels of a full wave
  r.nt = n_time;
  if (rows / full < static_cast<size_t>(n_time)) {
    // A long integration: stages of samples at a time rather than channels that leave SMs idle.  Every
    // piece of them after the first adds into the visibilities, so a piece has kPieceSamples of them
    // where the memory holds so many (4-bit: the fused kernel's own blocks, which add anyway).
    const size_t fits = rows / full, block = fits >= xc::kFusedWindowCI4 && fmt == XCORR_IN_CI4 ? xc::kFusedWindowCI4 : 128;
    size_t nt = fits < kPieceSamples ? kPieceSamples : fits;
    if (nt > rows) nt = rows;
    nt = nt / block * block;
    if (nt == 0 && rows < static_cast<size_t>(n_time)) return r;  // (4-bit under a tight memory limit: the ring of planes)
    if (nt > 0 && nt < static_cast<size_t>(n_time)) r.nt = static_cast<int>(nt);
  }
  r.nc = rows / r.nt < static_cast<size_t>(C) ? static_cast<int>(rows / r.nt) : C;
  if (r.nc < C) {  // several pieces: whole waves of the X kernel where a piece holds one
    const int whole = static_cast<int>(static_cast<int64_t>(r.nc) * per_chan / wave * wave / per_chan);
    if (whole > 0) r.nc = whole;
  }
  r.pitch = static_cast<int>(fmt == XCORR_IN_CI4 ? row : row / 2);
  return r;
}

// The tensor-memory-A kernel's launch shape for a stage variant; the other kernels' variants mean its
// default here.
int padded_shape(int v) {
  return v == xc::kSmallFusedVariant ? 3 : v >= 4 && v <= 6 ? v - 4 : xc::kDefaultFusedVariant - 4;
}

// Correlate nch channels through padded rows: d_in at the first of them, in rows of the plan's channels,
// target at its visibilities.
cudaError_t run_repitched(xcorr_plan plan, const Pieces& r, const void* d_in, int nch, int n_time, int2* target,
                          bool fresh, cudaStream_t s) {
  const int C = plan->cfg.n_channels, N = plan->n_inputs;
  const bool ci4 = plan->cfg.fmt == XCORR_IN_CI4;
  const size_t row = static_cast<size_t>(N) * (ci4 ? 1 : 2);  // one channel of one sample
  const uint8_t* in = static_cast<const uint8_t*>(d_in);
  const uint8_t* end = in + row * (static_cast<size_t>(C) * (n_time - 1) + nch);
  const int shape = padded_shape(plan->tune_variant);
  for (int t0 = 0; t0 < n_time; t0 += r.nt) {
    const int nt = n_time - t0 < r.nt ? n_time - t0 : r.nt;
    for (int c0 = 0; c0 < nch; c0 += r.nc) {
      const int nc = nch - c0 < r.nc ? nch - c0 : r.nc;
      cudaError_t e = xc::launch_repitch(in + (static_cast<size_t>(t0) * C + c0) * row, end, plan->planes,
                                         static_cast<int>(row), C, nc, nt, plan->num_sms, s);
      if (e != cudaSuccess) return e;
      int2* out = target + static_cast<int64_t>(c0) * plan->n_pairs;
      const bool add = !fresh || t0 > 0;
      e = ci4 ? xc::launch_xcorr_tc_fused_ta_ci4(static_cast<const uint8_t*>(plan->planes), nc, shape, nt, nc, N, r.pitch,
                                                 out, add, plan->status, plan->num_sms, s)
              : xc::launch_xcorr_tc_raw_pair(static_cast<const int8_t*>(plan->planes), nc, nt, nc, N, r.pitch, out, add,
                                             plan->status, plan->num_sms, s);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}

// The kernels that run_repitched launches for a storing execute of the plan's channels.
int repitched_launches(xcorr_plan plan, const Pieces& r, int n_time) {
  const int C = plan->cfg.n_channels, shape = padded_shape(plan->tune_variant);
  const auto piece = [&](int nt, int nc, bool first) {
    return 1 + (plan->cfg.fmt != XCORR_IN_CI4 ? 1
                : first ? xc::fused_ta_launches(shape, nt, nc, plan->n_inputs, r.pitch, plan->num_sms)
                        : (nt + xc::kFusedWindowCI4 - 1) / xc::kFusedWindowCI4);
  };
  const auto pieces = [&](int nt, bool first) {
    return nt == 0 ? 0 : C / r.nc * piece(nt, r.nc, first) + (C % r.nc ? piece(nt, C % r.nc, first) : 0);
  };
  return pieces(r.nt, true) + (n_time / r.nt - 1) * pieces(r.nt, false) + pieces(n_time % r.nt, false);
}

// Unpack channels [c0, c0 + nc) of the input into the plan's planes.
cudaError_t unpack_group(xcorr_plan plan, const void* d_in, int n_time, int c0, int nc, cudaStream_t s) {
  const int C = plan->cfg.n_channels, N = plan->n_inputs, T = plan->cfg.max_time_per_exec;
  switch (plan->cfg.fmt) {
    case XCORR_IN_CI4:
      return xc::launch_unpack_ci4_e4m3_channels(static_cast<const uint8_t*>(d_in), static_cast<uint8_t*>(plan->planes),
                                                 n_time, C, c0, nc, N, plan->ni_pad, T, plan->num_sms, s);
    case XCORR_IN_CI8:
      return xc::launch_unpack_ci8_bf16(static_cast<const int8_t*>(d_in), static_cast<uint16_t*>(plan->planes), n_time,
                                        C, c0, nc, N, plan->ni_pad, T, plan->num_sms, s);
    default:
      return xc::launch_unpack_cf32_digits(static_cast<const float*>(d_in), static_cast<uint16_t*>(plan->planes),
                                           plan->exps, n_time, C, c0, nc, N, plan->pack, plan->ni_pad, T, plan->window_samples,
                                           plan->exp_windows, s);
  }
}

int even_groups(int C, int n, int* edge) {
  const int most = C < xc::kMaxGroups ? C : xc::kMaxGroups, G = n < most ? n : most;
  for (int g = 0; g <= G; ++g) edge[g] = static_cast<int>(static_cast<int64_t>(C) * g / G);
  return G;
}

// The channel groups of a host-to-host execute that moves `bytes` in and out.  A column of at least a
// quarter of a sample's channels comes up at the link's rate beside a copy down (256 MB each way, rows of
// 16 to 512 KB: 1.58-1.61 ms); an eighth does not (2.1 ms).  Nothing comes down during the first group's
// way up, so that one is narrow; its head start no longer matters where the copies take milliseconds.  A
// group costs about 10 us.  (512 inputs x 128 channels x 1024 samples, 67 MB up, 134 MB down: one group
// 1140 us, four equal ones 897, these 853; the copies alone 749.  1024 samples of 256 inputs x 64 channels,
// 33 MB in all: 227, 182, 183.  524 MB each way: four equal ones 3.88 ms, these 4.39.)
int host_groups(int C, size_t bytes, int* edge) {
  const size_t mb = bytes >> 20;
  if (mb < 24 || C < 8) return even_groups(C, mb < 8 ? 1 : 2, edge);
  if (mb >= 512) return even_groups(C, 4, edge);
  const int sixteenths[5] = {0, 2, 6, 11, 16};
  for (int g = 0; g <= 4; ++g) edge[g] = static_cast<int>(static_cast<int64_t>(C) * sixteenths[g] / 16);
  return 4;
}

// Host memory that is not pinned.
bool pageable(const void* p) {
  cudaPointerAttributes a{};
  return cudaPointerGetAttributes(&a, p) == cudaSuccess && a.type == cudaMemoryTypeUnregistered;
}

// The most groups of an int8 host execute.  However few its channels, a group's launch takes the time of one
// channel's samples (0.0106 us each; padded rows share their memory, so one group after the other; else two
// at a time): together no more than the way up at 200 GB/s.  (18 inputs x 64 channels x 14,563 samples: one
// group 388 us, two 486, four 780.)
int ci8_host_groups(size_t bytes, int n_time, bool two_streams) {
  const double n = (two_streams ? 2 : 1) * (5e-6 * bytes) / (0.0106 * n_time);
  return n < 1 ? 1 : n > xc::kMaxGroups ? xc::kMaxGroups : static_cast<int>(n);
}

// Correlate n_time samples into target (the plan's accumulator, or the
// caller's buffer for a fused dump).  target_fresh: store instead of add.
xcorr_status run_execute(xcorr_plan plan, const void* d_in, int n_time, void* target, bool target_fresh,
                         cudaStream_t s) {
  const int C = plan->cfg.n_channels, N = plan->n_inputs;
  const bool staged_ci8 = staged_execute(plan, d_in, n_time);
  cudaError_t e;
  cudaEvent_t* ev = nullptr;
  if (plan->prof_cap) {
    const int64_t slot = plan->prof_count % plan->prof_cap;
    ev = plan->prof_events + xc::kProfileEvents * slot;
    if ((e = cudaEventRecord(ev[0], s)) != cudaSuccess) return cuda_fail(e, "profile event");
  }
  if (plan->engine == XCORR_ENGINE_TENSOR && fused_applies(plan, d_in)) {
    // 4-bit input with the unpack on chip: one launch per exact block, on the caller's stream
    if (ev && ((e = cudaEventRecord(ev[1], s)) != cudaSuccess || (e = cudaEventRecord(ev[2], s)) != cudaSuccess))
      return cuda_fail(e, "profile event");
    e = xc::launch_xcorr_tc_fused_ci4(static_cast<const uint8_t*>(d_in), C, plan->tune_variant, n_time, C, N,
                                      static_cast<int2*>(target), !target_fresh, plan->status, plan->num_sms, s);
    if (e != cudaSuccess) return cuda_fail(e, "fused X kernel launch");
    if (ev && (e = cudaEventRecord(ev[3], s)) != cudaSuccess) return cuda_fail(e, "profile event");
    if (ev) plan->prof_ngroups[plan->prof_count % plan->prof_cap] = 1;
  } else if (!staged_ci8 && raw_ci8_applies(plan, d_in)) {
    // int8 input decoded on chip: one launch on the caller's stream
    if (ev && ((e = cudaEventRecord(ev[1], s)) != cudaSuccess || (e = cudaEventRecord(ev[2], s)) != cudaSuccess))
      return cuda_fail(e, "profile event");
    e = xc::launch_xcorr_tc_raw_pair(static_cast<const int8_t*>(d_in), C, n_time, C, N, N, static_cast<int2*>(target),
                                     !target_fresh, plan->status, plan->num_sms, s);
    if (e != cudaSuccess) return cuda_fail(e, "CTA-pair X kernel launch");
    if (ev && (e = cudaEventRecord(ev[3], s)) != cudaSuccess) return cuda_fail(e, "profile event");
    if (ev) plan->prof_ngroups[plan->prof_count % plan->prof_cap] = 1;
  } else if (const Pieces pieces = staged_ci8 ? Pieces{} : repitch_pieces(plan, n_time); pieces.pitch) {
    // the same kernels over padded rows, piece by piece on the caller's stream
    if (ev && ((e = cudaEventRecord(ev[1], s)) != cudaSuccess || (e = cudaEventRecord(ev[2], s)) != cudaSuccess))
      return cuda_fail(e, "profile event");
    if ((e = run_repitched(plan, pieces, d_in, C, n_time, static_cast<int2*>(target), target_fresh, s)) != cudaSuccess)
      return cuda_fail(e, "padded rows: copy or X kernel launch");
    if (ev && (e = cudaEventRecord(ev[3], s)) != cudaSuccess) return cuda_fail(e, "profile event");
    if (ev) plan->prof_ngroups[plan->prof_count % plan->prof_cap] = 1;
  } else if (plan->pair) {
    // one launch on the caller's stream: unpack warps feed the CTA pairs through the ring
    if (ev && ((e = cudaEventRecord(ev[1], s)) != cudaSuccess || (e = cudaEventRecord(ev[2], s)) != cudaSuccess))
      return cuda_fail(e, "profile event");
    xc::PairLaunch L;
    L.fmt = plan->cfg.fmt;
    L.in = d_in;
    L.n_time = n_time;
    L.n_chan = C;
    L.n_inputs = N;
    L.accumulate = !target_fresh;
    L.out = target;
    L.status = plan->status;
    L.ring = &plan->ring;
    L.ring_mem = plan->planes;
    L.flags = plan->ring_flags;
    L.exps = plan->exps;
    L.exp_windows = plan->exp_windows;
    L.exp_pitch = plan->ni_pad;
    if ((e = xc::launch_xcorr_tc_pair(L, s)) != cudaSuccess) return cuda_fail(e, "CTA-pair X kernel launch");
    if (ev && (e = cudaEventRecord(ev[3], s)) != cudaSuccess) return cuda_fail(e, "profile event");
    if (ev) plan->prof_ngroups[plan->prof_count % plan->prof_cap] = 1;
  } else if (plan->engine == XCORR_ENGINE_TENSOR) {
    const int variant = plan->pack > 1 ? 0 : xc::planes_variant(plan->tune_variant);
    const int row_inputs = plan->pack > 1 ? plan->ni_pad : N, Cp = packed_channels(plan);
    if (plan->tmap_ntime != n_time || plan->tmap_variant != variant) {
      std::string err;
      if (!xc::encode_plane_tmap(&plan->tmap, plan->planes, plan->elem_bytes, row_inputs, plan->ni_pad, n_time,
                                 plan->cfg.max_time_per_exec, Cp * plan->planes_per_chan,
                                 xc::tc_stage_samples(plan->elem_bytes, variant), &err))
        return fail(XCORR_ERR_CUDA, err);
      plan->tmap_ntime = n_time;
      plan->tmap_variant = variant;
    }
    xc::TcLaunch L;
    L.elem_bytes = plan->elem_bytes;
    L.variant = variant;
    L.float_out = plan->cfg.fmt == XCORR_IN_CF32;
    L.n_time = n_time;
    L.n_inputs = row_inputs;
    L.pack = plan->pack;
    L.true_inputs = N;
    L.true_chans = C;
    L.planes_per_chan = plan->planes_per_chan;
    if (plan->cfg.fmt == XCORR_IN_CF32) {
      // the six digit products d_p d_q with p + q <= 2
      L.exps = plan->exps;
      L.exp_windows = plan->exp_windows;
      L.ni_pad = plan->ni_pad;
      const int pp[6] = {0, 0, 1, 0, 2, 1}, pq[6] = {0, 1, 0, 2, 0, 1};
      L.n_pairs_k = 6;
      for (int k = 0; k < 6; ++k) {
        L.pair_p[k] = pp[k];
        L.pair_q[k] = pq[k];
      }
    }
    L.window_samples = plan->window_samples;
    L.accumulate = !target_fresh;
    L.out = target;
    L.status = plan->status;
    L.num_sms = plan->num_sms;
    const int G = tensor_groups(plan);
    const int per = (Cp + G - 1) / G;
    const int nxs = plan->tune_x_streams == 1 ? 1 : 2;
    // several groups: the internal streams fork from s after everything queued on it so far (one
    // group's two launches follow one another on s itself)
    const bool forked = per < Cp;
    cudaStream_t su = forked ? plan->s_unpack : s;
    if (forked) {
      if ((e = cudaEventRecord(plan->ev_fork, s)) != cudaSuccess) return cuda_fail(e, "fork event");
      if ((e = cudaStreamWaitEvent(plan->s_unpack, plan->ev_fork, 0)) != cudaSuccess ||
          (e = cudaStreamWaitEvent(plan->s_x[0], plan->ev_fork, 0)) != cudaSuccess ||
          (e = cudaStreamWaitEvent(plan->s_x[1], plan->ev_fork, 0)) != cudaSuccess)
        return cuda_fail(e, "fork wait");
    }
    int used = 0;
    for (int g = 0, c0 = 0; c0 < Cp; ++g, c0 += per) {
      const int nc = (Cp - c0 < per) ? Cp - c0 : per;
      const int first = c0 * plan->pack, last = (c0 + nc) * plan->pack < C ? (c0 + nc) * plan->pack : C;
      if ((e = unpack_group(plan, d_in, n_time, first, last - first, su)) != cudaSuccess)
        return cuda_fail(e, "unpack launch");
      cudaStream_t sx = forked ? plan->s_x[g % nxs] : s;
      if (forked) {
        if ((e = cudaEventRecord(plan->ev_unpacked[g], su)) != cudaSuccess) return cuda_fail(e, "event");
        if ((e = cudaStreamWaitEvent(sx, plan->ev_unpacked[g], 0)) != cudaSuccess) return cuda_fail(e, "wait");
      }
      if (ev && !forked && (e = cudaEventRecord(ev[1], s)) != cudaSuccess) return cuda_fail(e, "profile event");
      if (ev && (e = cudaEventRecord(ev[2 + 2 * g], sx)) != cudaSuccess) return cuda_fail(e, "profile event");
      L.chan0 = c0;
      L.n_chan = nc;
      if ((e = xc::launch_xcorr_tc(&plan->tmap, L, sx)) != cudaSuccess)
        return cuda_fail(e, "tensor-core X kernel launch");
      if (ev && (e = cudaEventRecord(ev[3 + 2 * g], sx)) != cudaSuccess) return cuda_fail(e, "profile event");
      used = g + 1;
    }
    if (ev && forked && (e = cudaEventRecord(ev[1], su)) != cudaSuccess) return cuda_fail(e, "profile event");
    // join: s continues after both X streams (which waited for every unpack)
    for (int k = 0; forked && k < 2; ++k) {
      if ((e = cudaEventRecord(plan->ev_x_done[k], plan->s_x[k])) != cudaSuccess ||
          (e = cudaStreamWaitEvent(s, plan->ev_x_done[k], 0)) != cudaSuccess)
        return cuda_fail(e, "join");
    }
    if (ev) plan->prof_ngroups[plan->prof_count % plan->prof_cap] = used;
  } else {
    const int ks = xc::cuda_core_ksplit(n_time, C, N, plan->num_sms);
    int mode = target_fresh ? xc::MODE_STORE : xc::MODE_ADD;
    if (ks > 1) {
      if (target_fresh) {
        e = cudaMemsetAsync(target, 0, (size_t)C * plan->n_pairs * sizeof(int2), s);
        if (e != cudaSuccess) return cuda_fail(e, "accumulator clear");
      }
      mode = xc::MODE_ATOMIC;
    }
    if (ev && ((e = cudaEventRecord(ev[1], s)) != cudaSuccess || (e = cudaEventRecord(ev[2], s)) != cudaSuccess))
      return cuda_fail(e, "profile event");
    e = xc::launch_xcorr_cuda_core(plan->cfg.fmt, d_in, n_time, C, N, static_cast<int2*>(target), mode, ks, s);
    if (e != cudaSuccess) return cuda_fail(e, "CUDA-core X kernel launch");
    if (ev && (e = cudaEventRecord(ev[3], s)) != cudaSuccess) return cuda_fail(e, "profile event");
    if (ev) plan->prof_ngroups[plan->prof_count % plan->prof_cap] = 1;
  }
  if (ev) ++plan->prof_count;
  return XCORR_OK;
}

}  // namespace

namespace xc {
xcorr_status set_error(xcorr_status st, const std::string& msg) { return fail(st, msg); }
xcorr_status plan_check(xcorr_plan plan) { return plan_ok(plan); }
xcorr_status execute_into(xcorr_plan plan, const void* d_in, int n_time, void* target, bool target_fresh,
                          cudaStream_t s) {
  return run_execute(plan, d_in, n_time, target, target_fresh, s);
}
xcorr_status read_device_status(xcorr_plan plan) {
  int code = 0;
  cudaError_t e = cudaMemcpy(&code, plan->status, sizeof(int), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "status read");
  if (code) plan->sticky = code;
  return plan_ok(plan);
}
}  // namespace xc

extern "C" {

const char* xcorr_last_error(void) { return g_last_error.c_str(); }

xcorr_status xcorr_plan_create(xcorr_plan* out, const xcorr_config* cfg) {
  if (!out) return fail(XCORR_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  if (!cfg) return fail(XCORR_ERR_INVALID_ARG, "cfg is NULL");
  const xcorr_config c = *cfg;
  if (c.n_pols != 2) return fail(XCORR_ERR_INVALID_ARG, "n_pols must be 2");
  if (c.n_stations < 1 || c.n_stations > (1 << 20))
    return fail(XCORR_ERR_INVALID_ARG, "n_stations must be in [1, 2^20]");
  if (c.n_channels < 1) return fail(XCORR_ERR_INVALID_ARG, "n_channels must be >= 1");
  if (c.max_time_per_exec < 1) return fail(XCORR_ERR_INVALID_ARG, "max_time_per_exec must be >= 1");
  if (c.fmt != XCORR_IN_CI4 && c.fmt != XCORR_IN_CI8 && c.fmt != XCORR_IN_CF32)
    return fail(XCORR_ERR_INVALID_ARG, "unknown input format");
  if (c.engine != XCORR_ENGINE_AUTO && c.engine != XCORR_ENGINE_TENSOR && c.engine != XCORR_ENGINE_CUDA_CORE)
    return fail(XCORR_ERR_INVALID_ARG, "unknown engine");

  // AUTO: the engine the per-call device times favour (graph-replayed execute_dump; 4-bit input
  // over inputs 2-256, channels 16-256, K 256-2048; int8 over inputs 2-256, channels 16-64,
  // K 256-1024).  The CUDA-core kernel wins only at most 16 channels: for 4-bit input below 16
  // inputs (the tensor path then pads the rows first: two launches), for int8 input up to 64 inputs;
  // the tensor cores everywhere else.
  const int cc_inputs = c.fmt == XCORR_IN_CI4 ? 15 : c.fmt == XCORR_IN_CI8 ? 64 : 0;
  const int engine = c.engine != XCORR_ENGINE_AUTO ? c.engine
                     : (c.n_stations <= cc_inputs / 2 && c.n_channels <= 16) ? XCORR_ENGINE_CUDA_CORE
                                                                            : XCORR_ENGINE_TENSOR;
  if (engine == XCORR_ENGINE_CUDA_CORE && c.fmt == XCORR_IN_CF32)
    return fail(XCORR_ERR_UNSUPPORTED, "the CUDA-core engine takes integer input only");

  const int64_t max_int = c.fmt == XCORR_IN_CI4   ? xc::kMaxIntegrationCI4
                          : c.fmt == XCORR_IN_CI8 ? xc::kMaxIntegrationCI8
                                                  : xc::kMaxIntegrationCF32;
  if (c.max_time_per_exec > max_int)
    return fail(XCORR_ERR_OVERFLOW, "max_time_per_exec exceeds the range of one integration, " +
                                        std::to_string(max_int) + " samples");

  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  cudaDeviceProp prop;
  e = cudaGetDeviceProperties(&prop, dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDeviceProperties");
  if (prop.major != 10 || prop.minor != 3)
    return fail(XCORR_ERR_UNSUPPORTED, std::string("this library is built for sm_103a (GB300); device is ") +
                                           prop.name + " sm_" + std::to_string(prop.major * 10 + prop.minor));

  const int n_inputs = 2 * c.n_stations;
  int ni_pad = (n_inputs + 15) / 16 * 16;
  const int64_t n_pairs = n_pairs_of(n_inputs);
  const int elem_bytes = c.fmt == XCORR_IN_CI4 ? 1 : 2;
  const int ppc = c.fmt == XCORR_IN_CF32 ? 6 : 2;
  const size_t acc_bytes = (size_t)c.n_channels * (size_t)n_pairs * 8;
  // Float input of at most 64 inputs: channels side by side in the 128 rows of a tile, which costs the same
  // however few are used, as many as shorten the longest CTA's work; none past the last channel under a
  // memory limit.  (16 inputs x 64 channels x 1024 samples: 57 us with a tile per channel, 28 so; 40 x
  // 500 x 1024: 589, 290.  Always as many as fit: 16 x 16 x 256 17.3 -> 20.0, 50 x 33 x 700 32.6 -> 41.8.)
  int pack = 1;
  if (engine == XCORR_ENGINE_TENSOR && c.fmt == XCORR_IN_CF32 && n_inputs <= 64) {
    const int blocks = 6 * ((c.max_time_per_exec + xc::kTcWindowBF16 - 1) / xc::kTcWindowBF16);
    int64_t best = 0;
    for (int k = 1; k <= 128 / ni_pad && k <= c.n_channels; k *= 2) {  // the blocks that the busiest CTA drains
      const int64_t tiles = (c.n_channels + k - 1) / k, split = xc::tc_float_split(tiles, blocks, prop.multiProcessorCount);
      const int64_t cost = (tiles + prop.multiProcessorCount - 1) / prop.multiProcessorCount * ((blocks + split - 1) / split);
      if (k > 1 && (cost >= best || (c.n_channels % k && c.hbm_budget_bytes))) continue;
      best = cost;
      pack = k;
    }
  }
  const int plane_chans = (c.n_channels + pack - 1) / pack;
  ni_pad *= pack;
  const int exp_windows = (c.max_time_per_exec + xc::kTcWindowBF16 - 1) / xc::kTcWindowBF16;
  const size_t exps_bytes = (engine == XCORR_ENGINE_TENSOR && c.fmt == XCORR_IN_CF32)
                                ? (size_t)plane_chans * exp_windows * ni_pad * 2
                                : 0;
  const size_t all_planes = (size_t)plane_chans * ppc * (size_t)c.max_time_per_exec * ni_pad * elem_bytes;
  // Where the operands come from.  int8: decoded on chip, or planes of all channels.  Two or more 128-input
  // tiles a side of the others: a small ring of planes, or all of them; one tile: all of them.  (4-bit
  // input that is decoded on chip never touches its planes: they take no more memory than padded rows
  // may.)  All planes take at most the caller's limit, or a quarter of the memory where there is none.
  const bool tensor = engine == XCORR_ENGINE_TENSOR;
  const bool planes_fit = acc_bytes + all_planes + exps_bytes + 256 <= (c.hbm_budget_bytes ? c.hbm_budget_bytes : prop.totalGlobalMem / 4);
  const bool staged_ci8 = tensor && c.fmt == XCORR_IN_CI8 && planes_fit &&
                          ci8_from_planes(n_inputs, c.n_channels, c.max_time_per_exec, prop.multiProcessorCount, n_inputs % 8 == 0);
  const bool decoded_ci8 = tensor && c.fmt == XCORR_IN_CI8 && !staged_ci8;
  bool pair = tensor && c.fmt != XCORR_IN_CI8 && (n_inputs + 127) / 128 >= xc::kTcPairMinTiles &&
                    !(planes_fit && (c.fmt == XCORR_IN_CF32 || all_planes <= kPieceBytes) &&
                      planes_beat_ring(c.fmt, n_inputs, c.n_channels, c.max_time_per_exec, prop.multiProcessorCount));
  size_t planes_bytes = tensor && !decoded_ci8 && !pair ? all_planes : 0;
  xc::PairRing ring;
  const size_t other = acc_bytes + exps_bytes + 256;
  const size_t room = c.hbm_budget_bytes > other ? c.hbm_budget_bytes - other : 1;
  // Memory for padded rows (run_repitched), for integer input whose rows are not whole 16-byte units:
  // one piece.  Whole rows need it only at an odd address (int8; 4-bit uses its planes memory then).
  const size_t row_bytes = (size_t)n_inputs * (c.fmt == XCORR_IN_CI4 ? 1 : 2);
  const size_t padded = padded_row_bytes(c.fmt, n_inputs);
  size_t piece = padded * c.n_channels * (size_t)c.max_time_per_exec;
  const size_t piece_cap = row_bytes % 16 != 0 ? kPieceBytes : kOddAddressPieceBytes;
  if (piece > piece_cap) piece = piece_cap;
  if (decoded_ci8) {
    const size_t least = padded * (size_t)(c.max_time_per_exec < 128 ? c.max_time_per_exec : 128);
    if (c.hbm_budget_bytes && piece > room) piece = room;
    planes_bytes = piece > least ? piece : least;
  }
  if (pair) {
    e = xc::pair_ring_layout(c.fmt, n_inputs, c.n_channels, c.max_time_per_exec, 0, &ring);
    if (e != cudaSuccess && e != cudaErrorNotSupported) return cuda_fail(e, "ring layout");
    // Under a limit the ring is cut short only where all planes do not fit either: they take less than a
    // ring of whole tiles and chunks where samples or channels are few.
    const bool over = e == cudaSuccess && c.hbm_budget_bytes && ring.bytes + ring.flag_bytes > room;
    if (e == cudaErrorNotSupported || (over && planes_fit)) {
      pair = false;
      ring = xc::PairRing{};
    } else if (over) {
      e = xc::pair_ring_layout(c.fmt, n_inputs, c.n_channels, c.max_time_per_exec, room, &ring);
      if (e != cudaSuccess) return cuda_fail(e, "ring layout");
    }
    planes_bytes = pair ? ring.bytes : all_planes;
    if (pair && c.fmt == XCORR_IN_CI4 && row_bytes % 16 != 0) {
      const size_t left = room > ring.flag_bytes ? room - ring.flag_bytes : 0;
      if (c.hbm_budget_bytes && piece > left) piece = left;
      if (piece > planes_bytes) planes_bytes = piece;
    }
  }
  const size_t dev_bytes = acc_bytes + planes_bytes + ring.flag_bytes + exps_bytes + 256;
  if (c.hbm_budget_bytes && dev_bytes > c.hbm_budget_bytes)
    return fail(XCORR_ERR_BUDGET, "plan needs " + std::to_string(dev_bytes) + " device bytes, budget is " +
                                      std::to_string(c.hbm_budget_bytes));

  xcorr_plan plan = new (std::nothrow) xcorr_plan_s();
  if (!plan) return fail(XCORR_ERR_OOM, "host allocation failed");
  plan->cfg = c;
  plan->cfg.engine = static_cast<xcorr_engine>(engine);
  plan->device = dev;
  plan->num_sms = prop.multiProcessorCount;
  plan->n_inputs = n_inputs;
  plan->ni_pad = ni_pad;
  plan->pack = pack;
  plan->staged_ci8 = staged_ci8;
  plan->n_pairs = n_pairs;
  plan->engine = engine;
  plan->max_integration = max_int;
  plan->planes_bytes = planes_bytes;
  plan->device_bytes = dev_bytes;
  plan->elem_bytes = elem_bytes;
  plan->planes_per_chan = ppc;
  plan->pair = pair;
  plan->ring = ring;
  plan->window_samples = c.fmt == XCORR_IN_CI4 ? xc::kTcWindowCI4 : xc::kTcWindowBF16;
  plan->exp_windows = exp_windows;
  // 4-bit input starts on the fused kernel with the A operand in tensor memory (the fastest
  // shape measured), in its small-problem layout where that measured faster: at most 64 inputs
  // (channels packed per tile) with 1024 or more samples per execute or 256 or more channels;
  // the planes path reads the same tuning as its 4 x 48 KB ring
  plan->tune_variant = c.fmt != XCORR_IN_CI4 ? 0
                       : (n_inputs <= 64 && (c.max_time_per_exec >= 1024 || c.n_channels >= 256)) ? xc::kSmallFusedVariant
                                                                                                   : xc::kDefaultFusedVariant;

  if ((e = cudaMalloc(&plan->acc, acc_bytes)) != cudaSuccess ||
      (planes_bytes && (e = cudaMalloc(&plan->planes, planes_bytes)) != cudaSuccess) ||
      (exps_bytes && (e = cudaMalloc(&plan->exps, exps_bytes)) != cudaSuccess) ||
      (pair && (e = cudaMalloc(&plan->ring_flags, ring.flag_bytes)) != cudaSuccess) ||
      (e = cudaMalloc(&plan->status, 256)) != cudaSuccess ||
      (e = cudaMallocHost(&plan->status_host, sizeof(int))) != cudaSuccess) {
    release(plan);
    delete plan;
    cudaGetLastError();
    return fail(e == cudaErrorMemoryAllocation ? XCORR_ERR_OOM : XCORR_ERR_CUDA,
                std::string("device allocation failed: ") + cudaGetErrorString(e));
  }
  *plan->status_host = 0;
  if (engine == XCORR_ENGINE_TENSOR) {
    e = cudaStreamCreateWithFlags(&plan->s_unpack, cudaStreamNonBlocking);
    for (int k = 0; k < 2 && e == cudaSuccess; ++k) e = cudaStreamCreateWithFlags(&plan->s_x[k], cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&plan->ev_fork, cudaEventDisableTiming);
    for (int k = 0; k < xc::kMaxGroups && e == cudaSuccess; ++k)
      e = cudaEventCreateWithFlags(&plan->ev_unpacked[k], cudaEventDisableTiming);
    for (int k = 0; k < 2 && e == cudaSuccess; ++k) e = cudaEventCreateWithFlags(&plan->ev_x_done[k], cudaEventDisableTiming);
    if (e != cudaSuccess) {
      release(plan);
      delete plan;
      return cuda_fail(e, "stream or event creation");
    }
  }
  if (pair) {
    // a last tile's inputs past n_inputs are read but never written: any finite number will do
    if ((n_inputs % 128 && (e = cudaMemset(plan->planes, 0, ring.bytes)) != cudaSuccess) ||
        (e = cudaMemset(plan->ring_flags, 0, ring.flag_bytes)) != cudaSuccess) {
      release(plan);
      delete plan;
      return cuda_fail(e, "ring initialisation");
    }
  }
  if (plan->exps && (e = cudaMemset(plan->exps, 0, exps_bytes)) != cudaSuccess) {
    release(plan);
    delete plan;
    return cuda_fail(e, "exponent clear");
  }
  if ((e = cudaMemset(plan->status, 0, 256)) != cudaSuccess || (e = cudaDeviceSynchronize()) != cudaSuccess) {
    release(plan);
    delete plan;
    return cuda_fail(e, "plan initialisation");
  }
  *out = plan;
  return XCORR_OK;
}

xcorr_status xcorr_execute(xcorr_plan plan, const void* d_in, int n_time, void* stream) {
  xc::NvtxRange range("xcorr_execute");
  xcorr_status st = check_execute(plan, d_in, n_time);
  if (st != XCORR_OK) return st;
  st = run_execute(plan, d_in, n_time, plan->acc, plan->fresh, static_cast<cudaStream_t>(stream));
  if (st != XCORR_OK) return st;
  plan->samples += n_time;
  plan->fresh = false;
  return XCORR_OK;
}

}  // extern "C"

namespace {

// store: a wide output is written, not added to.
xcorr_status dump(xcorr_plan plan, void* out, int out_on_device, unsigned flags, bool store, void* stream,
                  int64_t* n_samples) {
  xc::NvtxRange range("xcorr_dump");
  xcorr_status st = plan_ok(plan);
  if (st != XCORR_OK) return st;
  if (!out) return fail(XCORR_ERR_INVALID_ARG, "out is NULL");
  if (flags & ~(XCORR_DUMP_RESET | XCORR_DUMP_ADD_WIDE)) return fail(XCORR_ERR_INVALID_ARG, "unknown dump flag");
  const bool wide = (flags & XCORR_DUMP_ADD_WIDE) != 0;
  if (wide && !out_on_device) return fail(XCORR_ERR_INVALID_ARG, "XCORR_DUMP_ADD_WIDE needs device memory");
  if (wide && reinterpret_cast<uintptr_t>(out) % 16)
    return fail(XCORR_ERR_INVALID_ARG, "the wide output must be 16-byte aligned");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int64_t total = (int64_t)plan->cfg.n_channels * plan->n_pairs;
  const size_t bytes = (size_t)total * 8;
  cudaError_t e;
  if (plan->fresh) {  // nothing integrated since the last reset: the integration is zero
    e = cudaMemsetAsync(plan->acc, 0, bytes, s);
    if (e != cudaSuccess) return cuda_fail(e, "accumulator clear");
    plan->fresh = false;
  }
  if (wide) {
    if (plan->cfg.fmt == XCORR_IN_CF32)
      e = xc::launch_fold_wide_f64(static_cast<const float2*>(plan->acc), static_cast<double*>(out), total, !store, s);
    else
      e = xc::launch_fold_wide_i64(static_cast<const int2*>(plan->acc), static_cast<int64_t*>(out), total, !store, s);
    if (e != cudaSuccess) return cuda_fail(e, "fold launch");
  } else {
    e = cudaMemcpyAsync(out, plan->acc, bytes, out_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return cuda_fail(e, "dump copy");
  }
  e = cudaMemcpyAsync(plan->status_host, plan->status, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return cuda_fail(e, "status copy");
  if (n_samples) *n_samples = plan->samples;
  if (flags & XCORR_DUMP_RESET) {
    plan->samples = 0;
    plan->fresh = true;
  }
  return XCORR_OK;
}

}  // namespace

extern "C" {

xcorr_status xcorr_dump(xcorr_plan plan, void* out, int out_on_device, unsigned flags, void* stream,
                        int64_t* n_samples) {
  return dump(plan, out, out_on_device, flags, false, stream, n_samples);
}

// For the Python binding, which makes the wide output itself: xcorr_dump with XCORR_DUMP_ADD_WIDE into
// device memory that holds zeros, without the zeros.
xcorr_status xcorr_dump_wide_new_(xcorr_plan plan, void* out, unsigned flags, void* stream, int64_t* n_samples) {
  return dump(plan, out, 1, flags | XCORR_DUMP_ADD_WIDE, true, stream, n_samples);
}

xcorr_status xcorr_accum_load(xcorr_plan plan, const void* src, int src_on_device, int64_t n_samples, void* stream) {
  xcorr_status st = plan_ok(plan);
  if (st != XCORR_OK) return st;
  if (!src) return fail(XCORR_ERR_INVALID_ARG, "src is NULL");
  if (n_samples < 0) return fail(XCORR_ERR_INVALID_ARG, "n_samples must be >= 0");
  if (n_samples > plan->max_integration)
    return fail(XCORR_ERR_OVERFLOW, "n_samples exceeds " + std::to_string(plan->max_integration) +
                                        " samples (the exact range of one dump)");
  if (!plan->fresh || plan->samples != 0)
    return fail(XCORR_ERR_INVALID_ARG, "the plan holds an integration: dump it with XCORR_DUMP_RESET first");
  const size_t bytes = (size_t)plan->cfg.n_channels * plan->n_pairs * 8;
  const cudaError_t e = cudaMemcpyAsync(plan->acc, src, bytes,
                                        src_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                                        static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return cuda_fail(e, "accumulator load");
  plan->samples = n_samples;
  plan->fresh = false;
  return XCORR_OK;
}

xcorr_status xcorr_execute_dump(xcorr_plan plan, const void* d_in, int n_time, void* out, int out_on_device,
                                unsigned flags, void* stream, int64_t* n_samples) {
  xc::NvtxRange range("xcorr_execute_dump");
  xcorr_status st = check_execute(plan, d_in, n_time);
  if (st != XCORR_OK) return st;
  if (!out) return fail(XCORR_ERR_INVALID_ARG, "out is NULL");
  if (flags & ~(XCORR_DUMP_RESET | XCORR_DUMP_ADD_WIDE)) return fail(XCORR_ERR_INVALID_ARG, "unknown dump flag");
  const bool direct = plan->fresh && (flags & XCORR_DUMP_RESET) && !(flags & XCORR_DUMP_ADD_WIDE) && out_on_device;
  if (!direct) {
    st = xcorr_execute(plan, d_in, n_time, stream);
    if (st != XCORR_OK) return st;
    return xcorr_dump(plan, out, out_on_device, flags, stream, n_samples);
  }
  // This execute is the whole integration and it is not kept: the X kernel
  // writes it straight into the caller's buffer and the plan stays reset.  (No
  // copy of the status word follows, which would put a copy between every two
  // kernels of back-to-back calls: a kernel failure is reported by xcorr_sync.)
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  st = run_execute(plan, d_in, n_time, out, true, s);
  if (st != XCORR_OK) return st;
  if (n_samples) *n_samples = n_time;
  return XCORR_OK;
}

xcorr_status xcorr_execute_dump_host(xcorr_plan plan, const void* h_in, int n_time, void* h_out, int n_groups,
                                     void* stream) {
  xc::NvtxRange range("xcorr_execute_dump_host");
  xcorr_status st = check_execute(plan, h_in, n_time);
  if (st != XCORR_OK) return st;
  if (!h_out) return fail(XCORR_ERR_INVALID_ARG, "h_out is NULL");
  if (!plan->fresh || plan->samples != 0)
    return fail(XCORR_ERR_INVALID_ARG, "the plan holds an integration: dump it with XCORR_DUMP_RESET first");
  if (n_groups < 0) return fail(XCORR_ERR_INVALID_ARG, "n_groups must be >= 0");
  const int C = plan->cfg.n_channels, N = plan->n_inputs;
  const size_t in_elem = plan->cfg.fmt == XCORR_IN_CI4 ? 1 : plan->cfg.fmt == XCORR_IN_CI8 ? 2 : 8;
  const size_t chan_bytes = in_elem * N;  // one channel of one sample
  const size_t row_bytes = chan_bytes * C;
  const size_t stage_bytes = row_bytes * plan->cfg.max_time_per_exec;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e;
  // made on first use, each piece on its own so that a failed call leaves nothing half-made
  if (!plan->host_stage) {
    if ((e = cudaMalloc(&plan->host_stage, stage_bytes)) != cudaSuccess) {
      plan->host_stage = nullptr;
      cudaGetLastError();
      return fail(XCORR_ERR_OOM, "host-execute staging buffer: " + std::string(cudaGetErrorString(e)));
    }
    plan->host_stage_bytes = stage_bytes;
    plan->device_bytes += stage_bytes;
  }
  if (!plan->s_down && (e = cudaStreamCreateWithFlags(&plan->s_down, cudaStreamNonBlocking)) != cudaSuccess) {
    plan->s_down = nullptr;
    return cuda_fail(e, "stream create");
  }
  for (cudaEvent_t* ev : {&plan->ev_down}) {
    if (!*ev && (e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming)) != cudaSuccess) {
      *ev = nullptr;
      return cuda_fail(e, "event create");
    }
  }
  for (int g = 0; g < xc::kMaxGroups; ++g)
    for (cudaEvent_t* ev : {&plan->ev_up[g], &plan->ev_group_done[g]})
      if (!*ev && (e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming)) != cudaSuccess) {
        *ev = nullptr;
        return cuda_fail(e, "event create");
      }
  uint8_t* stage = static_cast<uint8_t*>(plan->host_stage);
  const size_t out_chan_bytes = static_cast<size_t>(plan->n_pairs) * 8;
  const bool staged = staged_execute(plan, stage, n_time);
  const bool fused = plan->engine == XCORR_ENGINE_TENSOR && fused_applies(plan, stage), raw = !staged && raw_ci8_applies(plan, stage);
  const Pieces pieces = fused || raw || staged ? Pieces{} : repitch_pieces(plan, n_time);
  if (!fused && !raw && !pieces.pitch) {
    // one piece: up, X-stage, down, in order on the caller's stream
    if ((e = cudaMemcpyAsync(stage, h_in, row_bytes * n_time, cudaMemcpyHostToDevice, s)) != cudaSuccess)
      return cuda_fail(e, "input copy");
    if ((st = run_execute(plan, stage, n_time, plan->acc, true, s)) != XCORR_OK) return st;
    if ((e = cudaMemcpyAsync(h_out, plan->acc, out_chan_bytes * C, cudaMemcpyDeviceToHost, s)) != cudaSuccess)
      return cuda_fail(e, "output copy");
  } else {
    // channel groups: group g goes up on s_unpack, is correlated on s_x[g % 2] (a
    // launch can start on the SMs the previous one's tail leaves idle) and comes
    // down on s_down while later groups are still moving
    int edge[xc::kMaxGroups + 1];  // group g: channels edge[g] .. edge[g + 1] - 1
    int G = host_groups(C, row_bytes * n_time + out_chan_bytes * C, edge);
    int most = fused ? xc::kMaxGroups : G;  // (padded rows and int8: more groups than the library's choice only add launches)
    if (plan->cfg.fmt == XCORR_IN_CI8) {
      const int m = ci8_host_groups(row_bytes * n_time, n_time, raw);
      if (m < most) most = m;
    }
    if (pageable(h_in) || pageable(h_out)) most = 1;  // (its copies overlap nothing, and narrow columns of it take longer)
    if (n_groups > 0 || G > most) G = even_groups(C, n_groups > 0 && n_groups < most ? n_groups : most, edge);
    // timed as other executes: no unpack, a launch (or a piece's two) per group
    cudaEvent_t* ev = plan->prof_cap && !fused ? plan->prof_events + xc::kProfileEvents * (plan->prof_count % plan->prof_cap) : nullptr;
    if (ev && ((e = cudaEventRecord(ev[0], s)) != cudaSuccess || (e = cudaEventRecord(ev[1], s)) != cudaSuccess))
      return cuda_fail(e, "profile event");
    int timed = 0;
    if ((e = cudaEventRecord(plan->ev_fork, s)) != cudaSuccess) return cuda_fail(e, "fork event");
    for (cudaStream_t t : {plan->s_unpack, plan->s_x[0], plan->s_x[1], plan->s_down})
      if ((e = cudaStreamWaitEvent(t, plan->ev_fork, 0)) != cudaSuccess) return cuda_fail(e, "fork wait");
    for (int g = 0; g < G; ++g) {
      const int c0 = edge[g], c1 = edge[g + 1];
      if (c1 <= c0) continue;
      const size_t off = chan_bytes * c0, width = chan_bytes * (c1 - c0);
      cudaStream_t sx = plan->s_x[pieces.pitch ? 0 : g & 1];  // (padded rows: one piece of memory)
      int2* out_g = static_cast<int2*>(plan->acc) + static_cast<int64_t>(c0) * plan->n_pairs;
      // (all channels: one run of bytes, which the copy engines take faster than as rows)
      if ((e = width == row_bytes ? cudaMemcpyAsync(stage, h_in, row_bytes * n_time, cudaMemcpyHostToDevice, plan->s_unpack)
                                  : cudaMemcpy2DAsync(stage + off, row_bytes, static_cast<const uint8_t*>(h_in) + off, row_bytes,
                                                      width, n_time, cudaMemcpyHostToDevice, plan->s_unpack)) != cudaSuccess ||
          (e = cudaEventRecord(plan->ev_up[g], plan->s_unpack)) != cudaSuccess ||
          (e = cudaStreamWaitEvent(sx, plan->ev_up[g], 0)) != cudaSuccess)
        return cuda_fail(e, "group input copy");
      if (ev && (e = cudaEventRecord(ev[2 + 2 * timed], sx)) != cudaSuccess) return cuda_fail(e, "profile event");
      e = fused ? xc::launch_xcorr_tc_fused_ci4(stage + off, C, plan->tune_variant, n_time, c1 - c0, N, out_g, false,
                                                plan->status, plan->num_sms, sx)
          : raw ? xc::launch_xcorr_tc_raw_pair(reinterpret_cast<const int8_t*>(stage + off), C, n_time, c1 - c0, N, N, out_g,
                                               false, plan->status, plan->num_sms, sx)
                : run_repitched(plan, pieces, stage + off, c1 - c0, n_time, out_g, true, sx);
      if (e != cudaSuccess) return cuda_fail(e, "X kernel launch");
      if (ev && (e = cudaEventRecord(ev[3 + 2 * timed], sx)) != cudaSuccess) return cuda_fail(e, "profile event");
      ++timed;
      if ((e = cudaEventRecord(plan->ev_group_done[g], sx)) != cudaSuccess ||
          (e = cudaStreamWaitEvent(plan->s_down, plan->ev_group_done[g], 0)) != cudaSuccess ||
          (e = cudaMemcpyAsync(static_cast<uint8_t*>(h_out) + out_chan_bytes * c0, out_g, out_chan_bytes * (c1 - c0),
                               cudaMemcpyDeviceToHost, plan->s_down)) != cudaSuccess)
        return cuda_fail(e, "group output copy");
    }
    if (ev) {
      plan->prof_ngroups[plan->prof_count % plan->prof_cap] = timed;
      ++plan->prof_count;
    }
    // join: every group's copy-out is on s_down, after its X launch and its input copy
    if ((e = cudaEventRecord(plan->ev_down, plan->s_down)) != cudaSuccess ||
        (e = cudaStreamWaitEvent(s, plan->ev_down, 0)) != cudaSuccess)
      return cuda_fail(e, "join");
  }
  if ((e = cudaMemcpyAsync(plan->status_host, plan->status, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess)
    return cuda_fail(e, "status copy");
  return XCORR_OK;
}

xcorr_status xcorr_sync(xcorr_plan plan, void* stream) {
  xcorr_status st = plan_ok(plan);
  if (st != XCORR_OK) return st;
  cudaError_t e = cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
  int code = 0;
  e = cudaMemcpy(&code, plan->status, sizeof(int), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "status read");
  if (code) {
    plan->sticky = code;
    return plan_ok(plan);
  }
  return XCORR_OK;
}

xcorr_status xcorr_plan_query(xcorr_plan plan, xcorr_plan_info* info) {
  if (!plan || !info) return fail(XCORR_ERR_INVALID_ARG, "plan or info is NULL");
  info->n_inputs = plan->n_inputs;
  info->n_channels = plan->cfg.n_channels;
  info->n_pairs = plan->n_pairs;
  info->engine = plan->engine;
  info->samples_integrated = plan->samples;
  info->max_integration = plan->max_integration;
  info->device_bytes = plan->device_bytes;
  info->output_bytes = (size_t)plan->cfg.n_channels * plan->n_pairs * 8;
  const bool fused = plan->engine == XCORR_ENGINE_TENSOR && plan->cfg.fmt == XCORR_IN_CI4 && !plan->tune_unfused &&
                     plan->n_inputs % 16 == 0;
  // (int8: a 16-byte aligned input, nullptr standing for one)
  const bool raw = !plan->staged_ci8 && raw_ci8_applies(plan, nullptr), one_launch = plan->pair || raw;
  const Pieces pieces = fused || raw || plan->staged_ci8 ? Pieces{} : repitch_pieces(plan, plan->cfg.max_time_per_exec);
  info->kernels_per_execute = fused ? xc::fused_launches(plan->tune_variant, plan->cfg.max_time_per_exec, plan->cfg.n_channels,
                                                         plan->n_inputs, plan->num_sms)
                              : pieces.pitch ? repitched_launches(plan, pieces, plan->cfg.max_time_per_exec)
                              : one_launch                          ? 1
                              : plan->engine == XCORR_ENGINE_TENSOR ? 2 * tensor_groups(plan)
                                                                     : 1;
  info->tuning.stage_variant = plan->tune_variant;
  info->tuning.groups = fused || one_launch || pieces.pitch ? 1 : tensor_groups(plan);
  info->tuning.x_streams = plan->tune_x_streams;
  info->tuning.unfused = plan->tune_unfused;
  return XCORR_OK;
}

xcorr_status xcorr_plan_set_tuning(xcorr_plan plan, const xcorr_tuning* t) {
  xcorr_status st = plan_ok(plan);
  if (st != XCORR_OK) return st;
  if (!t) return fail(XCORR_ERR_INVALID_ARG, "tuning is NULL");
  if (t->stage_variant < 0 || t->stage_variant >= xc::kFusedVariants)
    return fail(XCORR_ERR_INVALID_ARG, "stage_variant must be in [0, " + std::to_string(xc::kFusedVariants - 1) + "]");
  if (t->groups < 0 || t->groups > xc::kMaxGroups) return fail(XCORR_ERR_INVALID_ARG, "groups must be in [0, 8]");
  if (t->x_streams != 1 && t->x_streams != 2) return fail(XCORR_ERR_INVALID_ARG, "x_streams must be 1 or 2");
  if (t->unfused != 0 && t->unfused != 1) return fail(XCORR_ERR_INVALID_ARG, "unfused must be 0 or 1");
  plan->tune_variant = t->stage_variant;
  plan->tune_groups = t->groups;
  plan->tune_x_streams = t->x_streams;
  plan->tune_unfused = t->unfused;
  return XCORR_OK;
}

xcorr_status xcorr_autotune(xcorr_plan plan, const void* d_in, int n_time, void* stream, xcorr_tuning* best,
                            float* best_ms) {
  xcorr_status st = plan_ok(plan);
  if (st != XCORR_OK) return st;
  if (!d_in || n_time < 1 || n_time > plan->cfg.max_time_per_exec)
    return fail(XCORR_ERR_INVALID_ARG, "d_in must be set and n_time in [1, max_time_per_exec]");
  if (plan->engine != XCORR_ENGINE_TENSOR) {  // nothing to tune
    if (best) *best = xcorr_tuning{plan->tune_variant, plan->tune_groups, plan->tune_x_streams, plan->tune_unfused};
    if (best_ms) *best_ms = 0.f;
    return XCORR_OK;
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaError_t e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  if (e != cudaSuccess) {
    if (e0) cudaEventDestroy(e0);
    return cuda_fail(e, "cudaEventCreate");
  }
  const int saved_cap = plan->prof_cap;
  plan->prof_cap = 0;  // candidates are not profiled
  const int group_choices[] = {1, 2, 4, 8};
  xcorr_tuning winner{plan->tune_variant, plan->tune_groups, plan->tune_x_streams, plan->tune_unfused};
  float winner_ms = 1e30f;
  // candidates: the fused 4-bit kernels' shapes where one applies (over padded rows: those of the
  // kernel that takes them), then every planes-based shape
  plan->tune_unfused = 0;
  const bool fused_ok = fused_applies(plan, d_in);
  const bool padded_ci4 = !fused_ok && plan->cfg.fmt == XCORR_IN_CI4 && repitch_pieces(plan, n_time).pitch > 0;
  for (int uf = fused_ok || padded_ci4 ? 0 : 1; uf <= 1 && st == XCORR_OK; ++uf)
  for (int v = 0; v < (uf == 0 ? xc::kFusedVariants : xc::kTcVariants) && st == XCORR_OK; ++v) {
    for (int gi = 0; gi < 4 && st == XCORR_OK; ++gi) {
      for (int xs = 1; xs <= 2 && st == XCORR_OK; ++xs) {
        if (group_choices[gi] == 1 && xs == 2) continue;  // one group has one X launch
        if (uf == 0 && (gi > 0 || xs > 1)) continue;      // the fused kernel is one launch
        if (uf == 0 && padded_ci4 && padded_shape(v) != v - 4 && v != xc::kSmallFusedVariant) continue;
        // the CTA-pair kernels have one shape each
        if (uf == 1 && (plan->pair || (plan->cfg.fmt == XCORR_IN_CI8 && !staged_execute(plan, d_in, n_time))) && (v > 0 || gi > 0)) continue;
        if (uf == 1 && plan->pack > 1 && v > 0) continue;  // nor have packed channels another
        plan->tune_variant = v;
        plan->tune_groups = group_choices[gi];
        plan->tune_x_streams = xs;
        plan->tune_unfused = uf;
        float best_rep = 1e30f;
        for (int rep = 0; rep < 3 && st == XCORR_OK; ++rep) {  // the first run warms up
          cudaEventRecord(e0, s);
          st = run_execute(plan, d_in, n_time, plan->acc, true, s);
          cudaEventRecord(e1, s);
          if (st != XCORR_OK) break;
          if ((e = cudaEventSynchronize(e1)) != cudaSuccess) {
            st = cuda_fail(e, "autotune timing");
            break;
          }
          float ms = 0.f;
          cudaEventElapsedTime(&ms, e0, e1);
          if (rep > 0 && ms < best_rep) best_rep = ms;
        }
        if (st == XCORR_OK && best_rep < winner_ms) {
          winner_ms = best_rep;
          winner = xcorr_tuning{v, group_choices[gi], xs, uf};
        }
      }
    }
  }
  plan->prof_cap = saved_cap;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  // the candidates overwrote the accumulator: the plan starts a new integration
  plan->samples = 0;
  plan->fresh = true;
  plan->tune_variant = winner.stage_variant;
  plan->tune_groups = winner.groups;
  plan->tune_x_streams = winner.x_streams;
  plan->tune_unfused = winner.unfused;
  if (st != XCORR_OK) return st;
  if (best) *best = winner;
  if (best_ms) *best_ms = winner_ms;
  return XCORR_OK;
}

xcorr_status xcorr_autotune_cached(xcorr_plan plan, const void* d_in, int n_time, void* stream, xcorr_tuning* best,
                                   float* best_ms, int* from_cache) {
  xcorr_status st = plan_ok(plan);
  if (st != XCORR_OK) return st;
  if (!d_in || n_time < 1 || n_time > plan->cfg.max_time_per_exec)
    return fail(XCORR_ERR_INVALID_ARG, "d_in must be set and n_time in [1, max_time_per_exec]");
  if (from_cache) *from_cache = 0;
  if (plan->engine != XCORR_ENGINE_TENSOR) return xcorr_autotune(plan, d_in, n_time, stream, best, best_ms);
  const xc::TuneKey key = xc::tune_key("plan", plan->cfg.fmt, plan->n_inputs, plan->cfg.n_channels, n_time);
  xcorr_tuning t{};
  float ms = 0.f;
  if (xc::tune_cache_get(key, &t, &ms)) {
    st = xcorr_plan_set_tuning(plan, &t);
    if (st != XCORR_OK) return st;
    plan->samples = 0;  // as the timed path: the plan starts a new integration
    plan->fresh = true;
    if (best) *best = t;
    if (best_ms) *best_ms = ms;
    if (from_cache) *from_cache = 1;
    return XCORR_OK;
  }
  st = xcorr_autotune(plan, d_in, n_time, stream, &t, &ms);
  if (st != XCORR_OK) return st;
  xc::tune_cache_put(key, t, ms);
  if (best) *best = t;
  if (best_ms) *best_ms = ms;
  return XCORR_OK;
}

xcorr_status xcorr_profile_enable(xcorr_plan plan, int capacity) {
  xcorr_status st = plan_ok(plan);
  if (st != XCORR_OK) return st;
  if (capacity < 0 || capacity > (1 << 16)) return fail(XCORR_ERR_INVALID_ARG, "capacity must be in [0, 65536]");
  free_profile(plan);
  if (capacity == 0) return XCORR_OK;
  const int64_t n = (int64_t)xc::kProfileEvents * capacity;
  plan->prof_events = new (std::nothrow) cudaEvent_t[n]();
  plan->prof_ngroups = new (std::nothrow) int[capacity]();
  if (!plan->prof_events || !plan->prof_ngroups) {
    free_profile(plan);
    return fail(XCORR_ERR_OOM, "host allocation failed");
  }
  plan->prof_cap = capacity;
  for (int64_t k = 0; k < n; ++k) {
    cudaError_t e = cudaEventCreate(&plan->prof_events[k]);
    if (e != cudaSuccess) {
      free_profile(plan);
      return cuda_fail(e, "cudaEventCreate");
    }
  }
  return XCORR_OK;
}

xcorr_status xcorr_profile_read(xcorr_plan plan, float* ms, int capacity, int* count) {
  xcorr_status st = plan_ok(plan);
  if (st != XCORR_OK) return st;
  if (!ms || !count || capacity < 0) return fail(XCORR_ERR_INVALID_ARG, "ms or count is NULL");
  *count = 0;
  if (!plan->prof_cap) return XCORR_OK;
  const int64_t have = plan->prof_count < plan->prof_cap ? plan->prof_count : plan->prof_cap;
  const int64_t n = have < capacity ? have : capacity;
  for (int64_t k = 0; k < n; ++k) {
    const int64_t slot = (plan->prof_count - n + k) % plan->prof_cap;
    cudaEvent_t* ev = plan->prof_events + xc::kProfileEvents * slot;
    const int groups = plan->prof_ngroups[slot];
    float unpack = 0.f, x = 0.f;
    cudaError_t e = cudaEventSynchronize(ev[1]);
    if (e == cudaSuccess) e = cudaEventElapsedTime(&unpack, ev[0], ev[1]);
    for (int g = 0; g < groups && e == cudaSuccess; ++g) {
      float d = 0.f;
      e = cudaEventSynchronize(ev[3 + 2 * g]);
      if (e == cudaSuccess) e = cudaEventElapsedTime(&d, ev[2 + 2 * g], ev[3 + 2 * g]);
      x += d;
    }
    if (e != cudaSuccess) return cuda_fail(e, "profile read");
    ms[2 * k] = unpack;
    ms[2 * k + 1] = x;
  }
  *count = static_cast<int>(n);
  return XCORR_OK;
}

xcorr_status xcorr_destroy(xcorr_plan plan) {
  if (!plan) return XCORR_OK;
  cudaSetDevice(plan->device);
  cudaError_t e = cudaDeviceSynchronize();
  release(plan);
  delete plan;
  if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceSynchronize at destroy");
  return XCORR_OK;
}

xcorr_status xcorr_baseline_index(int n_stations, int a, int b, int p, int q, int64_t* idx, int* conj) {
  if (!idx || !conj) return fail(XCORR_ERR_INVALID_ARG, "idx or conj is NULL");
  if (n_stations < 1 || a < 0 || a >= n_stations || b < 0 || b > a || p < 0 || p > 1 || q < 0 || q > 1)
    return fail(XCORR_ERR_INVALID_ARG, "need 0 <= b <= a < n_stations and pols in {0, 1}");
  int64_t i = 2LL * a + p, j = 2LL * b + q;
  *conj = 0;
  if (j > i) {  // only for a == b, p < q: the stored pair is (j, i)
    const int64_t t = i;
    i = j;
    j = t;
    *conj = 1;
  }
  *idx = i * (i + 1) / 2 + j;
  return XCORR_OK;
}

}  // extern "C"
