// pair_common.cuh -- what the CTA-pair X kernels share: which tile pair a CTA
// works on, and writing a finished 128 x 128 tile into the packed triangle.
#pragma once
#include <cstdint>

#include "fused_pairing.h"
#include "sm103_ptx.cuh"

namespace xc {
namespace pairs {

constexpr int kBlk = 128;          // inputs per tile side
constexpr int kHalf = 64;          // column-tile inputs each CTA provides; columns per epilogue thread
constexpr int kEpiWarps = 8;       // two per TMEM lane quarter, 64 columns each
constexpr int kAccCols = 256;      // [Re | X] of columns 0-63, [Re | X] of columns 64-127
constexpr uint32_t kTmemCols = 512;
constexpr int kOutCols = 8;        // columns per shared-memory transpose step
constexpr int kOutPitch = kOutCols + 1;  // 8-byte words per staged row
constexpr int kStagingBytes = kEpiWarps * 32 * kOutPitch * 8;
constexpr uint32_t kSignalBytes = 16;    // a signal from the odd CTA to the even one

struct Item {
  int chan, S, R;  // channel, column tile, this CTA's row tile (-1: none)
  bool has_row, transposed;
};

// Entry q (channel-major) of a problem of nb tiles a side, n_entries pair entries a channel.
__device__ __forceinline__ Item item_of(int nb, int n_entries, int q, uint32_t rank) {
  Item it;
  it.chan = q / n_entries;
  int r0, r1;
  fused::pair_entry(nb, q - it.chan * n_entries, it.S, r0, r1);
  it.R = rank == 0 ? r0 : r1;
  it.has_row = it.R >= 0;
  it.transposed = it.has_row && it.R < it.S;
  return it;
}

// An epilogue warp's 32 rows x 64 columns of a tile: where its pairs go.  Rows are written 8 columns
// at a time through shared memory, a quarter-warp 8 consecutive pairs of a row (64 bytes).  The row
// addresses are made once, and a part wholly below the diagonal and inside the inputs takes no
// comparisons.
struct RowsOut {
  uint2* base;  // row lane / 8, column lane % 8
  int off[8];   // from there to rows 4 r + lane / 8
  int row, col0, n_inputs;
  bool whole;
};

__device__ __forceinline__ void rows_out(RowsOut& o, uint2* out_c, int row0, int col0, int n_inputs, int lane) {
  o.row = row0 + (lane >> 3);
  o.col0 = col0 + (lane & 7);
  o.n_inputs = n_inputs;
  o.whole = col0 + kHalf - 1 <= row0 && row0 + 31 < n_inputs;
  o.base = out_c + (int64_t)o.row * (o.row + 1) / 2 + o.col0;
#pragma unroll
  for (int r = 0; r < 8; ++r) o.off[r] = 4 * r * o.row + 2 * r * (4 * r + 1);  // i (i + 1) / 2 at i = row + 4 r
}

template <bool FLOAT>
__device__ __forceinline__ uint2 add_pair(uint2 v, uint2 old) {
  if (FLOAT)
    return make_uint2(__float_as_uint(__uint_as_float(v.x) + __uint_as_float(old.x)),
                      __float_as_uint(__uint_as_float(v.y) + __uint_as_float(old.y)));
  return make_uint2(v.x + old.x, v.y + old.y);
}

// Columns ch .. ch + 7 of the part (lane = row): v -> memory, added to what is there if ADD.
template <bool FLOAT, bool ADD>
__device__ __forceinline__ void put_rows(const RowsOut& o, uint2* stage_rows, const uint2 (&v)[8], int ch, int lane) {
#pragma unroll
  for (int k = 0; k < 8; ++k) stage_rows[lane * kOutPitch + k] = v[k];
  __syncwarp();
  uint2 w[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) w[r] = stage_rows[(4 * r + (lane >> 3)) * kOutPitch + (lane & 7)];
  const int j = o.col0 + ch;
  if (ADD) {  // all loads of the lane in flight together
    uint2 old[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int i = o.row + 4 * r;
      old[r] = o.whole || (i < o.n_inputs && j <= i) ? o.base[o.off[r] + ch] : make_uint2(0u, 0u);
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) w[r] = add_pair<FLOAT>(w[r], old[r]);
  }
  if (o.whole) {
#pragma unroll
    for (int r = 0; r < 8; ++r) o.base[o.off[r] + ch] = w[r];
  } else {
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int i = o.row + 4 * r;
      if (i < o.n_inputs && j <= i) o.base[o.off[r] + ch] = w[r];
    }
  }
  __syncwarp();
}

// A transposed part: V[b][a] = conj(W[a][b]), lane = a; the warp's 32 values of output row b are
// consecutive.  `row` points at pair (b0, a) and `len` is b0 + 1, the distance to the next row's.
struct ColsOut {
  uint2* row;
  int len, left;  // rows left before n_inputs
};

__device__ __forceinline__ void cols_out(ColsOut& o, uint2* out_c, int row0, int col0, int n_inputs, int lane) {
  o.row = out_c + (int64_t)col0 * (col0 + 1) / 2 + row0 + lane;
  o.len = col0 + 1;
  o.left = n_inputs - col0;
}

// The next 8 columns b of the part; v already holds conj(W[a][b]).
template <bool FLOAT, bool ADD>
__device__ __forceinline__ void put_cols(ColsOut& o, const uint2 (&v)[8]) {
  uint2* dst[8];
  uint2 old[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    dst[k] = o.row;
    o.row += o.len++;
    old[k] = ADD && k < o.left ? *dst[k] : make_uint2(0u, 0u);
  }
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if (k < o.left) *dst[k] = ADD ? add_pair<FLOAT>(v[k], old[k]) : v[k];
  o.left -= 8;
}

}  // namespace pairs
}  // namespace xc
