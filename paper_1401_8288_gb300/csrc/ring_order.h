// ring_order.h -- the order of the CTA-pair kernel's ring of planes
// (xcorr_tc_pair.cu): which places there are, who reads them, when a reader reports
// and which place had a slot before.  Plain integer arithmetic for the device and the host, so that
// every size can be checked without a GPU.
//
// An entry is a pair of tile pairs of one channel, an item an entry of the launch
// (channel-major).  Items run one per cluster at a time; a batch is the items that
// run side by side, so its channels are consecutive.  A place is one time chunk of
// one channel of a batch, in the order (batch, chunk, channel of the batch); place
// u is unpacked into slot u % slots.  A batch whose channels do not fill its
// batch_chans leaves places without readers, which nobody unpacks.
#pragma once

#ifdef __CUDACC__
#define XC_RING_FN __host__ __device__ __forceinline__
#else
#define XC_RING_FN inline
#endif

namespace xc {
namespace ring {

struct Order {
  int n_items;      // entries of the launch
  int n_entries;    // of one channel
  int clusters;     // items of a batch
  int n_chunks;     // chunks along time
  int batch_chans;  // channel places of a batch
  int n_batches;
  int slots;        // ring slots
};

// The order of n_chan channels on `clusters` clusters (the caller chooses the slots).
XC_RING_FN Order make_order(int n_chan, int n_entries, int clusters, int n_chunks, int slots) {
  Order o;
  o.n_items = n_chan * n_entries;
  o.n_entries = n_entries;
  o.clusters = clusters;
  o.n_chunks = n_chunks;
  const int most = (clusters - 1) / n_entries + 2;  // channels that a batch can touch
  o.batch_chans = most < n_chan ? most : n_chan;
  o.n_batches = (o.n_items + clusters - 1) / clusters;
  o.slots = slots;
  return o;
}

XC_RING_FN int places(const Order& o) { return o.n_batches * o.n_chunks * o.batch_chans; }

// Place of (batch, chunk, channel of the batch).
XC_RING_FN int place_of(const Order& o, int batch, int chunk, int j) {
  return (batch * o.n_chunks + chunk) * o.batch_chans + j;
}

// First channel of a batch.
XC_RING_FN int first_chan(const Order& o, int batch) { return batch * o.clusters / o.n_entries; }

// CTAs that read the chunk at place u: two per entry of its channel in its batch.
XC_RING_FN int readers_of(const Order& o, int u) {
  const int j = u % o.batch_chans, batch = u / (o.batch_chans * o.n_chunks);
  const int i0 = batch * o.clusters, i1 = i0 + o.clusters < o.n_items ? i0 + o.clusters : o.n_items;
  const int c = i0 / o.n_entries + j;
  const int a = c * o.n_entries > i0 ? c * o.n_entries : i0, b = (c + 1) * o.n_entries < i1 ? (c + 1) * o.n_entries : i1;
  return b > a ? 2 * (b - a) : 0;
}

// The place whose readers have to be done before place u is unpacked: the last one before it in its
// slot that has any (a place without readers held nothing, and the slot still belongs to the one
// before), or -1.
XC_RING_FN int slot_user(const Order& o, int u) {
  int v = u - o.slots;
  while (v >= 0 && readers_of(o, v) == 0) v -= o.slots;
  return v >= 0 ? v : -1;
}

// When a CTA reports a chunk as read: once its copies have landed.  They are not waited for while
// there is work: the chunk is reported when its last stage's buffer comes round again, or at the next
// chunk's end.  But before the CTA waits for a chunk that is not unpacked yet it reports (and waits for
// the copies, which land by themselves): that unpack may be waiting for this very slot.
// So a report waits only for what is in flight, the unpack of a place only for reports of earlier
// places, and a reader only for the unpack of the place it is at: any ring of one slot or more ends.
struct Reads {
  int place = -1;  // read and not reported, or -1
  int end = 0;     // stages loaded at its end
  int stages = 0;  // stages loaded
  XC_RING_FN bool due_before_wait(bool unpacked) const { return place >= 0 && !unpacked; }
  XC_RING_FN bool due_after_stage(int stage_buffers) {
    ++stages;
    return place >= 0 && stages >= end + stage_buffers;
  }
  XC_RING_FN bool due_after_chunk() const { return place >= 0; }
  XC_RING_FN void reported() { place = -1; }
  XC_RING_FN void chunk_read(int u) {
    place = u;
    end = stages;
  }
};

}  // namespace ring
}  // namespace xc

#undef XC_RING_FN
