"""The order of the CTA-pair kernel's ring of planes (csrc/ring_order.h), checked on the host.

The unpack warps write place after place into the ring's slots while CTAs read earlier places; the
header says who reads a place and whose readers have to be done before a slot is written again.
This compiles it with g++ and goes through every place of many launches, with rings of every length
from one step of a batch on.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1401_8288_gb300", "csrc")
OUT = os.path.join(ROOT, "paper_1401_8288_gb300", "_lib")

COMMON = r'''
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "ring_order.h"
using namespace xc::ring;
struct Case { int n_chan, n_entries, clusters, n_chunks; };
// channels x entries of 2, 3, 4, 5 and 8 tiles a side x clusters (one per item, or the chip's) x chunks
static std::vector<Case> cases(int most_chan) {
  std::vector<Case> v;
  const int chans[] = {1, 2, 3, 5, 7, 16, 17, 24, 40, 77, 100};
  const int entries[] = {2, 3, 5, 8, 18}, clusters[] = {1, 2, 3, 7, 19, 75, 76}, chunks[] = {1, 2, 3, 5};
  for (int c : chans)
    for (int e : entries)
      for (int k : clusters)
        for (int t : chunks)
          if (c <= most_chan) v.push_back({c, e, c * e < k ? c * e : k, t});
  return v;
}
'''

CHECK_SLOTS = COMMON + r'''
int main() {
  long long skipped = 0, waits = 0;
  for (const Case& c : cases(100)) {
    Order o = make_order(c.n_chan, c.n_entries, c.clusters, c.n_chunks, 1);
    const int n = places(o), bc = o.batch_chans;
    // every entry of every batch reads exactly the places of its channel
    std::vector<int> readers(n, 0);
    for (int q = 0; q < o.n_items; ++q) {
      const int batch = q / o.clusters, j = q / o.n_entries - first_chan(o, batch);
      if (j < 0 || j >= bc) { std::printf("item %d: channel %d of its batch\n", q, j); return 1; }
      for (int k = 0; k < o.n_chunks; ++k) readers[place_of(o, batch, k, j)] += 2;
    }
    for (int u = 0; u < n; ++u)
      if (readers_of(o, u) != readers[u]) { std::printf("place %d: %d readers\n", u, readers_of(o, u)); return 1; }
    for (o.slots = bc; o.slots <= 3 * bc + 2 && o.slots <= n; ++o.slots) {
      std::vector<int> last(o.slots, -1);  // who wrote the slot last
      for (int u = 0; u < n; ++u) {
        if (!readers[u]) continue;
        const int s = u % o.slots;
        if (slot_user(o, u) != last[s]) {
          std::printf("%d channels, %d entries, %d clusters, %d chunks, %d slots: place %d waits for %d, slot of %d\n", c.n_chan,
                      c.n_entries, c.clusters, c.n_chunks, o.slots, u, slot_user(o, u), last[s]);
          return 1;
        }
        waits += last[s] >= 0;
        skipped += last[s] >= 0 && last[s] != u - o.slots;  // the place one ring before has no reader
        last[s] = u;
      }
    }
  }
  if (!skipped || !waits) { std::printf("no place with an empty one before it\n"); return 1; }
  std::printf("ok\n");
  return 0;
}
'''

# Every unpack warp and every reading CTA as a state machine that runs until it has to wait; waits only
# end by what others did, so if one schedule ends they all do.  argv[1]: 1 as the kernel, 0 without the
# report before a wait (which has to stop somewhere, or this shows nothing).
PLAY = COMMON + r'''
static bool play(const Order& o, int subs, int stages, int buffers, int warps, bool report_first, bool* overwrote) {
  const int n = places(o);
  std::vector<int> ready(n, 0), done(n, 0), left(n), slot(o.slots, -1);  // slot: the place whose samples it holds
  for (int u = 0; u < n; ++u) left[u] = readers_of(o, u);
  struct Warp { int u, sub; };
  std::vector<Warp> w;
  for (int k = 0; k < warps; ++k) w.push_back({0, k});
  struct Cta { int q, batch, k; Reads r; bool over; };
  std::vector<Cta> c;
  for (int k = 0; k < 2 * o.clusters; ++k) c.push_back({k / 2, 0, 0, Reads(), false});
  for (bool moved = true; moved;) {
    moved = false;
    for (Warp& x : w)
      for (;;) {
        x.u += x.sub / subs, x.sub %= subs;
        if (x.u >= n) break;
        if (readers_of(o, x.u)) {
          const int v = slot_user(o, x.u);
          if (v >= 0 && done[v] < readers_of(o, v)) break;
          const int s = x.u % o.slots;
          if (slot[s] != x.u) {
            if (slot[s] >= 0 && left[slot[s]]) *overwrote = true;
            slot[s] = x.u;
          }
          ++ready[x.u];
        }
        x.sub += warps;
        moved = true;
      }
    for (Cta& x : c)
      while (!x.over) {
        if (x.q >= o.n_items) {
          if (x.r.due_after_chunk()) ++done[x.r.place], x.r.reported();
          x.over = moved = true;
          break;
        }
        const int u = place_of(o, x.batch, x.k, x.q / o.n_entries - first_chan(o, x.batch));
        if (ready[u] < subs) {
          if (report_first && x.r.due_before_wait(false)) ++done[x.r.place], x.r.reported(), moved = true;
          break;
        }
        if (slot[u % o.slots] != u) *overwrote = true;
        for (int s = 0; s < stages; ++s)
          if (x.r.due_after_stage(buffers)) ++done[x.r.place], x.r.reported();
        if (x.r.due_after_chunk()) ++done[x.r.place], x.r.reported();
        x.r.chunk_read(u);
        --left[u];
        moved = true;
        if (++x.k == o.n_chunks) x.k = 0, ++x.batch, x.q += o.clusters;
      }
  }
  for (const Cta& x : c)
    if (!x.over) return false;
  return true;
}
int main(int argc, char** argv) {
  const bool report_first = std::atoi(argv[1]) != 0;
  int stopped = 0;
  for (const Case& c : cases(40)) {
    Order o = make_order(c.n_chan, c.n_entries, c.clusters, c.n_chunks, 1);
    const int n = places(o), bc = o.batch_chans, lens[] = {1, bc, bc + 1, 2 * bc - 1, 2 * bc, 3 * bc};
    for (int len : lens)
      for (int stages : {1, 8, 72}) {
        o.slots = len < n ? len : n;
        bool overwrote = false;
        if (!play(o, 5, stages, 6, 4 * 2 * o.clusters, report_first, &overwrote)) {
          ++stopped;
          if (report_first) {
            std::printf("%d channels, %d entries, %d clusters, %d chunks, %d slots, %d stages: stopped\n", c.n_chan, c.n_entries,
                        c.clusters, c.n_chunks, o.slots, stages);
            return 1;
          }
        }
        if (overwrote) { std::printf("a slot was overwritten before it was read\n"); return 1; }
      }
  }
  std::printf(stopped ? "stopped\n" : "ok\n");
  return 0;
}
'''


def run(name, source, *args):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    os.makedirs(OUT, exist_ok=True)
    src, exe = os.path.join(OUT, name + ".cpp"), os.path.join(OUT, name)
    with open(src, "w") as f:
        f.write(source)
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, src, "-o", exe], check=True)
    return subprocess.run([exe, *args], capture_output=True, text=True)


def test_a_slot_is_refilled_only_after_its_last_readers():
    r = run("ring_slots_check", CHECK_SLOTS)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout


def test_the_order_ends_with_any_ring():
    r = run("ring_play_check", PLAY, "1")
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout


def test_the_order_needs_the_report_before_a_wait():
    r = run("ring_play_check", PLAY, "0")
    assert r.returncode == 0 and r.stdout.strip() == "stopped", r.stdout
