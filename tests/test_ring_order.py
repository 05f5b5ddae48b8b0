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


def run(name, source):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    os.makedirs(OUT, exist_ok=True)
    src, exe = os.path.join(OUT, name + ".cpp"), os.path.join(OUT, name)
    with open(src, "w") as f:
        f.write(source)
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, src, "-o", exe], check=True)
    return subprocess.run([exe], capture_output=True, text=True)


def test_a_slot_is_refilled_only_after_its_last_readers():
    r = run("ring_slots_check", CHECK_SLOTS)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
