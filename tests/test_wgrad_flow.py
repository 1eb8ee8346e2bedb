"""Control flow of the weight-gradient kernel's worker threads (csrc/unet_wgrad_flow.h),
compiled for the host: every thread passes the same barriers whichever of them sees a wait
expire, and no copy is requested before the last reader of its slot is done."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_00822_gb300", "csrc")

MODEL = r"""
#include "unet_wgrad_flow.h"
#include <cstdio>
#include <vector>
using namespace bfcs::net;

// One thread: its wait for tile `expire` (and all later ones) runs out; -1: none does.  The
// barrier results are the thread's own `ok` if given == null, else given[i] for barrier i.
struct Thread {
  std::vector<int> barriers;   // results
  std::vector<int> groups;     // copy groups in flight at the barriers
  int missing = 0;             // barriers past the other thread's last one
  bool result = true, bad = false;
  int requested = 0, published = 0, drained = 0;
};

Thread run(int n, int nz, long long t0, int expire, const std::vector<int>* given) {
  Thread t;
  int tile = 0, done_tiles = 0, inflight = 0;
  bool expired = false;
  std::vector<int> yslot(kYRing, -1), pslot(kSeg + 3, -1);        // last tile that reads a slot
  long long zz = t0 % nz;
  int pos = 0;
  std::vector<int> tpos;                                          // positions in their segments, by an own count
  for (int k = 0; k < n; ++k) {
    tpos.push_back(pos);
    pos = zz + 1 == nz || pos + 1 == kSeg ? 0 : pos + 1;
    zz = (zz + 1) % nz;
  }
  auto request = [&](const WgTile& w, int slot) {
    const int j = t.requested++;
    t.bad = t.bad || j >= n || w.z != (t0 + j) % nz || w.col != (t0 + j) / nz || w.pos != tpos[j] || slot != j % kYRing;
    ++inflight;
    if (expired) return;                                           // the sums of these slots are dropped
    t.bad = t.bad || yslot[slot] >= done_tiles;
    yslot[slot] = j;
    for (int s = w.pos == 0 ? 0 : w.pos + 2; s <= w.pos + 2; ++s) {
      t.bad = t.bad || pslot[s] >= done_tiles;                     // a tile that still reads it
      pslot[s] = -1;
    }
    for (int s = w.pos; s <= w.pos + 2; ++s) pslot[s] = j;
  };
  auto landed = [&](int younger) {
    t.bad = t.bad || younger < 0;
    inflight = younger < inflight ? younger : inflight;
  };
  auto all = [&](bool ok) -> bool {
    const size_t i = t.barriers.size();
    int r = ok;
    if (given != nullptr) {
      if (i < given->size()) r = (*given)[i];
      else { t.missing++; r = 0; }                                 // the other thread never comes
    }
    t.barriers.push_back(r);
    t.groups.push_back(inflight);
    return r != 0;
  };
  auto publish = [&](int k) { t.bad = t.bad || k != t.published || k >= t.requested; ++t.published; };
  auto bias = [&](int) {};
  auto done = [&](int slot, int phase) {
    const int k = tile++;
    t.bad = t.bad || slot != k % kYRing || phase != (k / kYRing) % 2;
    expired = expired || (expire >= 0 && k >= expire);
    if (expire >= 0 && k >= expire) return false;
    done_tiles = k + 1;
    return true;
  };
  auto drain = [&](bool ok) { t.drained += ok; };
  t.result = wgrad3_workers(n, nz, t0, request, landed, all, publish, bias, done, drain);
  return t;
}

int main() {
  int cases = 0;
  for (int nz : {1, 2, 3, 7, 8, 9, 16, 24})
    for (int n : {1, 2, 3, 4, 7, 8, 9, 17, 40})
      for (long long t0 = 0; t0 < 2 * nz; t0 += nz < 4 ? 1 : 3) {
        const Thread fine = run(n, nz, t0, -1, nullptr);
        if (fine.bad || !fine.result || fine.requested != n || fine.published != n || fine.drained != (n + kFlush - 1) / kFlush) {
          std::printf("schedule n %d nz %d t0 %lld\n", n, nz, t0);
          return 1;
        }
        for (int k = 0; k < n; ++k) {
          const Thread a = run(n, nz, t0, k, nullptr);               // its wait expires at tile k
          const Thread b = run(n, nz, t0, -1, &a.barriers);          // the same block, no wait of its own expires
          ++cases;
          if (a.result || b.result || b.missing || a.barriers != b.barriers || a.groups != b.groups || a.bad || b.bad) {
            std::printf("expired at %d: n %d nz %d t0 %lld, barriers %zu and %zu\n", k, n, nz, t0, a.barriers.size(),
                        b.barriers.size());
            return 1;
          }
        }
      }
  std::printf("%d cases\n", cases);
  return 0;
}
"""


def test_every_worker_passes_the_same_barriers_when_a_wait_expires(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host compiler")
    src = tmp_path / "model.cpp"
    src.write_text(MODEL)
    exe = tmp_path / "model"
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-I", CSRC, str(src), "-o", str(exe)], check=True, timeout=120)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
