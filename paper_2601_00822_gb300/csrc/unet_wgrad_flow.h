// The control flow of k_wgrad3's worker threads (unet_wgrad.cu) apart from what its steps
// do: which tile is requested when, and which barriers a thread passes.  It names no
// device feature, so that it also compiles for the host, where a test checks the barrier
// counts of threads whose waits end differently.
#pragma once

#ifdef __CUDACC__
#define BFCS_FLOW __host__ __device__ __forceinline__
#else
#define BFCS_FLOW inline
#endif

namespace bfcs {
namespace net {

constexpr int kSeg = 8;                               // tiles per staged segment
constexpr int kYRing = 3;
constexpr int kFlush = 8;                             // tiles per accumulation in tensor memory

// position of the tile after one at plane z in its segment: segments end after kSeg tiles
// or with the column
BFCS_FLOW int wg_next_pos(int z, int nz, int pos) { return z + 1 == nz || pos + 1 == kSeg ? 0 : pos + 1; }

// Tile j's loads: at the start of a segment three planes, else one, and its dY; one
// copy group each.  They are requested up to three tiles ahead (two copies in flight
// under two tiles' MMAs: one tile ahead left the pass to the copies' latency, 4600
// clocks a tile), but not before the last reader of their slots is done: dY slot j % 3
// was read by tile j - 3, plane slot p + 2 of segment position p (and 0 and 1 for p =
// 0) last by position min(p + 2, L - 1) of the segment before, of length L.
struct WgTile { int col, z, pos, prev; };   // prev: length of the segment before (0: none)
BFCS_FLOW WgTile wg_after(WgTile t, int nz) {
  WgTile u;
  u.pos = wg_next_pos(t.z, nz, t.pos);
  u.z = t.z + 1 == nz ? 0 : t.z + 1;
  u.col = t.z + 1 == nz ? t.col + 1 : t.col;
  u.prev = u.pos == 0 ? t.pos + 1 : t.prev;
  return u;
}
BFCS_FLOW int wg_last_reader(WgTile t, int j) {
  const int p = t.pos + 2 < t.prev - 1 ? t.pos + 2 : t.prev - 1;
  return t.prev == 0 ? -1 : j - t.pos - t.prev + p;
}

// Tiles t0 .. t0 + n - 1 (n >= 1; z fastest, nz planes a column).  The steps:
//   request(tile, slot)  the tile's copies into dY slot `slot`, one copy group
//   landed(younger)      waits for all of this thread's copy groups but the `younger` last ones
//   all(ok)              barrier of the worker threads; whether ok held in all of them
//   publish(k)           tile k's operands are staged
//   bias(slot)           reads the dY in a slot
//   done(slot, phase)    wait for the MMAs of the tile in that slot; false once it expired
//   drain(ok)            adds the accumulators to the running sums
// Every thread passes the same barriers, also when its own wait expires and another's does
// not: what is requested (and so whether a tile was requested early, which decides the
// number of barriers of the next iteration) depends on n, nz and t0 alone.  After an
// expired wait the copies go on, from valid addresses into slots whose sums are dropped,
// until all threads leave, two barriers later at most.  Returns whether no wait expired in
// any thread.
template <class Request, class Landed, class All, class Publish, class Bias, class Done, class Drain>
BFCS_FLOW bool wgrad3_workers(int n, int nz, long long t0, Request request, Landed landed, All all, Publish publish,
                              Bias bias, Done done, Drain drain) {
  WgTile nt;                                          // next tile to request, number `next`
  nt.col = (int)(t0 / nz);
  nt.z = (int)(t0 % nz);
  nt.pos = nt.prev = 0;
  int next = 0;
  auto ask = [&] {
    request(nt, next % kYRing);
    nt = wg_after(nt, nz);
    ++next;
  };
  while (next < n && next < kYRing && wg_last_reader(nt, next) < 0) ask();
  landed(next - 1);
  bool ok = all(true);
  publish(0);
  bias(0);
  for (int k = 0; k < n; ++k) {
    const bool more = k + 1 < n, early = more && next > k + 1;
    const int ring = k % kYRing, ring1 = (k + 1) % kYRing;
    if (early) {                                      // tile k + 1, requested before
      landed(next - 2 - k);
      ok = all(ok);
      if (!ok) break;
      publish(k + 1);
      bias(ring1);
    }
    ok = done(ring, k / kYRing & 1) && ok;
    if (!more || (k + 1) % kFlush == 0) drain(ok);    // the next tile's MMAs wait for this
    // every thread has read the dY slots that are requested below (a step without the
    // barrier above needs one here)
    if (more && !early) ok = all(ok);
    while (next < n && next <= k + kYRing && wg_last_reader(nt, next) <= k) ask();
    if (more && !early) {
      landed(next - 2 - k);
      ok = all(ok);
      if (!ok) break;
      publish(k + 1);
      bias(ring1);
    }
  }
  landed(0);
  return all(ok);
}

}  // namespace net
}  // namespace bfcs
