// keyring.cuh -- the shared-memory ring through which a lookup warp's keys
// arrive and its indices leave (lookup.cu, serve.cu).
#pragma once

#include "common.cuh"

namespace bbh {

// Ring of a warp: keys on their way in, keys in the slots, indices until their
// block of kBlock keys has retired.  The warp takes keys from all but the
// block that is still arriving.
static constexpr unsigned kRing = 512, kBlock = 64, kAhead = kRing - kBlock;
static constexpr unsigned kFlushAt = 5 * kBlock;  // look for a retired block past this many keys

__device__ __forceinline__ void key_async(u64 *smem_dst, const u64 *gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void key_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void key_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// How the n keys of a batch are dealt to the `warps` resident warps: turns of
// kChunk keys a warp, then one turn of `last` keys each.  A stretch of deep keys
// (absent ones, say) so falls to all warps alike: 1e8 queries whose first 1e7 are
// absent 1.11 ms (64-byte sectors 1.62) against 1.33 (2.20) with one range a warp.
// Up to two chunks a warp are one range each: a multiple of 16 keys, a line, so
// that a batch of a few hundred keys a warp spreads evenly, but 128 rather than
// 33 to 127: both slots then refill once and half the CTAs start (3e5 queries
// 14.3 us against 16.4, 4.5e5 16.4 against 17.7).
static constexpr unsigned kChunk = 2048;
struct RingShape {
  u64 n, turn;         // keys; keys of a turn, and what lies between two chunks of a warp
  unsigned cut, last;  // a warp's keys in full turns; in the last one
};
inline RingShape ring_shape(u64 n, u64 warps) {
  RingShape sh;
  sh.n = n;
  sh.turn = warps * kChunk;
  const u64 full = n <= 2 * sh.turn ? 0 : n / sh.turn;
  sh.cut = (unsigned)(full * kChunk);
  sh.last = (unsigned)(((n - full * sh.turn + warps - 1) / warps + 15) & ~15ull);
  if (!full && sh.last > 32 && sh.last < 128) sh.last = 128;
  return sh;
}
// CTAs of `per_cta` warps that have keys, of the `most` resident ones.
inline unsigned ring_grid(const RingShape &sh, unsigned per_cta, u64 most) {
  if (sh.cut) return (unsigned)most;
  return (unsigned)(((sh.n + sh.last - 1) / sh.last + per_cta - 1) / per_cta);
}

// One warp's part: `len` keys, the i-th of them at place(i) of the batch, those
// of a block of kBlock next to each other.
struct RingPart {
  u64 head, tail;  // place of the first key of its full turns, and of the last, less cut
  unsigned len;
  __host__ __device__ __forceinline__ RingPart(const RingShape &sh, unsigned warp)
      : head((u64)warp * kChunk) {
    const u64 full = (u64)(sh.cut / kChunk) * sh.turn, at = full + (u64)warp * sh.last;
    const u64 left = at < sh.n ? sh.n - at : 0;
    tail = at - sh.cut;
    len = sh.cut + (unsigned)(left < sh.last ? left : sh.last);
  }
  __host__ __device__ __forceinline__ u64 place(const RingShape &sh, unsigned i) const {
    return i < sh.cut ? head + (u64)(i / kChunk) * sh.turn + i % kChunk : tail + i;
  }
};

}  // namespace bbh
