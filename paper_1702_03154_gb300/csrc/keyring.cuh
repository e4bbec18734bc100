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

// Keys for one range a resident warp: a multiple of 16, a line of keys, so that
// a batch of a few hundred keys a warp spreads evenly, but 128 rather than 33 to
// 127: both slots then refill once and half the CTAs start (3e5 queries 14.3 us
// against 16.4, 4.5e5 16.4 against 17.7).  A grid of more than one wave only
// past 2^30 keys a warp.
inline unsigned ring_range(u64 n, u64 warps) {
  u64 csz = ((n + warps - 1) / warps + 15) & ~15ull;
  if (csz > 32 && csz < 128) csz = 128;
  return csz > 1ull << 30 ? 1u << 30 : (unsigned)csz;
}

}  // namespace bbh
