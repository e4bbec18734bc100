// lookup.cu -- batched queries (Algorithm 3 with the minimal index of
// Sec. 2.2.3 and the ranks of Sec. 3.1).
//
// A key needs e^{1/gamma} level probes on average but up to L; a warp that
// kept 32 keys in lock-step would idle most lanes while its slowest key walks
// down the levels.  Instead every lane owns two independent query slots, each
// with its own (key, output index, level).  Each round every active slot
// probes its current level with one load of the record holding its bit (a
// 256-bit sector or an 8-byte unit, sector.cuh: the A word and a count of the
// ones before it come together); a slot whose bit is set finishes its rank
// from those registers and retires, the others move to the next level, and
// retired slots are refilled from the warp's range of input keys.  So lanes
// stay busy, each lane keeps two independent loads in flight, and a placed
// key costs one memory request per level probed.
//
// What bounds it: the probes' latency and rate at the L2 (about half of the 312
// G/s that nothing but loads reaches), or HBM's random-access rate beyond it.
// So nothing else may wait or scatter: a warp's keys arrive in a ring in shared
// memory by asynchronous copies ahead of the slots, the indices replace them
// there and leave in input order, a block of 64 at a time, once every key of
// the block has retired.  Measured, with the ring and with each key loaded when
// its slot is refilled and each index stored when its key retires: 1e8 queries of
// a 2e9-key function 3.64 / 3.70 ms, of a function in L2 1.03 / 1.06, with a
// tenth of absent keys 1.21 / 1.14 (a deep key holds its block back), 3e7 queries
// at gamma 1 0.49 / 0.55, in 64-byte sectors 0.72 / 0.83.
#include <cuda_runtime.h>
#include <stdlib.h>

#include "common.cuh"
#include "keyring.cuh"
#include "sector.cuh"

namespace bbh {

static constexpr int kLookupThreads = 256;

struct LevelTable {
  u64 s[MPHF_MAX_LEVELS];
  u64 m[MPHF_MAX_LEVELS];
  u64 off[MPHF_MAX_LEVELS];
};

struct LookupArgs {
  const unsigned *S;  // sectors: A with its ranks
  const u64 *SB;      // ones before each superblock
  const u64 *fb;
  u64 n_fb;
  u64 N;
  uint32_t L_used;
};

__device__ __forceinline__ u64 fallback_index(const LookupArgs &a, u64 x) {
  u64 lo = 0, hi = a.n_fb;
  while (lo < hi) {
    u64 mid = lo + ((hi - lo) >> 1);
    if (__ldg(a.fb + mid) < x) lo = mid + 1;
    else hi = mid;
  }
  if (lo < a.n_fb && __ldg(a.fb + lo) == x) return a.N - a.n_fb + lo;
  return MPHF_NOT_FOUND;
}

static constexpr int kLookupWarps = kLookupThreads / 32;
// kNarrow: every m_d < 2^32 and A short enough that bit g's word index
// g >> kQShift is below 2^32 (A below 2^36 bits); then a probe's position
// arithmetic is 32-bit: with off_d a multiple of 64,
//   g >> kQShift = (off_d >> kQShift) + (p >> kQShift),  g & mask = p & mask.
template <int W, bool kNarrow>
__global__ void __launch_bounds__(kLookupThreads, W == 15 ? 3 : 4)
k_lookup(const u64 *__restrict__ keys, RingShape sh, u64 *__restrict__ out, LookupArgs a,
         LevelTable t) {
  using LW = Lay<W>;
  __shared__ u64 ts[MPHF_MAX_LEVELS], tm[MPHF_MAX_LEVELS], toff[MPHF_MAX_LEVELS];
  __shared__ unsigned tm32[MPHF_MAX_LEVELS], toq[MPHF_MAX_LEVELS];
  __shared__ u64 rings[kLookupWarps][kRing];
  for (unsigned i = threadIdx.x; i < a.L_used; i += kLookupThreads) {
    ts[i] = t.s[i];
    tm[i] = t.m[i];
    toff[i] = t.off[i];
    tm32[i] = (unsigned)t.m[i];
    toq[i] = (unsigned)(t.off[i] >> LW::kQShift);
  }
  __syncthreads();

  const unsigned lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  u64 *ring = rings[threadIdx.x >> 5];
  const RingPart mine(sh, (blockIdx.x * kLookupThreads + threadIdx.x) >> 5);
  const unsigned len = mine.len;
  if (!len) return;
  unsigned cur = 0;   // keys taken
  unsigned base = 0;  // keys whose indices have left the ring
  // keys [i0, i0 + 64) of the warp's part into the ring
  auto fetch = [&](unsigned i0) {
    const u64 *src = keys + mine.place(sh, i0);
#pragma unroll
    for (unsigned u = lane; u < kBlock; u += 32)
      if (i0 + u < len) key_async(ring + ((i0 + u) & (kRing - 1)), src + u);
    key_commit();
  };
  for (unsigned i = 0; i < min(len, kRing); i += kBlock) fetch(i);
  key_wait<0>();
  __syncwarp();
  u64 x[2] = {0, 0};
  unsigned idx[2] = {0, 0}, lvl[2] = {0, 0};
  bool act[2] = {false, false};
  for (;;) {
    // refill retired slots, slot 0 first, lane by lane
    const unsigned avail = min(len, base + kAhead) - cur;
    const unsigned need0 = __ballot_sync(0xffffffffu, !act[0]);
    const unsigned need1 = __ballot_sync(0xffffffffu, !act[1]);
    const unsigned rk[2] = {(unsigned)__popc(need0 & lt),
                            (unsigned)(__popc(need0) + __popc(need1 & lt))};
#pragma unroll
    for (int s = 0; s < 2; s++) {
      if (!act[s] && rk[s] < avail) {
        idx[s] = cur + rk[s];
        x[s] = ring[idx[s] & (kRing - 1)];
        lvl[s] = 0;
        act[s] = true;
      }
    }
    cur += min((unsigned)(__popc(need0) + __popc(need1)), avail);
    // the oldest block leaves once its keys have retired; its place goes to
    // the keys that follow the ring's
    if (cur - base >= kFlushAt || cur == len) {
      const unsigned end = min(base + kBlock, len);
      const bool old = (act[0] && idx[0] < end) || (act[1] && idx[1] < end);
      if (!__any_sync(0xffffffffu, old)) {
        u64 *dst = out + mine.place(sh, base) + lane;
        __syncwarp();
#pragma unroll
        for (unsigned u = 0; u < kBlock; u += 32) {
          const unsigned i = base + u + lane;
          if (i < end) __stcs(dst + u, ring[i & (kRing - 1)]);
        }
        fetch(base + kRing);
        key_wait<1>();
        __syncwarp();
        base = end;
        if (base == len) break;
      }
    }

    // one probe per active slot: issue all loads, then resolve
    typename LW::Pos p[2];
    typename LW::Data v[2];
#pragma unroll
    for (int s = 0; s < 2; s++) {
      if (act[s]) {
        const unsigned d = lvl[s];
        if (kNarrow) {
          const unsigned pd = reduce_range32(mix64(x[s] ^ ts[d]), tm32[d]);
          p[s] = LW::pos_q(toq[d] + (pd >> LW::kQShift), pd & ((1u << LW::kQShift) - 1u));
        } else {
          p[s] = LW::pos(toff[d] + level_pos(x[s], ts[d], tm[d]));
        }
        v[s] = LW::load(a.S, p[s]);
      }
    }
#pragma unroll
    for (int s = 0; s < 2; s++) {
      if (act[s]) {
        unsigned w = 0;
        if (LW::hit(v[s], p[s], w)) {
          ring[idx[s] & (kRing - 1)] = LW::rank(v[s], p[s], w, a.SB);
          act[s] = false;
        } else if (++lvl[s] >= a.L_used) {
          ring[idx[s] & (kRing - 1)] = a.n_fb ? fallback_index(a, x[s]) : MPHF_NOT_FOUND;
          act[s] = false;
        }
      }
    }
  }
}

// Without a ring: each slot loads its next key itself and stores its index when
// its key retires; warps take chunks of csz keys in a fixed order.  For
//  - 8-byte units: their probes are ordinary cached loads that lean on a large L1
//    for the requests in flight, and the rings' 128 KB of shared memory a
//    multiprocessor leave little of it: 1e8 queries of a function in L2 1.01 ms,
//    1.52 with the ring;
//  - 32-byte sectors where a warp has 128 to 1024 keys: the ring's first 512 keys
//    would arrive before the first probe, and it leaves block by block at the end.
//    8e5 queries of a 3e7-key function 21.0 us (22.8 with the ring), 2.5e6 40.3
//    (42.0), 3e6 at gamma 5 34.2 (36.0), with 5% absent keys 44.3 (50.4); below
//    and above that range the ring is as fast or faster (5e5 18.7 / 18.6, 6e6
//    77.1 / 76.4 us).
template <int W, bool kNarrow>
__global__ void __launch_bounds__(kLookupThreads)
k_lookup_direct(const u64 *__restrict__ keys, u64 n, u64 csz, u64 *__restrict__ out, LookupArgs a,
                LevelTable t) {
  using LW = Lay<W>;
  __shared__ u64 ts[MPHF_MAX_LEVELS], tm[MPHF_MAX_LEVELS], toff[MPHF_MAX_LEVELS];
  __shared__ unsigned tm32[MPHF_MAX_LEVELS], toq[MPHF_MAX_LEVELS];
  for (unsigned i = threadIdx.x; i < a.L_used; i += kLookupThreads) {
    ts[i] = t.s[i];
    tm[i] = t.m[i];
    toff[i] = t.off[i];
    tm32[i] = (unsigned)t.m[i];
    toq[i] = (unsigned)(t.off[i] >> LW::kQShift);
  }
  __syncthreads();

  const unsigned lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const u64 nchunks = (n + csz - 1) / csz;
  const u64 warp_id = ((u64)blockIdx.x * kLookupThreads + threadIdx.x) >> 5;
  const u64 nwarps = ((u64)gridDim.x * kLookupThreads) >> 5;
  u64 chunk = warp_id;
  u64 cursor = chunk * csz;
  u64 cend = chunk < nchunks ? min(cursor + csz, n) : cursor;
  bool more = chunk < nchunks;

  u64 x[2], idx[2];
  unsigned lvl[2];
  bool act[2];
#pragma unroll
  for (int s = 0; s < 2; s++) {
    act[s] = false;
    lvl[s] = 0;
    x[s] = 0;
    idx[s] = 0;
  }

  for (;;) {
    // refill retired slots from the warp's input stream (warp-uniform
    // control); while the current chunk holds a key for every free slot they
    // are ranked lane by lane, slot 0 first, and filled in one pass
    unsigned rk[2], nfree = 0;
#pragma unroll
    for (int s = 0; s < 2; s++) {
      const unsigned need = __ballot_sync(0xffffffffu, !act[s]);
      rk[s] = nfree + __popc(need & lt);
      nfree += __popc(need);
    }
    if (nfree && cend - cursor >= nfree) {
#pragma unroll
      for (int s = 0; s < 2; s++) {
        if (!act[s]) {
          const u64 i = cursor + rk[s];
          idx[s] = i;
          x[s] = __ldcs(keys + i);
          lvl[s] = 0;
          act[s] = true;
        }
      }
      cursor += nfree;
    }
#pragma unroll
    for (int s = 0; s < 2; s++) {
      unsigned need = __ballot_sync(0xffffffffu, !act[s]);
      while (need && more) {
        if (cursor >= cend) {
          chunk += nwarps;
          if (chunk >= nchunks) {
            more = false;
            break;
          }
          cursor = chunk * csz;
          cend = min(cursor + csz, n);
        }
        const u64 avail = cend - cursor;
        const unsigned r = __popc(need & lt);
        const bool mine = ((need >> lane) & 1u) && (u64)r < avail;
        if (mine) {
          idx[s] = cursor + r;
          x[s] = __ldcs(keys + cursor + r);
          lvl[s] = 0;
          act[s] = true;
        }
        const unsigned taken = __ballot_sync(0xffffffffu, mine);
        need &= ~taken;
        cursor += __popc(taken);
      }
    }
    bool any = false;
#pragma unroll
    for (int s = 0; s < 2; s++) any |= act[s];
    if (!__any_sync(0xffffffffu, any)) break;

    // one probe per active slot: issue all loads, then resolve
    typename LW::Pos p[2];
    typename LW::Data v[2];
#pragma unroll
    for (int s = 0; s < 2; s++) {
      if (act[s]) {
        const unsigned d = lvl[s];
        if (kNarrow) {
          const unsigned pd = reduce_range32(mix64(x[s] ^ ts[d]), tm32[d]);
          p[s] = LW::pos_q(toq[d] + (pd >> LW::kQShift), pd & ((1u << LW::kQShift) - 1u));
        } else {
          p[s] = LW::pos(toff[d] + level_pos(x[s], ts[d], tm[d]));
        }
        v[s] = LW::load(a.S, p[s]);
      }
    }
#pragma unroll
    for (int s = 0; s < 2; s++) {
      if (act[s]) {
        unsigned w = 0;
        if (LW::hit(v[s], p[s], w)) {
          __stcs(out + idx[s], LW::rank(v[s], p[s], w, a.SB));
          act[s] = false;
        } else if (++lvl[s] >= a.L_used) {
          __stcs(out + idx[s], a.n_fb ? fallback_index(a, x[s]) : MPHF_NOT_FOUND);
          act[s] = false;
        }
      }
    }
  }
}

static void fill_tables(const mphf_t *h, LookupArgs &a, LevelTable &t) {
  a.S = (const unsigned *)h->S.p;
  a.SB = (const u64 *)h->SB.p;
  a.fb = (const u64 *)h->fb.p;
  a.n_fb = h->n_fb;
  a.N = h->N;
  a.L_used = h->L_used;
  for (uint32_t d = 0; d < MPHF_MAX_LEVELS; d++) {
    t.s[d] = d < h->L_used ? h->s[d] : 0;
    t.m[d] = d < h->L_used ? h->m[d] : 0;
    t.off[d] = d < h->L_used ? h->off[d] : 0;
  }
}

template <int W, bool NARROW>
static int launch_lookup(const u64 *keys, u64 n, u64 *out, const LookupArgs &a,
                         const LevelTable &t, cudaStream_t s) {
  static unsigned mb_dev[64] = {0};  // resident CTAs, per device
  unsigned &mb = mb_dev[cur_device()];
  if (!mb) mb = resident_grid(k_lookup<W, NARROW>, kLookupThreads, 0);
  const RingShape sh = ring_shape(n, (u64)mb * kLookupWarps);
  LaunchScope ls("lookup", s);
  k_lookup<W, NARROW><<<ring_grid(sh, kLookupWarps, mb), kLookupThreads, 0, s>>>(keys, sh, out, a,
                                                                                 t);
  MPHF_CUDA(cudaGetLastError());
  return MPHF_OK;
}

template <int W, bool NARROW>
static int launch_lookup_direct(const u64 *keys, u64 n, u64 *out, const LookupArgs &a,
                                const LevelTable &t, cudaStream_t s) {
  // one wave of resident CTAs: a second would only start after the first has
  // drained
  static unsigned mb_dev[64] = {0};  // per device
  unsigned &mb = mb_dev[cur_device()];
  if (!mb) mb = resident_grid(k_lookup_direct<W, NARROW>, kLookupThreads, 0);
  const u64 warps = (u64)mb * kLookupWarps;
  // sectors: two chunks a warp, so that a stretch of deep keys does not fall to
  // a few warps alone (3e6 queries, the first tenth absent: 50.6 us, 62.1 in one)
  const u64 csz = W == (int)kUnitBits ? lookup_chunk(n, warps)
                                      : ((n + 2 * warps - 1) / (2 * warps) + 15) & ~15ull;
  const u64 grid = ((n + csz - 1) / csz + kLookupWarps - 1) / kLookupWarps;
  LaunchScope ls("lookup", s);
  k_lookup_direct<W, NARROW><<<(unsigned)(grid > mb ? mb : grid), kLookupThreads, 0, s>>>(
      keys, n, csz, out, a, t);
  MPHF_CUDA(cudaGetLastError());
  return MPHF_OK;
}

// A batch of 32-byte sector lookups that is better without the ring.
static bool better_direct(u64 n) {
  const u64 warps = (u64)sm_count() * 4 * kLookupWarps;
  return n > 128 * warps && n <= 1024 * warps;
}

int lookup_impl(const mphf_t *h, const u64 *keys, u64 n, u64 *out, cudaStream_t s) {
  LookupArgs a;
  LevelTable t;
  fill_tables(h, a, t);
  const bool narrow = narrow_positions(h);
  if (h->sw == kSectWordsMini)
    return narrow ? launch_lookup<kSectWordsMini, true>(keys, n, out, a, t, s)
                  : launch_lookup<kSectWordsMini, false>(keys, n, out, a, t, s);
  if (h->sw == kUnitBits)
    return narrow ? launch_lookup_direct<(int)kUnitBits, true>(keys, n, out, a, t, s)
                  : launch_lookup_direct<(int)kUnitBits, false>(keys, n, out, a, t, s);
  if (better_direct(n))
    return narrow ? launch_lookup_direct<kSectWords, true>(keys, n, out, a, t, s)
                  : launch_lookup_direct<kSectWords, false>(keys, n, out, a, t, s);
  return narrow ? launch_lookup<kSectWords, true>(keys, n, out, a, t, s)
                : launch_lookup<kSectWords, false>(keys, n, out, a, t, s);
}

}  // namespace bbh

int bbh::g_lookup_wide = 0;

using namespace bbh;

extern "C" int mphf_debug_lookup_wide(int on) {
  g_lookup_wide = on ? 1 : 0;
  return MPHF_OK;
}

extern "C" int mphf_lookup(const mphf_t *h, const uint64_t *d_keys, uint64_t n, uint64_t *d_out,
                           void *stream) {
  if (!h) return MPHF_EINVAL;
  if (n == 0) return MPHF_OK;
  if (!d_keys || !d_out || (((uintptr_t)d_keys | (uintptr_t)d_out) & 7)) return MPHF_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  if (h->L_used == 0 && h->n_fb == 0) {  // empty function: every key is a miss
    MPHF_CUDA(cudaMemsetAsync(d_out, 0xff, n * 8, s));
    return MPHF_OK;
  }
  return lookup_impl(h, (const u64 *)d_keys, n, (u64 *)d_out, s);
}

// Large batches run as a three-stage pipeline over chunks of the batch: the
// copy in of chunk c+1 (side stream ci), the lookup of chunk c (the caller's
// stream) and the copy out of chunk c-1 (side stream co) overlap, so the
// batch costs about one pass over the host link instead of two plus the
// kernel.  The D2H copy of chunk c is enqueued after the lookup of chunk c+1,
// so that a pageable h_out (whose copy blocks the host) still leaves the next
// lookup queued.
extern "C" int mphf_lookup_host(const mphf_t *h, const uint64_t *h_keys, uint64_t n,
                                uint64_t *h_out, void *stream) {
  if (!h) return MPHF_EINVAL;
  if (n == 0) return MPHF_OK;
  if (!h_keys || !h_out) return MPHF_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  DevBuf kb, ob;
  int rc = dev_alloc(kb, n * 8, s);
  if (rc != MPHF_OK) return rc;
  rc = dev_alloc(ob, n * 8, s);
  if (rc != MPHF_OK) {
    dev_free(kb, s);
    return rc;
  }
  const u64 chunk = feed_chunk(n);
  cudaError_t e = cudaSuccess;
  if (!chunk) {
    e = cudaMemcpyAsync(kb.p, h_keys, n * 8, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) {
      rc = mphf_lookup(h, (const uint64_t *)kb.p, n, (uint64_t *)ob.p, stream);
      if (rc == MPHF_OK) e = cudaMemcpyAsync(h_out, ob.p, n * 8, cudaMemcpyDeviceToHost, s);
    }
  } else {
    SideSet ss;
    rc = side_set(2, &ss);
    if (rc != MPHF_OK) {
      dev_free(kb, s);
      dev_free(ob, s);
      return rc;
    }
    cudaStream_t ci = ss.s[0], co = ss.s[1];
    cudaEvent_t ev_in = ss.ev[0], ev_k = ss.ev[1];
    u64 *dk = (u64 *)kb.p, *dout = (u64 *)ob.p;
    // both buffers were allocated in s's order: the side streams start after
    e = cudaEventRecord(ev_in, s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(ci, ev_in, 0);
    u64 prev0 = 0, prevn = 0;  // chunk whose copy out is still to be enqueued
    for (u64 c0 = 0; c0 < n && e == cudaSuccess && rc == MPHF_OK; c0 += chunk) {
      const u64 cn = n - c0 < chunk ? n - c0 : chunk;
      e = cudaMemcpyAsync(dk + c0, (const u64 *)h_keys + c0, cn * 8, cudaMemcpyHostToDevice, ci);
      if (e == cudaSuccess) e = cudaEventRecord(ev_in, ci);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(s, ev_in, 0);
      if (e != cudaSuccess) break;
      rc = mphf_lookup(h, (const uint64_t *)(dk + c0), cn, (uint64_t *)(dout + c0), stream);
      if (rc != MPHF_OK) break;
      e = cudaEventRecord(ev_k, s);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(co, ev_k, 0);
      if (e == cudaSuccess && prevn)
        e = cudaMemcpyAsync((u64 *)h_out + prev0, dout + prev0, prevn * 8, cudaMemcpyDeviceToHost, co);
      prev0 = c0;
      prevn = cn;
    }
    if (e == cudaSuccess && rc == MPHF_OK && prevn)
      e = cudaMemcpyAsync((u64 *)h_out + prev0, dout + prev0, prevn * 8, cudaMemcpyDeviceToHost, co);
    // everything enqueued on the side streams is ordered before the frees
    cudaEventRecord(ev_in, ci);
    cudaStreamWaitEvent(s, ev_in, 0);
    cudaEventRecord(ev_k, co);
    cudaStreamWaitEvent(s, ev_k, 0);
  }
  dev_free(kb, s);
  dev_free(ob, s);
  cudaError_t e2 = cudaStreamSynchronize(s);
  if (e == cudaSuccess) e = e2;
  if (e != cudaSuccess) return cuda_fail(e, "mphf_lookup_host");
  return rc;
}
