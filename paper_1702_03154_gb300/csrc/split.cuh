// split.cuh -- write-combining multisplit: keys hashed to their level value
// and written to position buckets in full aligned runs.
#pragma once

#include "common.cuh"

namespace bbh {

// Inverse of mix64 (each xor-shift undone by its own series, each odd factor
// by its inverse modulo 2^64), so that a level's hash value stands for its
// key: x = unmix64(h_d(x)) ^ s_d.
__host__ __device__ __forceinline__ u64 unmix64(u64 z) {
  z = (z ^ (z >> 31) ^ (z >> 62)) * 0x319642B2D24D8EC3ull;
  z = (z ^ (z >> 27) ^ (z >> 54)) * 0x96DE1B173F119089ull;
  return z ^ (z >> 30) ^ (z >> 60);
}

// ---------------------------------------------------------------------------
// One CTA's share of a multisplit of n values.  Every destination has a ring
// of at least two quanta of 2^lq slots in shared memory.  A round pushes one tile: a
// value takes the next slot of its destination with one shared atomic and is
// stored there.  Then each destination that holds whole quanta has
// them reserved (one global atomic, by the lane that owns the destination) and
// written out by groups of 2^lq lanes of the same warp: runs that start on a
// quantum boundary of the bucket, so a bucket is filled by whole 128-byte
// lines (lq = 4; 64 bytes beyond ~780 destinations).  Nothing is scanned,
// sorted or tagged: a value costs one shared atomic, one store and one load,
// and a round two block barriers.
//
// A value whose ring is full goes to a short spill list instead (and, past
// its end, straight to its bucket); the list is written at the end.  The
// round length is chosen for rings that rarely fill.  The next tile is loaded
// (from L2: it was prefetched a round earlier) and hashed while the
// reservations are in flight.
//
// A bucket that overflows raises the status and is still filled to its end, so
// a reader that takes min(counter, cap) values never meets a slot of another
// bucket or of an earlier launch.
//
// Measured (1e8 values, hashed): 763 destinations 0.46 ms, 180 destinations
// 0.40 ms (16 bytes a value: 3.5 - 4.0 TB/s); of those 0.46 ms the shared
// atomics cost 0.11, the copies 0.08, the global atomics 0.08, the ring stores
// 0.04 (each left out in turn).  The counting-sort multisplit took 0.89 ms.
// ---------------------------------------------------------------------------
static constexpr int kWT = 1024;          // threads of a split CTA (or half as many)
static constexpr unsigned kWMaxNb = 2048; // destinations at most
static constexpr unsigned kWSpill = 512;  // entries of the spill list (at most a CTA's threads)
// shared memory of a CTA when `per_sm` of them share a multiprocessor
__host__ __device__ constexpr unsigned wc_smem(unsigned per_sm) {
  return (228u * 1024 / per_sm - 1024) & ~15u;
}

// A queued run: 2^lq ring entries from shared-memory byte `src` to global `dst`.
struct WcJob {
  unsigned src, count;
  u64 *dst;
};

struct WcShape {
  unsigned nb, ls, lq;
  unsigned per;  // destinations a warp owns
  unsigned nt, smem;  // threads and shared memory of the CTA
};

__host__ __device__ inline u64 wc_smem_bytes(const WcShape &s) {
  return (u64)(s.nt / 32) * (s.per << (s.ls - s.lq)) * sizeof(WcJob) +
         (((u64)s.nb << s.ls) + kWSpill) * 8 + (u64)s.nb * 4 + 16;
}

// Ring and quantum sizes for nb destinations: the largest ring that fits (at
// most 2048 slots), of two quanta or of quanta of a warp's 32 lanes.
__host__ __device__ inline WcShape wc_shape(unsigned nb, unsigned nt, unsigned smem) {
  WcShape s;
  s.nb = nb;
  s.nt = nt;
  s.smem = smem;
  s.per = (nb + nt / 32 - 1) / (nt / 32);
  for (s.ls = 11;; s.ls--) {
    s.lq = s.ls - 1 < 5 ? s.ls - 1 : 5;
    if (s.ls == 3 || wc_smem_bytes(s) <= smem) return s;
  }
}

// Values per thread and round: all the CTA has if that is little, and at most
// what fills three eighths of the rings (a ring rarely overflows then): one of
// 8, 6, 4, 2, 1.  0: so few destinations that a round takes less than one
// value per thread.
__host__ __device__ inline unsigned wc_round(const WcShape &s, u64 n, unsigned ctas) {
  const unsigned fill = (s.nb << s.ls) * 3 / 8 / s.nt;
  const u64 have = (n + (u64)ctas * s.nt - 1) / ((u64)ctas * s.nt);
  const u64 k = fill < have ? fill : have;
  return k >= 8 ? 8u : k >= 6 ? 6u : k >= 4 ? 4u : k >= 2 ? 2u : (unsigned)k;
}

// Threads of a CTA for nb destinations: two CTAs of 512 a multiprocessor where
// rings of half the memory still take eight values per thread and round (the
// phases of one overlap those of the other), one CTA of 1024 elsewhere.
// Measured on 1e8 hashed keys: 180 destinations 403 us against 456, 360 440
// against 456, but 128 442 against 442 and 512 508 against 504.
inline int wc_threads(unsigned nb) {
  const WcShape s = wc_shape(nb, kWT / 2, wc_smem(2));
  return nb <= (unsigned)kWT / 2 && wc_smem_bytes(s) <= s.smem &&
                 (nb << s.ls) * 3 / 8 / s.nt >= 8 ? kWT / 2 : kWT;
}

// The first n of a ring's entries to dst (a call: inlined, its registers cost the
// rounds 1.3% of a build of 3e9 keys).
__device__ __noinline__ static void wc_fill_end(const u64 *ring, unsigned head, unsigned mask,
                                                u64 *dst, u64 n) {
  for (unsigned e = 0; e < n; e++) dst[e] = ring[(head + e) & mask];
}

// The rounds of wc_split with KR values per thread and a tile of `tile` (at
// most KR NT) values.
template <int NT, int OWN, int KR, class Key, class Dst, class Dest>
__device__ __forceinline__ void wc_rounds(const u64 *__restrict__ in, u64 n, unsigned rank,
                                          unsigned ranks, unsigned tile, const WcShape &sh,
                                          unsigned char *smem, const Key &key, const Dst &dst,
                                          const Dest &dest, u64 *__restrict__ arena,
                                          unsigned *__restrict__ status) {
  static_assert(NT >= (int)kWSpill, "one spilled value per thread goes back to the rings");
  const unsigned nb = sh.nb, ls = sh.ls, lq = sh.lq, per = sh.per;
  const unsigned njw = per << (ls - lq);  // runs a warp can have queued
  const unsigned S = 1u << ls, Q = 1u << lq;
  const unsigned tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, lt = (1u << lane) - 1u;
  WcJob *jobs = reinterpret_cast<WcJob *>(smem) + warp * njw;  // this warp's queue
  const unsigned buf0 = (NT / 32) * njw * (unsigned)sizeof(WcJob);
  u64 *buf = reinterpret_cast<u64 *>(smem + buf0);
  u64 *spill = buf + ((u64)nb << ls);
  // per destination: (entries in the ring << 16) | tail; both only grow in a
  // round, the owner brings the tail back below S and takes the entries out
  unsigned *cnt = reinterpret_cast<unsigned *>(spill + kWSpill);
  unsigned *nspill = cnt + nb;
  for (unsigned i = tid; i < nb; i += NT) cnt[i] = 0;
  if (tid == 0) *nspill = 0;
  const u64 step = (u64)ranks * tile;
  u64 t0 = (u64)rank * tile;
  const unsigned full = S << 16;
  u64 y[KR] = {};  // inputs, then their stored values
  unsigned b[KR];  // destination
  // values of the tile at `at` that exist for this thread (k < that number)
  auto mine = [&](u64 at) -> unsigned {
    if (at >= n) return 0;
    const unsigned len = at + tile <= n ? tile : (unsigned)(n - at);
    return len == KR * NT ? KR : len > tid ? (len - tid + NT - 1) / NT : 0;
  };
  auto load = [&](u64 at, unsigned have) {
    const u64 *p = in + at + tid;
#pragma unroll
    for (int k = 0; k < KR; k++)
      if ((unsigned)k < have) y[k] = __ldcs(p + k * NT);
  };
  // the tile at `at` into L2, so that its loads a round later are short
  auto prefetch = [&](u64 at) {
    if (tid == 0 && at + tile <= n) {
      const uintptr_t p = ((uintptr_t)(in + at) + 15) & ~(uintptr_t)15;
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(tile * 8 - 16));
    }
  };
  auto hash = [&]() {  // values that do not exist are hashed too and not pushed
#pragma unroll
    for (int k = 0; k < KR; k++) {
      y[k] = key(y[k]);
      b[k] = dst(y[k]);
    }
  };
  const unsigned l = lane & (Q - 1), ng = 32u >> lq;
  auto move = [&](const WcJob &j) {
    j.dst[l] = *reinterpret_cast<const u64 *>(smem + j.src + 8 * l);
  };
  // write this warp's first nj queued runs: a group of Q lanes per run
  auto copy = [&](unsigned nj) {
    unsigned j = lane >> lq;
    for (; j + 3 * ng < nj; j += 4 * ng) {
      const WcJob a0 = jobs[j], a1 = jobs[j + ng], a2 = jobs[j + 2 * ng], a3 = jobs[j + 3 * ng];
      move(a0);
      move(a1);
      move(a2);
      move(a3);
    }
    for (; j < nj; j += ng) move(jobs[j]);
  };
  // a single value straight to its bucket; lanes with the same destination
  // share one reservation (keys that arrive in position order fill one ring
  // at a time, and most of them come this way)
  auto one = [&](u64 yy, unsigned bb) {
    const unsigned act = __activemask(), same = __match_any_sync(act, bb);
    const DestRun r = dest(bb);
    u64 g = 0;
    if (!(same & lt)) g = atomicAdd(r.counter, (u64)__popc(same));
    g = __shfl_sync(act, g, __ffs(same) - 1) + __popc(same & lt);
    if (g < r.cap) arena[r.base + g] = yy;
    else atomicOr(status, 1u);
  };
  auto spilled = [&](u64 yy, unsigned bb) {
    unsigned j = kWSpill;
    if (*(volatile unsigned *)nspill < kWSpill) j = atomicAdd(nspill, 1u);
    if (j < kWSpill) spill[j] = yy;
    else one(yy, bb);
  };
  auto push = [&](unsigned have) {
    unsigned c[KR], over = 0;
#pragma unroll
    for (int k = 0; k < KR; k++) {
      c[k] = 0;
      if ((unsigned)k < have) c[k] = atomicAdd(cnt + b[k], 0x10001u);
    }
#pragma unroll
    for (int k = 0; k < KR; k++) {
      if ((unsigned)k < have && c[k] < full) buf[(b[k] << ls) + (c[k] & (S - 1))] = y[k];
      over |= c[k] < full ? 0u : 1u << k;
    }
    if (over) {
#pragma unroll
      for (int k = 0; k < KR; k++)
        if ((over >> k) & 1u) spilled(y[k], b[k]);
    }
  };
  unsigned have = mine(t0);
  load(t0, have);
  prefetch(t0 + step);
  hash();
  __syncthreads();
  for (; t0 < n; t0 += step) {
    if (have == KR) push(KR);
    else push(have);
    have = mine(t0 + step);
    load(t0 + step, have);
    prefetch(t0 + 2 * step);
    __syncthreads();
    const unsigned ns = *(volatile unsigned *)nspill;
    unsigned nf[OWN], head[OWN];  // whole quanta held (at most S / Q), first entry
    u64 g[OWN];
#pragma unroll
    for (int o = 0; o < OWN; o++) {
      const unsigned li = lane + 32 * o, i = warp * per + li;
      nf[o] = 0;
      if (Dest::kShared) g[o] = 0;
      if (li < per && i < nb) {
        const unsigned c = cnt[i], m = min(c >> 16, S);
        head[o] = (c - (c >> 16)) & (S - 1);
        nf[o] = m >> lq;
        cnt[i] = ((m & (Q - 1)) << 16) | ((head[o] + m) & (S - 1));
        if (!Dest::kShared && nf[o]) g[o] = atomicAdd(dest(i).counter, (u64)(nf[o] << lq));
      }
    }
    // rings that share a counter: one atomic for those of a warp
    unsigned before[OWN], lead[OWN];
    if (Dest::kShared) {
#pragma unroll
      for (int o = 0; o < OWN; o++) {
        const unsigned li = lane + 32 * o, i = warp * per + li;
        u64 *ctr = li < per && i < nb ? dest(i).counter : nullptr;
        const unsigned same = __match_any_sync(0xffffffffu, (u64)ctr);
        unsigned sum = 0;
        before[o] = 0;
        for (unsigned bit = 0; bit <= ls - lq; bit++) {
          const unsigned bb = __ballot_sync(0xffffffffu, (nf[o] >> bit) & 1u) & same;
          before[o] += __popc(bb & lt) << bit;
          sum += __popc(bb) << bit;
        }
        lead[o] = __ffs(same) - 1;
        if (lane == lead[o] && sum) g[o] = atomicAdd(ctr, (u64)(sum << lq));
      }
    }
    // in a block of its own: the reservations are on their way before it
    if (have) hash();
    unsigned nj = 0;
#pragma unroll
    for (int o = 0; o < OWN; o++) {
      const unsigned i = warp * per + lane + 32 * o;
      WcJob j;
      if (Dest::kShared)
        g[o] = __shfl_sync(0xffffffffu, g[o], lead[o]) + ((u64)before[o] << lq);
      if (nf[o]) {
        const DestRun r = dest(i);
        if (g[o] + (nf[o] << lq) > r.cap) {
          // past the bucket's end: what fits is written, so that every slot below
          // min(counter, cap) always holds a value of this bucket
          if (g[o] < r.cap)
            wc_fill_end(buf + (i << ls), head[o], S - 1, arena + (r.base + g[o]), r.cap - g[o]);
          nf[o] = 0;
          atomicOr(status, 1u);
        }
        j.dst = arena + (r.base + g[o]);
        j.src = buf0 + 8 * ((i << ls) + head[o]);
        j.count = Q;
      }
      const unsigned b1 = __ballot_sync(0xffffffffu, nf[o] > 0);
      const unsigned b2 = __ballot_sync(0xffffffffu, nf[o] > 1);
      unsigned bq = __ballot_sync(0xffffffffu, nf[o] > 2);
      if (nf[o] > 0) jobs[nj + __popc(b1 & lt)] = j;
      nj += __popc(b1);
      auto next = [&](unsigned q, unsigned at) {
        j.src = buf0 + 8 * ((i << ls) + ((head[o] + (q << lq)) & (S - 1)));
        j.dst += Q;
        jobs[at] = j;
      };
      if (nf[o] > 1) next(1, nj + __popc(b2 & lt));
      nj += __popc(b2);
      for (unsigned q = 2; bq; q++) {  // rings of more than two quanta
        if (nf[o] > q) next(q, nj + __popc(bq & lt));
        nj += __popc(bq);
        bq = __ballot_sync(0xffffffffu, nf[o] > q + 1);
      }
    }
    __syncwarp();
    copy(nj);
    __syncthreads();
    // a spill list that fills up goes back through the rings
    if (ns > kWSpill / 2) {
      const bool mine_s = tid < min(ns, kWSpill);
      const u64 v = mine_s ? spill[tid] : 0;
      __syncthreads();
      if (tid == 0) *nspill = 0;
      __syncthreads();
      if (mine_s) {
        const unsigned bb = dst(v), c = atomicAdd(cnt + bb, 0x10001u);
        if (c < full) buf[(bb << ls) + (c & (S - 1))] = v;
        else spilled(v, bb);
      }
    }
  }
  __syncthreads();
  // what is left in the rings, then the spill list
  for (int pass = 0; pass < 2; pass++) {
    unsigned nj = 0;
#pragma unroll
    for (int o = 0; o < OWN; o++) {
      const unsigned li = lane + 32 * o, i = warp * per + li;
      const unsigned c = li < per && i < nb ? cnt[i] : 0u, left = min(c >> 16, S);
      const unsigned head = (c - (c >> 16)) & (S - 1);
      // first pass: whole quanta (after a push of the spill list), then the rest
      unsigned m = pass ? left & (Q - 1) : left & ~(Q - 1);
      if (!pass && left) cnt[i] = ((left & (Q - 1)) << 16) | ((head + left) & (S - 1));
      WcJob j;
      if (m) {
        const DestRun r = dest(i);
        const u64 g = atomicAdd(r.counter, (u64)m);
        if (g + m > r.cap) {  // what fits is written (see above)
          m = g < r.cap ? (unsigned)(r.cap - g) : 0;
          atomicOr(status, 1u);
        }
        j.dst = arena + (r.base + g);
      }
      for (unsigned q = 0;; q++) {
        const bool have_q = (q << lq) < m;
        const unsigned bq = __ballot_sync(0xffffffffu, have_q);
        if (!bq) break;
        if (have_q) {
          j.src = buf0 + 8 * ((i << ls) + ((head + (q << lq)) & (S - 1)));
          j.count = min(m - (q << lq), Q);
          jobs[nj + __popc(bq & lt)] = j;
          j.dst += Q;
        }
        nj += __popc(bq);
      }
    }
    __syncwarp();
    for (unsigned j = lane >> lq; j < nj; j += ng)
      if (l < jobs[j].count) move(jobs[j]);
    __syncwarp();
  }
  const unsigned ns = min(*nspill, kWSpill);
  for (unsigned j = tid; j < ns; j += NT) one(spill[j], dst(spill[j]));
}

// key(v): the value stored for input v; dst(y): its destination (< sh.nb);
// dest(b): the bucket's counter, base and capacity (Dest::kShared: destinations
// next to each other may share them).  The caller is CTA `rank`
// of the `ranks` that share the n values.  OWN: 1 up to NT destinations, 2
// beyond.
template <int NT, int OWN, class Key, class Dst, class Dest>
__device__ __forceinline__ void wc_split(const u64 *__restrict__ in, u64 n, unsigned rank,
                                         unsigned ranks, const WcShape &sh, unsigned char *smem,
                                         const Key &key, const Dst &dst, const Dest &dest,
                                         u64 *__restrict__ arena, unsigned *__restrict__ status) {
  if (wc_smem_bytes(sh) > sh.smem || sh.nb > (unsigned)(OWN * NT)) {  // rings that do not fit
    if (threadIdx.x == 0) atomicOr(status, 1u);
    return;
  }
  const unsigned kr = wc_round(sh, n, ranks);
  const unsigned tile = kr ? kr * NT : ((sh.nb << sh.ls) * 3 / 8 + 31) & ~31u;
#define WC_ROUNDS(KR) \
  wc_rounds<NT, OWN, KR>(in, n, rank, ranks, tile, sh, smem, key, dst, dest, arena, status)
  if (kr == 8) WC_ROUNDS(8);
  else if (kr == 6) WC_ROUNDS(6);
  else if (kr == 4) WC_ROUNDS(4);
  else if (kr == 2) WC_ROUNDS(2);
  else WC_ROUNDS(1);
#undef WC_ROUNDS
}

}  // namespace bbh
