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

// reduce_range for m < 2^32.
__device__ __forceinline__ unsigned reduce_range32(u64 h, unsigned m) {
  const u64 t = ((u64)(unsigned)h * m) >> 32;
  return (unsigned)(((u64)(unsigned)(h >> 32) * m + t) >> 32);
}

// ---------------------------------------------------------------------------
// One CTA's share of a multisplit of n values.  Every destination has a ring
// of two quanta of 2^lq slots in shared memory.  A round pushes one tile: a
// value takes the next slot of its destination with one shared atomic and is
// stored there.  Then each destination that holds a whole quantum (or two) has
// it reserved (one global atomic, by the lane that owns the destination) and
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
// ---------------------------------------------------------------------------
static constexpr int kWT = 1024;          // threads of a split CTA
static constexpr int kWK = 8;             // values per thread and round at most
static constexpr unsigned kWMaxNb = 2048; // destinations at most
static constexpr unsigned kWSpill = 512;  // entries of the spill list
static constexpr unsigned kWSmem = 227 * 1024;

// A queued run: 2^lq ring entries from shared-memory byte `src` to global `dst`.
struct WcJob {
  unsigned src, count;
  u64 *dst;
};

struct WcShape {
  unsigned nb, lq;
  unsigned per;  // destinations a warp owns
};

__host__ __device__ inline u64 wc_smem_bytes(const WcShape &s) {
  return (u64)(kWT / 32) * 2 * s.per * sizeof(WcJob) + (((u64)s.nb << (s.lq + 1)) + kWSpill) * 8 +
         (u64)s.nb * 4 + 16;
}

// Quantum size for nb destinations: the largest (at most a warp's lanes) whose
// rings fit.
__host__ __device__ inline WcShape wc_shape(unsigned nb) {
  WcShape s;
  s.nb = nb;
  s.per = (nb + kWT / 32 - 1) / (kWT / 32);
  for (s.lq = 5; s.lq > 2 && wc_smem_bytes(s) > kWSmem; s.lq--) {
  }
  return s;
}

// Values per thread and round: all the CTA has if that is little, and at most
// what fills a third of the rings (a ring rarely overflows then).  0: so few
// destinations that a round takes less than one value per thread.
__host__ __device__ inline unsigned wc_round(const WcShape &s, u64 n, unsigned ctas) {
  const unsigned fill = (s.nb << (s.lq + 1)) * 11 / 32 / kWT;
  const u64 have = (n + (u64)ctas * kWT - 1) / ((u64)ctas * kWT);
  const u64 k = fill < have ? fill : have;
  return k < kWK ? (unsigned)k : (unsigned)kWK;
}

// key(v): the value stored for input v; dst(y): its destination (< sh.nb);
// dest(b): the bucket's counter, base and capacity.  OWN: 1 up to kWT
// destinations, 2 beyond.
template <int OWN, class Key, class Dst, class Dest>
__device__ __forceinline__ void wc_split(const u64 *__restrict__ in, u64 n, const WcShape &sh,
                                         unsigned char *smem, const Key &key, const Dst &dst,
                                         const Dest &dest, u64 *__restrict__ arena,
                                         unsigned *__restrict__ status) {
  const unsigned nb = sh.nb, lq = sh.lq, ls = lq + 1, per = sh.per;
  const unsigned S = 1u << ls, Q = 1u << lq;
  const unsigned tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, lt = (1u << lane) - 1u;
  WcJob *jobs = reinterpret_cast<WcJob *>(smem) + warp * 2 * per;  // this warp's queue
  const unsigned buf0 = (kWT / 32) * 2 * per * (unsigned)sizeof(WcJob);
  u64 *buf = reinterpret_cast<u64 *>(smem + buf0);
  u64 *spill = buf + ((u64)nb << ls);
  // per destination: (entries in the ring << 16) | tail; both only grow in a
  // round, the owner brings the tail back below S and takes the entries out
  unsigned *cnt = reinterpret_cast<unsigned *>(spill + kWSpill);
  unsigned *nspill = cnt + nb;
  for (unsigned i = tid; i < nb; i += kWT) cnt[i] = 0;
  if (tid == 0) *nspill = 0;
  const unsigned kr0 = wc_round(sh, n, gridDim.x), kr = kr0 ? kr0 : 1u;
  const unsigned tile = kr0 ? kr0 * kWT : ((nb << ls) * 11 / 32 + 31) & ~31u;
  const u64 step = (u64)gridDim.x * tile;
  u64 t0 = (u64)blockIdx.x * tile;
  const unsigned full = S << 16;
  u64 y[kWK];       // inputs, then their stored values
  unsigned b[kWK];  // destination << ls
  // values of the tile at `at` that exist for this thread (k < that number)
  auto mine = [&](u64 at) -> unsigned {
    if (at >= n) return 0;
    const unsigned len = at + tile <= n ? tile : (unsigned)(n - at);
    return len == kr * kWT ? kr : len > tid ? (len - tid + kWT - 1) / kWT : 0;
  };
  auto load = [&](u64 at, unsigned have) {
    const u64 *p = in + at + tid;
#pragma unroll
    for (int k = 0; k < kWK; k++)
      if ((unsigned)k < have) y[k] = __ldcs(p + k * kWT);
  };
  // the tile at `at` into L2, so that its loads a round later are short
  auto prefetch = [&](u64 at) {
    if (tid == 0 && at + tile <= n) {
      const uintptr_t p = ((uintptr_t)(in + at) + 15) & ~(uintptr_t)15;
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(tile * 8 - 16));
    }
  };
  auto hash = [&](unsigned have) {
#pragma unroll
    for (int k = 0; k < kWK; k++)
      if ((unsigned)k < have) {
        y[k] = key(y[k]);
        b[k] = dst(y[k]) << ls;
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
  unsigned have = mine(t0);
  load(t0, have);
  prefetch(t0 + step);
  hash(have);
  __syncthreads();
  for (; t0 < n; t0 += step) {
#pragma unroll
    for (int k = 0; k < kWK; k++)
      if ((unsigned)k < have) {
        const unsigned c = atomicAdd(cnt + (b[k] >> ls), 0x10001u);
        if (c < full) {
          buf[b[k] | (c & (S - 1))] = y[k];
        } else {
          unsigned j = kWSpill;
          if (*(volatile unsigned *)nspill < kWSpill) j = atomicAdd(nspill, 1u);
          if (j < kWSpill) spill[j] = y[k];
          else one(y[k], b[k] >> ls);
        }
      }
    have = mine(t0 + step);
    load(t0 + step, have);
    prefetch(t0 + 2 * step);
    __syncthreads();
    unsigned nf[OWN], head[OWN];  // whole quanta held (0, 1 or 2), first entry
    u64 g[OWN];
#pragma unroll
    for (int o = 0; o < OWN; o++) {
      const unsigned li = lane + 32 * o, i = warp * per + li;
      nf[o] = 0;
      if (li < per && i < nb) {
        const unsigned c = cnt[i], m = min(c >> 16, S);
        head[o] = (c - (c >> 16)) & (S - 1);
        nf[o] = m >> lq;
        cnt[i] = ((m & (Q - 1)) << 16) | ((head[o] + m) & (S - 1));
        if (nf[o]) g[o] = atomicAdd(dest(i).counter, (u64)(nf[o] << lq));
      }
    }
    hash(have);
    unsigned nj = 0;
#pragma unroll
    for (int o = 0; o < OWN; o++) {
      const unsigned i = warp * per + lane + 32 * o;
      WcJob j;
      if (nf[o]) {
        const DestRun r = dest(i);
        if (g[o] + (nf[o] << lq) > r.cap) {  // past the bucket's end: dropped
          nf[o] = 0;
          atomicOr(status, 1u);
        }
        j.dst = arena + (r.base + g[o]);
        j.src = buf0 + 8 * ((i << ls) + head[o]);
        j.count = Q;
      }
      const unsigned b1 = __ballot_sync(0xffffffffu, nf[o] != 0);
      const unsigned b2 = __ballot_sync(0xffffffffu, nf[o] == 2);
      if (nf[o]) jobs[nj + __popc(b1 & lt)] = j;
      nj += __popc(b1);
      if (nf[o] == 2) {
        j.src = buf0 + 8 * ((i << ls) + (head[o] ^ Q));
        j.dst += Q;
        jobs[nj + __popc(b2 & lt)] = j;
      }
      nj += __popc(b2);
    }
    __syncwarp();
    copy(nj);
    __syncthreads();
  }
  // what is left in the rings (less than a quantum each), then the spill list
  unsigned nj = 0;
#pragma unroll
  for (int o = 0; o < OWN; o++) {
    const unsigned li = lane + 32 * o, i = warp * per + li;
    const unsigned c = li < per && i < nb ? cnt[i] : 0u, m = c >> 16;
    WcJob j;
    j.count = 0;
    if (m) {
      const DestRun r = dest(i);
      const u64 g = atomicAdd(r.counter, (u64)m);
      if (g + m <= r.cap) j.count = m;
      else atomicOr(status, 1u);
      j.src = buf0 + 8 * ((i << ls) + ((c - m) & (S - 1)));
      j.dst = arena + (r.base + g);
    }
    const unsigned bb = __ballot_sync(0xffffffffu, j.count != 0);
    if (j.count) jobs[nj + __popc(bb & lt)] = j;
    nj += __popc(bb);
  }
  __syncwarp();
  for (unsigned j = lane >> lq; j < nj; j += ng)
    if (l < jobs[j].count) move(jobs[j]);
  const unsigned ns = min(*nspill, kWSpill);
  for (unsigned j = tid; j < ns; j += kWT) one(spill[j], dst(spill[j]));
}

}  // namespace bbh
