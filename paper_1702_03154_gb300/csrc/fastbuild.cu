// fastbuild.cu -- bucketed construction: ArrayFill in shared memory.
//
// A level runs in two launches.  k_split hashes the level's keys and writes
// them to position buckets (P consecutive positions of A_d, P a power of two)
// through the write-combining multisplit of split.cuh.  k_fill_compact then
// runs Algorithm 2 for a bucket with its hit / collision bits in shared memory
// (no L2 atomics), writes the bucket's slice of A_d, and appends the keys whose
// bit is 0 to F_{d+1}.  Once every bucket is done |F_{d+1}| and |A_{d+1}| are
// known and level d+1's split can run.  Levels with at most T keys run in a
// single CTA (k_tail) that keeps keys and bit arrays in shared memory and loops
// over all remaining levels, sorting the fallback (Sec. 3.5) at the end.
//
// Buckets and F hold h_d(x), not x: the hash is a bijection of 64-bit values
// (unmix64), so its value stands for the key, the position costs one multiply
// instead of a stored 4-byte position or a second hash, and only the survivors
// of a level are hashed again.  A visit of a key reads and writes 8 bytes in
// the split, reads 8 twice in the fill (the second time partly from L2) and
// writes 8 per survivor.
//
// Every bound (bucket capacity, bucket count, F) is checked on the device;
// when one is exceeded the build is redone by the unbucketed path in build.cu,
// so results never depend on these choices.
//
// Measured (GB300, 1e8 keys, gamma = 2, 763 buckets at level 0): split of
// level 0 0.43 ms, of all levels 0.88 ms; fill and compaction 0.38 / 0.76 ms;
// build 1.79 ms.  A counting-sort multisplit that stored (key, position) pairs,
// with a fill and a compaction that fed the next level's multisplit, took 0.89
// ms for level 0, 0.32 + 1.02 ms for fills and compactions, 2.34 ms in all.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>

#include "fastbuild.cuh"
#include "sector.cuh"
#include "split.cuh"

namespace bbh {


// Position of hash value y in A_d, modulo 2^32 (NARROW: m < 2^32).
template <bool NARROW>
__device__ __forceinline__ unsigned position(u64 y, u64 m) {
  return NARROW ? reduce_range32(y, (unsigned)m) : (unsigned)__umul64hi(y, m);
}

// Split of level d: the caller's keys (d = 0) or the survivors of level d - 1
// (F, as values h_{d-1}) to the position buckets of A_d, as values h_d.
template <int OWN, bool FIRST>
__global__ void __launch_bounds__(kWT, 1)
k_split(const u64 *__restrict__ keys, u64 n, FastMeta *__restrict__ meta, int d, FastCfg cfg,
        unsigned nb_max) {
  extern __shared__ __align__(16) unsigned char smem[];
  // one decision for the whole CTA: another CTA may be raising the status now
  if (__syncthreads_or(meta->lv[d].mode != LM_BUCKETED || *(volatile unsigned *)&meta->status))
    return;
  const FLevel lv = meta->lv[d];
  if (lv.B > nb_max) {  // more buckets than the rings were sized for
    if (threadIdx.x == 0) atomicOr(&meta->status, ST_OVERFLOW);
    return;
  }
  const WcShape sh = wc_shape((unsigned)lv.B, kWT, wc_smem(1));
  const u64 s_d = level_seed(cfg.seed, d);
  const u64 s_x = FIRST ? s_d : s_d ^ level_seed(cfg.seed, d - 1);
  const unsigned m = (unsigned)lv.m, shift = ilog2_u64(lv.P);
  wc_split<kWT, OWN>(
      FIRST ? keys : cfg.F, FIRST ? n : lv.n, blockIdx.x, gridDim.x, sh, smem,
      [=](u64 v) { return mix64((FIRST ? v : unmix64(v)) ^ s_x); },
      [=](u64 y) { return reduce_range32(y, m) >> shift; }, UniformDest{cfg.cnt, lv.cap}, cfg.X,
      &meta->status);
}

// |F_{d+1}| = |F_d| - weight(A_d); level d+1's size and where it lives.
__device__ void finish_level(FastMeta *meta, int d, const FastCfg &cfg) {
  volatile FLevel *vl = meta->lv;
  const u64 n = vl[d].n, m = vl[d].m, w = vl[d].weight;
  if (w > n) atomicOr(&meta->status, ST_INTERNAL);
  const u64 nn = w > n ? 0 : n - w;
  FLevel nx;
  memset(&nx, 0, sizeof(nx));
  nx.n = nn;
  nx.off = vl[d].off + m;
  if (nn == 0) {
    nx.mode = LM_DONE;
    meta->levels_used = d + 1;
  } else if ((uint32_t)(d + 1) == cfg.L) {
    nx.mode = LM_FLAT;  // fallback
  } else if (nn <= cfg.T) {
    nx.mode = LM_FLAT;  // tail
    nx.m = level_bits(nn, cfg.gamma);
  } else if (nn <= cfg.Tmid && level_bits(nn, cfg.gamma) <= cfg.mmid) {
    nx.mode = LM_MID;
    nx.m = level_bits(nn, cfg.gamma);
  } else {
    size_bucketed(nx, nn, cfg.gamma, cfg.Pmin, cfg.Pmax, cfg.Btarget, cfg.cap_scale);
    nx.off = vl[d].off + m;
    nx.mode = LM_BUCKETED;
    // the arena was allocated before level 0 ran (from a bound on |F_1|): a
    // level that does not fit sends the build to the unbucketed path
    const bool a_fits = ((nx.off - cfg.m0) >> 6) + (nx.m >> 6) <= cfg.arena_words;
    if (nx.B > cfg.Bmax || nx.B * nx.cap > cfg.capX || !a_fits) {
      atomicOr(&meta->status, ST_OVERFLOW);
      nx.mode = LM_NONE;
    }
  }
  meta->lv[d + 1] = nx;
  __threadfence();
}

// ---------------------------------------------------------------------------
// ArrayFill (Algorithm 2) and compaction (Algorithm 1) of buckets of one
// level, a bucket per CTA iteration with its hit and collision bits in shared
// memory.  Pass 1 streams the bucket's values and sets the bits; A_d's words
// of the bucket leave and their ones are counted, which also fixes the number
// of survivors (values in the bucket less ones), so one global atomic reserves
// the whole bucket's run of F_{d+1}.  Pass 2 streams the values again, last
// first, and writes those whose bit is 0, each warp taking its part of the run
// with a shared-memory atomic.
// ---------------------------------------------------------------------------
struct FillArgs {
  const u64 *X;    // values, bucket b at [b cap, b cap + cnt[b])
  const u64 *cnt;
  u64 cap, B;      // slots of a bucket, buckets
  u64 m, P, p0;    // |A_d|; positions of a bucket; first position of bucket 0
  u64 *A;          // A_d
  u64 *F, F_cap, *n_out;
  unsigned *status;
};

static constexpr unsigned kFillStage = 256;  // survivors a warp stages at most
__host__ __device__ constexpr size_t fill_smem(u64 P) {
  return (size_t)P / 4 + (size_t)(kTT / 32) * kFillStage * 8;
}

// Adds the ones of the CTA's buckets and the values found in them to wtot and
// got (thread 0).
template <bool NARROW>
__device__ __forceinline__ void fill_compact(const FillArgs &a, unsigned char *smem, u64 &wtot,
                                             u64 &got) {
  __shared__ u64 red[kTT / 32];
  __shared__ u64 s_base;
  __shared__ unsigned s_count, s_room;
  const unsigned Pw = (unsigned)(a.P >> 5);  // 32-bit words per bit array
  unsigned *hit = reinterpret_cast<unsigned *>(smem);
  unsigned *col = hit + Pw;
  const unsigned lane = threadIdx.x & 31, lt = (1u << lane) - 1u;
  u64 *stage = reinterpret_cast<u64 *>(col + Pw) + (threadIdx.x >> 5) * kFillStage;
  for (u64 b = blockIdx.x; b < a.B; b += gridDim.x) {
    for (unsigned i = threadIdx.x; i < Pw / 2; i += kTT)
      reinterpret_cast<uint4 *>(smem)[i] = make_uint4(0, 0, 0, 0);
    const unsigned nk = (unsigned)min(a.cnt[b], a.cap);
    const u64 *yb = a.X + b * a.cap;
    const uint4 *y4 = reinterpret_cast<const uint4 *>(yb);  // cap % 16 == 0
    const unsigned p0 = (unsigned)(a.p0 + b * a.P);  // positions modulo 2^32
    const unsigned nv = nk >> 1;  // pairs of values
    auto val0 = [](const uint4 &v) { return ((u64)v.y << 32) | v.x; };
    auto val1 = [](const uint4 &v) { return ((u64)v.w << 32) | v.z; };
    // position in the bucket; -p0 rides in the upper half of the last product's
    // addend
    auto local = [&](u64 y) -> unsigned {
      if (NARROW) {
        const unsigned m = (unsigned)a.m;
        const u64 t = ((u64)(unsigned)y * m) >> 32;
        return (unsigned)(((u64)(unsigned)(y >> 32) * m + (((u64)(0u - p0) << 32) | t)) >> 32);
      }
      return (unsigned)__umul64hi(y, a.m) - p0;
    };
    __syncthreads();
    constexpr int U = 4;  // pairs in flight per thread
    constexpr unsigned kStep = U * kTT;
    const unsigned nfull = nv / kStep, nsteps = (nv + kStep - 1) / kStep;
    // step s of the bucket into L2 (its loads come later)
    auto ahead = [&](unsigned s) {
      if (threadIdx.x == 0 && s < nsteps)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(y4 + s * kStep),
                     "r"(min(kStep, nv - s * kStep) * 16));
    };
    // pass 1: every value lies in this bucket, whatever the input (a split fills
    // an overflowing bucket to its end), so positions need no mask
    auto set = [&](u64 y) {
      const unsigned q = local(y);
      const unsigned bit = 1u << (q & 31);
      const unsigned old = atomicOr(hit + (q >> 5), bit);
      if (old & bit) atomicOr(col + (q >> 5), bit);
    };
    ahead(1);
    for (unsigned st = 0; st < nfull; st++) {
      ahead(st + 2);
      const uint4 *src = y4 + st * kStep + threadIdx.x;
      uint4 v[U];
#pragma unroll
      for (int u = 0; u < U; u++) v[u] = __ldcg(src + u * kTT);
#pragma unroll
      for (int u = 0; u < U; u++) {
        set(val0(v[u]));
        set(val1(v[u]));
      }
    }
    for (unsigned i = nfull * kStep + threadIdx.x; i < nv; i += kTT) {
      const uint4 v = __ldcg(y4 + i);
      set(val0(v));
      set(val1(v));
    }
    if ((nk & 1) && threadIdx.x == 0) set(yb[nk - 1]);
    __syncthreads();
    // A_d words of this bucket's positions; hit keeps A
    const u64 w0 = (a.p0 + b * a.P) >> 6;
    const unsigned nw = (unsigned)((min(a.p0 + (b + 1) * a.P, a.m) >> 6) - w0);
    unsigned wsum = 0;
    for (unsigned w = threadIdx.x; w < nw; w += kTT) {
      const uint2 h2 = reinterpret_cast<uint2 *>(hit)[w], c2 = reinterpret_cast<uint2 *>(col)[w];
      const uint2 k2 = make_uint2(h2.x & ~c2.x, h2.y & ~c2.y);
      reinterpret_cast<uint2 *>(hit)[w] = k2;
      a.A[w0 + w] = ((u64)k2.y << 32) | k2.x;
      wsum += __popc(k2.x) + __popc(k2.y);
    }
    wsum = __reduce_add_sync(0xffffffffu, wsum);
    if (lane == 0) red[threadIdx.x >> 5] = wsum;
    __syncthreads();
    if (threadIdx.x == 0) {
      u64 w = 0;
      for (int i = 0; i < kTT / 32; i++) w += red[i];
      wtot += w;
      got += a.cnt[b];
      const u64 ns = w > nk ? 0 : nk - w;
      const u64 at = ns ? atomicAdd(a.n_out, ns) : 0;
      const bool fits = w <= nk && at + ns <= a.F_cap;
      if (!fits) atomicOr(a.status, ST_OVERFLOW);
      s_base = at;
      s_room = fits ? (unsigned)ns : 0u;
      s_count = 0;
    }
    __syncthreads();
    u64 *out = a.F + s_base;
    const unsigned room = s_room;
    // pass 2, last step first (it is the likeliest to be still in L2): each
    // warp packs its survivors in its stage and writes them out as one run
    unsigned cnt = 0;
    auto flush = [&]() {
      __syncwarp();
      unsigned at = 0;
      if (lane == 0) at = atomicAdd(&s_count, cnt);
      at = __shfl_sync(0xffffffffu, at, 0);
      if (at + cnt <= room)  // else F_{d+1} is full (status raised)
        for (unsigned j = lane; j < cnt; j += 32) out[at + j] = stage[j];
      __syncwarp();
      cnt = 0;
    };
    auto put = [&](bool ok, u64 y) {
      const unsigned q = local(y) & (unsigned)(a.P - 1);  // in range for a value that is none, too
      const bool keep = ok && !((hit[q >> 5] >> (q & 31)) & 1u);
      const unsigned bal = __ballot_sync(0xffffffffu, keep);
      if (keep) stage[cnt + __popc(bal & lt)] = y;
      cnt += __popc(bal);
    };
    static_assert(kFillStage >= 4 * 32 + 4 * 32, "four puts after a stage that was not flushed");
    for (unsigned st = nsteps; st-- > 0;) {
      ahead(st - 2);
      const unsigned i0 = st * kStep + threadIdx.x;
      uint4 v[U];
      const bool all = st < nfull;
#pragma unroll
      for (int u = 0; u < U; u++)
        v[u] = all || i0 + u * kTT < nv ? __ldcs(y4 + i0 + u * kTT) : make_uint4(0, 0, 0, 0);
#pragma unroll
      for (int u = 0; u < U; u += 2) {
        put(all || i0 + u * kTT < nv, val0(v[u]));
        put(all || i0 + u * kTT < nv, val1(v[u]));
        put(all || i0 + (u + 1) * kTT < nv, val0(v[u + 1]));
        put(all || i0 + (u + 1) * kTT < nv, val1(v[u + 1]));
        if (cnt > kFillStage - 4 * 32) flush();
      }
    }
    if (threadIdx.x < 32 && (nk & 1)) put(lane == 0, yb[nk - 1]);
    if (cnt) flush();
    __syncthreads();
  }
}

// Level d of the device-driven loop; the last CTA sizes level d+1.
__global__ void __launch_bounds__(kTT, 2)
k_fill_compact(FastMeta *__restrict__ meta, int d, FastCfg cfg) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ bool last;
  if (__syncthreads_or(meta->lv[d].mode != LM_BUCKETED || *(volatile unsigned *)&meta->status))
    return;
  const FLevel lv = meta->lv[d];
  u64 *Alev = (d == 0) ? cfg.A0 : cfg.arena + ((lv.off - cfg.m0) >> 6);
  u64 wtot = 0, got = 0;
  fill_compact<true>(FillArgs{cfg.X, cfg.cnt, lv.cap, lv.B, lv.m, lv.P, 0, Alev, cfg.F, cfg.F_cap,
                              &meta->n_out[d], &meta->status},
                     smem, wtot, got);
  if (threadIdx.x == 0) {
    if (wtot) atomicAdd(&meta->lv[d].weight, wtot);
    if (got) atomicAdd(&meta->seen[d], got);
    __threadfence();
    unsigned t = atomicAdd(&meta->lv[d].done, 1u);
    last = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (last && threadIdx.x == 0) {
    __threadfence();
    // the buckets must hold exactly |F_d| keys
    if (*(volatile u64 *)&meta->seen[d] != meta->lv[d].n) atomicOr(&meta->status, ST_INTERNAL);
    finish_level(meta, d, cfg);
  }
  if (last) {
    __syncthreads();
    // zero the bucket counters for level d+1's split
    const FLevel nx = meta->lv[d + 1];
    if (nx.mode == LM_BUCKETED)
      for (u64 i = threadIdx.x; i < nx.B; i += kTT) cfg.cnt[i] = 0;
  }
}

// ---------------------------------------------------------------------------
// Levels with more buckets than one split takes well are grouped in two
// steps: all values to coarse slabs of 2^cs positions (k_gsplit),
// then, a batch of slabs at a time, each slab's values to its fine buckets of
// 2^kGroupShift positions (k_fsplit: a group of CTAs per slab) and the batch's
// buckets filled and compacted (k_gfill).  Measured at 3e9 keys (gamma = 2):
// coarse 20.5 ms, fine 18.8, fill and compaction 14.6 for the three grouped
// levels (4.6e9 values, 16 bytes a split), build 58 ms; counting-sort
// multisplits and a fill from stored positions took 54.5 + 23.1 ms, build 81.
// ---------------------------------------------------------------------------
static constexpr unsigned kGroupShift = 17;
static constexpr unsigned kBatchFine = 2048;  // fine buckets per batch

// Coarse slabs of a level of m positions: 2^shift positions each, so that the
// two splits have about as many destinations (a third or three times as many
// slabs: within 3% at 3e9 keys).
static unsigned coarse_shift(u64 m) {
  unsigned sh = kGroupShift;
  while (ceil_div(m, 1ull << sh) > 1ull << (sh - kGroupShift) && sh < kGroupShift + 9) sh++;
  return sh;
}
// Group a level of more buckets than one split takes.  Both sides measured at
// 2.6e8 keys (gamma 2, 1984 buckets): one split 5.3 ms a build, two steps 6.1.
static constexpr u64 kGroupMinB = kBmax;

// A launch behind an overflow does nothing (the host looks once a level).  One
// decision for the whole CTA: another one may be raising the status now.
__device__ __forceinline__ bool raised(const unsigned *status) {
  return __syncthreads_or(*(const volatile unsigned *)status) != 0;
}

template <int NT, bool FIRST, bool NARROW>
__global__ void __launch_bounds__(NT, kWT / NT)
k_gsplit(const u64 *__restrict__ in, u64 n, u64 m, unsigned cs, u64 s_x, unsigned nb,
         u64 *__restrict__ cnt, u64 cap, u64 *__restrict__ out, unsigned *__restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (raised(status)) return;
  wc_split<NT, 1>(
      in, n, blockIdx.x, gridDim.x, wc_shape(nb, NT, wc_smem(kWT / NT)), smem,
      [=](u64 v) { return mix64((FIRST ? v : unmix64(v)) ^ s_x); },
      [=](u64 y) {
        return NARROW ? reduce_range32(y, (unsigned)m) >> cs : (unsigned)(__umul64hi(y, m) >> cs);
      },
      UniformDest{cnt, cap}, out, status);
}

// Slabs [s0, s0 + ns) of R (cap_c slots each) into fine buckets of cap_f
// slots; gridDim.x = ns * (CTAs a slab).
template <int NT, bool NARROW>
__global__ void __launch_bounds__(NT, kWT / NT)
k_fsplit(const u64 *__restrict__ R, const u64 *__restrict__ cnt_c, u64 cap_c, unsigned s0,
         unsigned ns, unsigned nf, u64 m, u64 *__restrict__ cnt_f, u64 cap_f, u64 *__restrict__ T,
         unsigned *__restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (raised(status)) return;
  const unsigned per = gridDim.x / ns, j = blockIdx.x / per;
  const u64 n = min(cnt_c[s0 + j], cap_c);
  const unsigned f0 = (s0 + j) * nf;  // the slab's first fine bucket
  wc_split<NT, 1>(
      R + (s0 + j) * cap_c, n, blockIdx.x - j * per, per, wc_shape(nf, NT, wc_smem(kWT / NT)), smem,
      [](u64 v) { return v; },
      [=](u64 y) {
        return (NARROW ? reduce_range32(y, (unsigned)m) >> kGroupShift
                       : (unsigned)(__umul64hi(y, m) >> kGroupShift)) - f0;
      },
      UniformDest{cnt_f + j * nf, cap_f}, T + (u64)j * nf * cap_f, status);
}

template <bool NARROW>
__global__ void __launch_bounds__(kTT, 2)
k_gfill(FillArgs a, u64 *__restrict__ weight, u64 *__restrict__ seen) {
  extern __shared__ __align__(16) unsigned char smem[];
  if (raised(a.status)) return;
  u64 wtot = 0, got = 0;
  fill_compact<NARROW>(a, smem, wtot, got);
  if (threadIdx.x == 0) {
    if (wtot) atomicAdd(weight, wtot);
    if (got) atomicAdd(seen, got);
  }
}

// A fallback too large for the tail: the values h_{L-1} of F back to keys.
__global__ void k_unhash(u64 *__restrict__ F, u64 n, u64 s) {
  const u64 stride = (u64)gridDim.x * blockDim.x;
  for (u64 i = (u64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
    F[i] = unmix64(F[i]) ^ s;
}

// ---------------------------------------------------------------------------
// Levels of at most Tmid keys, down to the tail, in one cooperative launch of
// one CTA a multiprocessor.  A level of 10^4 to 10^6 keys is bound by latency:
// two launches of a split and a fill took 20 us whatever its size.  Here each
// CTA keeps its share of the keys in shared memory, the hit and collision bits
// are in L2 (64-bit words: bits 0-31 hit, 32-63 collision, so a key costs one
// atomic and the collided ones a second), and a level is: set the bits, grid
// barrier, test them, drop the placed keys and write A_d, grid barrier.  The
// two bit arrays take turns; a level clears the other one behind it.
// Both sides measured (gamma = 2): build of 2e5 keys 150 us against 225, 1e6 166
// against 243, 3e6 231 against 330; reach of 1e6 / 3.5e6 keys: build of 3e6 249
// / 231, of 2e7 strings 1079 / 1061.
// A CTA takes half a multiprocessor's registers and threads, with eight keys a
// thread in flight, so that lookups of a server run beside it: with 1024 threads
// of four keys, builds of 1e5 to 1e6 keys among 1.6e5 requests/s brought the
// lookups' p99 to 0.091 ms, with 512 to 0.081 (1e6 to 3.4e6: 0.137 / 0.107);
// builds take the same time (1e6 172 us, 2.7e6 218, 3.4e6 235 / 243).
// ---------------------------------------------------------------------------
static constexpr int kMidThreads = 512;
static constexpr unsigned kMidKeys = 24576;  // of a CTA
static constexpr u64 kMidMax = 3500000;      // keys of a level at most
static constexpr u64 kMidBits = 1ull << 24;  // bits of a level at most (4 MB of words)

static constexpr unsigned kMidPolls = 1u << 22;
unsigned g_mid_polls = kMidPolls;
unsigned g_mid_ctas = 0;  // CTAs of a launch (0: one a multiprocessor)

// All CTAs' threads wait here; false after `polls` looks, about a second (the
// status is raised and the launch winds down).
__device__ __forceinline__ bool grid_barrier(unsigned *bar, unsigned &round, unsigned polls,
                                             unsigned *status) {
  __shared__ int ok;
  __syncthreads();
  round++;
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    const unsigned want = round * gridDim.x;
    unsigned spin = 0;
    while (*(volatile unsigned *)bar < want && spin < polls) {
      __nanosleep(20);
      spin++;
    }
    ok = spin < polls;
    if (!ok) atomicOr(status, ST_TIMEOUT);
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

__global__ void __launch_bounds__(kMidThreads, 2)
k_mid(const u64 *__restrict__ keys0, FastMeta *__restrict__ meta, int dlim, FastCfg cfg) {
  extern __shared__ __align__(16) unsigned char smem[];
  u64 *keys = reinterpret_cast<u64 *>(smem);
  __shared__ int t_level;
  __shared__ unsigned s_cnt, s_ones;
  __shared__ u64 s_m, s_seed, s_nn, s_at;
  const unsigned tid = threadIdx.x, lane = tid & 31;
  if (tid == 0) {
    int t = -1;
    if (!*(volatile unsigned *)&meta->status)
      for (int d = 0; d <= dlim && d < (int)cfg.L; d++)
        if (meta->lv[d].mode == LM_MID) {
          t = d;
          break;
        }
    t_level = t;
  }
  __syncthreads();
  // the same decision in every CTA: nothing writes these records before the
  // first grid barrier
  int d = t_level;
  if (d < 0) return;
  u64 n = meta->lv[d].n, off = meta->lv[d].off, m = meta->lv[d].m;
  const u64 per = (n + gridDim.x - 1) / gridDim.x;
  const u64 lo = min(n, per * blockIdx.x);
  unsigned c = (unsigned)min(per, n - lo);  // this CTA's keys
  if (d == 0) {
    stage_keys<kMidThreads>(keys0 + lo, c, keys, [](u64 v) { return v; });
  } else {
    const u64 s_b = level_seed(cfg.seed, d - 1);
    stage_keys<kMidThreads>(cfg.F + lo, c, keys,
                                           [=](u64 v) { return unmix64(v) ^ s_b; });
  }
  // words [w0, w1) of a level are this CTA's to clear and to write out
  auto share = [&](u64 words, u64 &w0, u64 &w1) {
    const u64 step = (words + gridDim.x - 1) / gridDim.x;
    w0 = min(words, step * blockIdx.x);
    w1 = min(words, w0 + step);
  };
  u64 w0, w1;
  share(m >> 6, w0, w1);
  for (u64 w = w0 + tid; w < w1; w += kMidThreads)
    reinterpret_cast<ulonglong2 *>(cfg.AC[d & 1])[w] = make_ulonglong2(0, 0);
  unsigned round = 0;
  if (tid == 0) s_seed = level_seed(cfg.seed, d);
  if (!grid_barrier(&meta->bar, round, cfg.polls, &meta->status)) return;
  for (;;) {
    const u64 s = s_seed;
    const unsigned m32 = (unsigned)m;
    u64 *AC = cfg.AC[d & 1];
    auto at = [&](u64 x) { return reduce_range32(mix64(x ^ s), m32); };
    constexpr unsigned U = 8;
    for (unsigned i0 = tid; i0 < c; i0 += U * kMidThreads) {
      unsigned p[U];
      u64 old[U];
#pragma unroll
      for (unsigned u = 0; u < U; u++) {
        const unsigned i = i0 + u * kMidThreads;
        p[u] = i < c ? at(keys[i]) : 0;
        old[u] = i < c ? atomicOr(AC + (p[u] >> 5), 1ull << (p[u] & 31)) : 0;
      }
#pragma unroll
      for (unsigned u = 0; u < U; u++)
        if ((old[u] >> (p[u] & 31)) & 1ull) atomicOr(AC + (p[u] >> 5), 1ull << (32 + (p[u] & 31)));
    }
    if (tid == 0) s_cnt = s_ones = 0;
    if (!grid_barrier(&meta->bar, round, cfg.polls, &meta->status)) return;
    // keep the keys whose bit is not a lone hit; a chunk is read before any of
    // it is written, and what is written lies before what is still to be read
    for (unsigned i0 = 0; i0 < c; i0 += U * kMidThreads) {
      u64 x[U];
      unsigned keep = 0, mine = 0;
#pragma unroll
      for (unsigned u = 0; u < U; u++) {
        const unsigned i = i0 + u * kMidThreads + tid;
        x[u] = i < c ? keys[i] : 0;
        const unsigned p = at(x[u]) , b = p & 31;
        const u64 w = i < c ? __ldcg(AC + (p >> 5)) : 0;
        if (i < c && !(((w >> b) & 1ull) && !((w >> (32 + b)) & 1ull))) keep |= 1u << u;
      }
      mine = __popc(keep);
      unsigned pre = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned v = __shfl_up_sync(0xffffffffu, pre, o);
        if (lane >= (unsigned)o) pre += v;
      }
      __syncthreads();  // the chunk is read
      unsigned base = 0;
      if (lane == 31 && pre) base = atomicAdd(&s_cnt, pre);
      unsigned to = __shfl_sync(0xffffffffu, base, 31) + pre - mine;
#pragma unroll
      for (unsigned u = 0; u < U; u++)
        if ((keep >> u) & 1u) keys[to++] = x[u];
      __syncthreads();
    }
    // A_d, and the other array cleared
    u64 *Alev = (d == 0) ? cfg.A0 : cfg.arena + ((off - cfg.m0) >> 6);
    const bool fits = d == 0 || ((off - cfg.m0) >> 6) + (m >> 6) <= cfg.arena_words;
    unsigned ones = 0;
    share(m >> 6, w0, w1);
    for (u64 w = w0 + tid; w < w1; w += kMidThreads) {
      const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(AC) + w);
      const unsigned a0 = v.x & ~v.y, a1 = v.z & ~v.w;
      if (fits) Alev[w] = ((u64)a1 << 32) | a0;
      ones += __popc(a0) + __popc(a1);
      reinterpret_cast<ulonglong2 *>(cfg.AC[(d + 1) & 1])[w] = make_ulonglong2(0, 0);
    }
    ones = __reduce_add_sync(0xffffffffu, ones);
    if (lane == 0 && ones) atomicAdd(&s_ones, ones);
    __syncthreads();
    c = s_cnt;
    if (tid == 0) {
      if (c) atomicAdd(&meta->n_out[d], (u64)c);
      if (s_ones) atomicAdd(&meta->lv[d].weight, (u64)s_ones);
      if (!fits) atomicOr(&meta->status, ST_OVERFLOW);
    }
    if (!grid_barrier(&meta->bar, round, cfg.polls, &meta->status)) return;
    if (tid == 0) {
      const u64 nn = __ldcg(&meta->n_out[d]);
      s_nn = nn;
      s_m = nn && (uint32_t)(d + 1) < cfg.L ? level_bits(nn, cfg.gamma) : 0;
      s_seed = level_seed(cfg.seed, d + 1);
    }
    __syncthreads();
    const u64 nn = s_nn;
    const bool last = !fits || nn <= cfg.T || (uint32_t)(d + 1) == cfg.L;
    if (blockIdx.x == 0 && tid == 0) {
      FLevel &lv = meta->lv[d], &nx = meta->lv[d + 1];
      if (__ldcg(&lv.weight) + nn != n) atomicOr(&meta->status, ST_INTERNAL);
      lv.mode = LM_BUCKETED;
      lv.m = m;
      nx.n = nn;
      nx.off = off + m;
      nx.m = s_m;
      nx.mode = nn == 0 ? LM_DONE : last ? LM_FLAT : LM_BUCKETED;
      if (nn == 0) meta->levels_used = d + 1;
    }
    off += m;
    n = nn;
    m = s_m;
    d++;
    if (last) break;
  }
  // what is left goes to F as values of the last level, for the tail
  if (n == 0 || c == 0) return;
  const u64 s_l = level_seed(cfg.seed, d - 1);
  if (tid == 0) s_at = atomicAdd(&meta->n_mid, (u64)c);
  __syncthreads();
  for (unsigned i = tid; i < c; i += kMidThreads)
    if (s_at + i < cfg.F_cap) cfg.F[s_at + i] = mix64(keys[i] ^ s_l);
}

// ---------------------------------------------------------------------------
// Tail of the bucketed build: finds the first level (<= dlim) whose keys were
// sent to the flat buffer and runs the remaining levels there (cta_levels).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kTailThreads, 1)
k_tail(FastMeta *__restrict__ meta, int dlim, FastCfg cfg, u64 mcap) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int t_level;
  if (meta->status || meta->tail_done) return;
  if (threadIdx.x == 0) {
    int t = -1;
    for (int d = 0; d <= dlim && d <= (int)cfg.L; d++) {
      const unsigned md = meta->lv[d].mode;
      if (md == LM_FLAT || md == LM_DONE) {
        t = d;
        break;
      }
      if (md != LM_BUCKETED) break;
    }
    t_level = t;
  }
  __syncthreads();
  const int t = t_level;
  if (t < 0) return;  // not reached yet: the host enqueues more levels
  FLevel *lvs = meta->lv;
  if (lvs[t].mode == LM_DONE) {
    if (threadIdx.x == 0) meta->tail_done = 1;
    return;
  }
  const u64 n = lvs[t].n;
  if (threadIdx.x == 0 && t > 0 && meta->n_out[t - 1] != n) atomicOr(&meta->status, ST_INTERNAL);
  if ((uint32_t)t == cfg.L && n > kTailMaxKeys) {
    // large fallback: sorted on the host side of the build (sort.cu)
    if (threadIdx.x == 0) {
      meta->n_fb = n;
      meta->levels_used = cfg.L;
      meta->tail_done = 2;
    }
    return;
  }
  TailSmem sm = carve_tail(smem, mcap, cfg.T);
  // F holds the values of the level before (at t = 0 the caller's keys)
  const u64 s_b = t > 0 ? level_seed(cfg.seed, t - 1) : 0;
  stage_keys<kTailThreads>(
      cfg.F, (unsigned)n, sm.keys, [=](u64 v) { return t > 0 ? unmix64(v) ^ s_b : v; });
  __syncthreads();
  unsigned used = cta_levels<kTailThreads, (int)kTailMaxKeys>(
      sm, n, t, lvs[t].off, lvs, cfg.gamma, cfg.L, cfg.seed, cfg.A0,
                             cfg.arena, cfg.m0, cfg.arena_words, cfg.F, &meta->n_fb,
                             &meta->status);
  if (threadIdx.x == 0) {
    meta->levels_used = used;
    meta->tail_done = 1;
  }
}

// ---------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------
static DeviceOnce g_attrs;
double g_cap_scale = 1.0;

using SplitFn = void (*)(const u64 *, u64, FastMeta *, int, FastCfg, unsigned);
static SplitFn split_fn(unsigned nb_max, bool first) {
  if (nb_max <= (unsigned)kWT) return first ? k_split<1, true> : k_split<1, false>;
  return first ? k_split<2, true> : k_split<2, false>;
}

using GsplitFn = void (*)(const u64 *, u64, u64, unsigned, u64, unsigned, u64 *, u64, u64 *,
                          unsigned *);
template <int NT>
static GsplitFn gsplit_nt(bool first, bool narrow) {
  if (first) return narrow ? k_gsplit<NT, true, true> : k_gsplit<NT, true, false>;
  return narrow ? k_gsplit<NT, false, true> : k_gsplit<NT, false, false>;
}
static GsplitFn gsplit_fn(int nt, bool first, bool narrow) {
  return nt == kWT ? gsplit_nt<kWT>(first, narrow) : gsplit_nt<kWT / 2>(first, narrow);
}
using FsplitFn = void (*)(const u64 *, const u64 *, u64, unsigned, unsigned, unsigned, u64, u64 *,
                          u64, u64 *, unsigned *);
static FsplitFn fsplit_fn(int nt, bool narrow) {
  if (nt == kWT) return narrow ? k_fsplit<kWT, true> : k_fsplit<kWT, false>;
  return narrow ? k_fsplit<kWT / 2, true> : k_fsplit<kWT / 2, false>;
}

static int set_attrs() {
  for (int v = 0; v < 4; v++)
    MPHF_CUDA(cudaFuncSetAttribute(split_fn(v & 1 ? kWMaxNb : 1, (v & 2) != 0),
                                   cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wc_smem(1)));
  MPHF_CUDA(cudaFuncSetAttribute(k_fill_compact, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)fill_smem(kPmax)));
  for (int v = 0; v < 8; v++) {
    const int nt = v & 4 ? kWT : kWT / 2;
    MPHF_CUDA(cudaFuncSetAttribute(gsplit_fn(nt, v & 1, v & 2),
                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)wc_smem(kWT / nt)));
    MPHF_CUDA(cudaFuncSetAttribute(fsplit_fn(nt, v & 1),
                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)wc_smem(kWT / nt)));
  }
  MPHF_CUDA(cudaFuncSetAttribute(k_gfill<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)fill_smem(1ull << kGroupShift)));
  MPHF_CUDA(cudaFuncSetAttribute(k_gfill<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)fill_smem(1ull << kGroupShift)));
  MPHF_CUDA(cudaFuncSetAttribute(k_mid, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(kMidKeys * 8)));
  MPHF_CUDA(cudaFuncSetAttribute(k_tail, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kTailSmemMax));
  return MPHF_OK;
}

// One split launch of (at most) n values into at most nb_max buckets.
static void launch_split(const u64 *keys, u64 n, FastMeta *meta, int d, const FastCfg &cfg,
                         unsigned nb_max, cudaStream_t st) {
  const unsigned g = grid_for(n, kWT, (unsigned)sm_count());
  LaunchScope ls("split", st);
  split_fn(nb_max, d == 0)<<<g, kWT, wc_smem(1), st>>>(keys, n, meta, d, cfg, nb_max);
}

// Expected |F_{d+1}| from |F_d| (a key is alone with probability (1 - 1/m)^(n-1)).
static double expect_next(double n, double gamma) {
  const double m = (double)level_bits((u64)n, gamma);
  return n * (1.0 - pow(1.0 - 1.0 / m, n - 1.0));
}

struct FastScratch {
  DevBuf meta, X, cnt, F, A0, arena, T, AC;
  void release(cudaStream_t s) {
    dev_free(meta, s); dev_free(X, s); dev_free(cnt, s); dev_free(F, s);
    dev_free(A0, s); dev_free(arena, s); dev_free(T, s); dev_free(AC, s);
  }
};

// Level 1's bucket arena, allocated before level 0 runs: slots for any level
// size the device may pick for |F_1| <= n1_hi = E|F_1| + 10 sqrt(N) + 256
// (|F_1| has a standard deviation below sqrt(N)).  With B <= Bb buckets of
// cap = cap_scale (mean + 8 sqrt(mean) + 64) slots, the means summing to at
// most n + P, B cap <= cap_scale (n + P + 8 sqrt(B (n + P)) + 64 B) + 16 B.
static u64 level1_bound(u64 N, double gamma, u64 Btarget, u64 Pmax, double cap_scale,
                        u64 *n1_hi_out, u64 *Bb_out) {
  const double ev1 = expect_next((double)N, gamma);  // E|F_1|
  u64 n1_hi = (u64)ceil(ev1 + 10.0 * sqrt((double)N) + 256.0);
  if (n1_hi > N) n1_hi = N;
  const u64 m1_hi = level_bits(n1_hi, gamma);
  u64 Bb = ceil_div(m1_hi, Pmax);
  if (Bb < Btarget) Bb = Btarget;
  const double tot = (double)(n1_hi + Pmax);
  *n1_hi_out = n1_hi;
  *Bb_out = Bb;
  return (u64)(cap_scale * (tot + 8.0 * sqrt((double)Bb * tot) + 64.0 * (double)Bb)) + 16 * Bb + 64;
}

// Slots of a bucket that expects `mean` values.
static u64 group_cap(double mean, double cap_scale) {
  const u64 cap = (u64)(cap_scale * (mean + 8.0 * sqrt(mean) + 64.0));
  return (cap + 15) & ~15ull;
}

// Levels [0, ...) of a build whose level 0 has more than kGroupMinB buckets:
// runs every level that large, one host round trip per level, and leaves hm
// with the records of those levels and of the first level after them, whose
// values are in cfg.F.  *first receives that level's number.
static int grouped_levels(const u64 *keys, u64 N, const FastCfg &cfg, FastMeta *meta,
                          FastMeta *hm, FastScratch &sc, int *first, cudaStream_t st) {
  u64 n = N, off = 0;
  int d = 0;
  for (;; d++) {
    const u64 m = level_bits(n, cfg.gamma);
    FLevel &lv = hm->lv[d];
    if (d > 0 && ceil_div(m, cfg.Pmax) <= kGroupMinB) break;
    lv.n = n;
    lv.m = m;
    lv.off = off;
    lv.mode = LM_BUCKETED;
    const unsigned cs = coarse_shift(m), nf = 1u << (cs - kGroupShift), batch = kBatchFine / nf;
    const unsigned nc = (unsigned)ceil_div(m, 1ull << cs);
    const u64 cap_c = group_cap((double)n * (double)(1ull << cs) / (double)m, cfg.cap_scale);
    const u64 cap_f =
        group_cap((double)n * (double)(1ull << kGroupShift) / (double)m, cfg.cap_scale);
    u64 *cnt_c = (u64 *)sc.cnt.p, *cnt_f = cnt_c + kWMaxNb;
    if (nc > (unsigned)kWT || nc * cap_c > cfg.capX || (u64)kBatchFine * cap_f * 8 > sc.T.bytes) {
      hm->status = ST_OVERFLOW;  // redone by the unbucketed path, like any bound exceeded
      break;
    }
    MPHF_CUDA(cudaMemsetAsync(cnt_c, 0, kWMaxNb * 8, st));
    const bool narrow = (m >> 32) == 0;
    const u64 s_d = level_seed(cfg.seed, d);
    {
      LaunchScope ls("split_coarse", st);
      const int nt = wc_threads(nc);
      gsplit_fn(nt, d == 0, narrow)<<<(unsigned)(sm_count() * (kWT / nt)), nt, wc_smem(kWT / nt),
                                      st>>>(
          d == 0 ? keys : cfg.F, n, m, cs, d == 0 ? s_d : s_d ^ level_seed(cfg.seed, d - 1), nc,
          cnt_c, cap_c, cfg.X, &meta->status);
    }
    u64 *Alev = d == 0 ? cfg.A0 : cfg.arena + ((off - cfg.m0) >> 6);
    for (unsigned s0 = 0; s0 < nc; s0 += batch) {
      const unsigned ns = nc - s0 < batch ? nc - s0 : batch;
      MPHF_CUDA(cudaMemsetAsync(cnt_f, 0, (size_t)ns * nf * 8, st));
      const int nt = wc_threads(nf);
      const unsigned per = (unsigned)(sm_count() * (kWT / nt)) / ns;
      {
        LaunchScope ls("split_fine", st);
        fsplit_fn(nt, narrow)<<<ns * per, nt, wc_smem(kWT / nt), st>>>(
            cfg.X, cnt_c, cap_c, s0, ns, nf, m, cnt_f, cap_f, (u64 *)sc.T.p, &meta->status);
      }
      FillArgs a;
      a.X = (const u64 *)sc.T.p;
      a.cnt = cnt_f;
      a.cap = cap_f;
      a.m = m;
      a.P = 1ull << kGroupShift;
      a.p0 = (u64)s0 << cs;
      a.B = ceil_div(std::min((u64)ns << cs, m - a.p0), a.P);
      a.A = Alev;
      a.F = cfg.F;
      a.F_cap = cfg.F_cap;
      a.n_out = &meta->n_out[d];
      a.status = &meta->status;
      {
        LaunchScope ls("fill_grouped", st);
        (narrow ? k_gfill<true> : k_gfill<false>)<<<grid_for(a.B, 1, (unsigned)sm_count() * 2), kTT,
                                                    fill_smem(a.P), st>>>(
            a, &meta->lv[d].weight, &meta->seen[d]);
      }
    }
    MPHF_CUDA(cudaGetLastError());
    FastMeta got;
    MPHF_CUDA(cudaMemcpyAsync(&got, meta, sizeof(got), cudaMemcpyDeviceToHost, st));
    MPHF_CUDA(cudaStreamSynchronize(st));
    hm->status = got.status;
    if (got.status) break;
    lv.weight = got.lv[d].weight;
    hm->seen[d] = got.seen[d];
    hm->n_out[d] = got.n_out[d];
    if (got.seen[d] != n || lv.weight > n || got.n_out[d] != n - lv.weight) {
      hm->status = ST_INTERNAL;
      break;
    }
    n -= lv.weight;
    off += m;
    FLevel &nx = hm->lv[d + 1];
    nx.n = n;
    nx.off = off;
    if (n == 0) {
      nx.mode = LM_DONE;
      hm->levels_used = d + 1;
    } else if ((uint32_t)(d + 1) == cfg.L || n <= cfg.T) {
      nx.mode = LM_FLAT;
      if ((uint32_t)(d + 1) < cfg.L) nx.m = level_bits(n, cfg.gamma);
    } else if (n <= cfg.Tmid && level_bits(n, cfg.gamma) <= cfg.mmid) {
      nx.mode = LM_MID;
      nx.m = level_bits(n, cfg.gamma);
    } else {
      size_bucketed(nx, n, cfg.gamma, cfg.Pmin, cfg.Pmax, cfg.Btarget, cfg.cap_scale);
      nx.off = off;
      nx.mode = LM_BUCKETED;
      if (((off - cfg.m0) >> 6) + (nx.m >> 6) > cfg.arena_words) {
        hm->status = ST_OVERFLOW;
        break;
      }
    }
    if (nx.mode != LM_BUCKETED) {
      d++;
      break;
    }
  }
  *first = d;
  return MPHF_OK;
}

// Largest level size the tail may take for this gamma (keys, positions and two
// bit arrays in shared memory).
static u64 tail_limit(double gamma, u64 *mcap_out) {
  u64 T = kTailMaxKeys;
  while (T > 64) {
    u64 mc = level_bits(T, gamma);
    if (tail_smem_bytes(mc, T) <= kTailSmemMax) {
      *mcap_out = mc;
      return T;
    }
    T >>= 1;
  }
  *mcap_out = level_bits(64, gamma);
  return 64;
}

// k_mid on levels of at most n keys each, found by the device at levels <= dlim.
// false: the launch was refused (a context that owns fewer multiprocessors than
// the device reports cannot hold the grid).
static bool launch_mid(const u64 *keys, u64 n, FastMeta *meta, int dlim, const FastCfg &cfg,
                       cudaStream_t st) {
  LaunchScope ls("mid", st);
  const unsigned g = g_mid_ctas ? g_mid_ctas : (unsigned)sm_count();
  // Past 64 KB of keys a CTA asks for more than half a multiprocessor's shared
  // memory: two of 106 KB each landed on one (2e6 keys: 122 us, alone 96)
  size_t smem = (size_t)ceil_div(n, g) * 8;
  if (smem > 64 * 1024) smem = std::max(smem, (size_t)116 * 1024);
  void *args[] = {(void *)&keys, (void *)&meta, (void *)&dlim, (void *)&cfg};
  if (cudaLaunchCooperativeKernel((const void *)k_mid, dim3(g), dim3(kMidThreads), args, smem,
                                  st) == cudaSuccess)
    return true;
  cudaGetLastError();
  return false;
}

// Returns MPHF_OK with *fallback_needed = false on success; *fallback_needed =
// true (and nothing allocated) when a device-side bound was exceeded, or when
// there is no room for a grouped level's slabs.  use_mid = false: every level of
// more than T keys runs in buckets.
static int fast_build_levels(const u64 *keys, u64 N, double gamma, uint32_t L, u64 seed,
                             cudaStream_t st, mphf_t *h, bool *fallback_needed, KeyFeed *feed,
                             bool use_mid, bool *refused) {
  *fallback_needed = false;
  int rc = once_per_device(g_attrs, set_attrs);
  if (rc != MPHF_OK) return rc;
  u64 mcap = 0;
  const u64 T = tail_limit(gamma, &mcap);
  if (level_bits(T, gamma) > mcap) mcap = level_bits(T, gamma);
  FastScratch sc;
  FastCfg cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gamma = gamma;
  cfg.L = L;
  cfg.seed = seed;
  cfg.Bmax = kBmax;
  cfg.T = T;
  cfg.Pmin = 4096;
  cfg.Pmax = kPmax;
  cfg.Btarget = (u64)sm_count() * 4;
  cfg.cap_scale = g_cap_scale;
  cfg.polls = g_mid_polls;
  FastMeta hm;
  memset(&hm, 0, sizeof(hm));
  const u64 m0 = level_bits(N, gamma);
  cfg.m0 = m0;
  FastMeta *meta = nullptr;
  int dlim = 0;
  int D = 1;  // levels (from 0) launched before the first look at the device's progress
  // no room for the slabs of a grouped build: the unbucketed path can do with
  // less (it leaves the keys in their order), so it is asked
  bool redo_small = false;

#define FTRY(x)                    \
  do {                             \
    rc = (x);                      \
    if (rc != MPHF_OK) goto fail;  \
  } while (0)
#define FCUDA(x)                                        \
  do {                                                  \
    cudaError_t e_ = (x);                               \
    if (e_ != cudaSuccess) {                            \
      rc = cuda_fail(e_, #x);                           \
      goto fail;                                        \
    }                                                   \
  } while (0)

  // k_mid's reach (a shrunken bucket capacity, as tests set, keeps to buckets)
  if (use_mid && cfg.cap_scale == 1.0) {
    cfg.Tmid = std::min(kMidMax, (u64)sm_count() * kMidKeys);
    cfg.mmid = std::min(level_bits(cfg.Tmid, gamma), kMidBits);
    if (cfg.Tmid <= T) cfg.Tmid = 0;
  }
  FTRY(dev_alloc(sc.meta, sizeof(FastMeta), st));
  meta = (FastMeta *)sc.meta.p;
  FTRY(dev_alloc(sc.A0, m0 / 8, st));
  cfg.A0 = (u64 *)sc.A0.p;
  if (cfg.Tmid && N > T) {
    const u64 words = std::min(m0, cfg.mmid) / 32;
    FTRY(dev_alloc(sc.AC, 2 * words * 8, st));
    cfg.AC[0] = (u64 *)sc.AC.p;
    cfg.AC[1] = cfg.AC[0] + words;
  }
  if (N <= T) {
    // the whole function in one CTA
    hm.lv[0].n = N;
    hm.lv[0].m = m0;
    hm.lv[0].mode = LM_FLAT;
    FTRY(dev_alloc(sc.F, N * 8, st));
    cfg.F = (u64 *)sc.F.p;
    cfg.F_cap = N;
    u64 arena_words = (u64)(L > 1 ? L - 1 : 1) * (level_bits(N, gamma) / 64);
    FTRY(dev_alloc(sc.arena, arena_words * 8, st));
    cfg.arena = (u64 *)sc.arena.p;
    cfg.arena_words = arena_words;
    if (feed) FTRY(feed->ensure(N, st));
    FCUDA(cudaMemcpyAsync(cfg.F, keys, N * 8, cudaMemcpyDeviceToDevice, st));
    FCUDA(cudaMemcpyAsync(meta, &hm, sizeof(hm), cudaMemcpyHostToDevice, st));
    {
      LaunchScope ls("tail", st);
      k_tail<<<1, kTailThreads, tail_smem_bytes(mcap, T), st>>>(meta, 0, cfg, mcap);
    }
    FCUDA(cudaGetLastError());
  } else if (N <= cfg.Tmid && m0 <= cfg.mmid) {
    // every level in k_mid and the tail
    hm.lv[0].n = N;
    hm.lv[0].m = m0;
    hm.lv[0].mode = LM_MID;
    cfg.F_cap = N;
    FTRY(dev_alloc(sc.F, N * 8, st));
    cfg.F = (u64 *)sc.F.p;
    u64 n1_hi = 0, Bb = 0;
    level1_bound(N, gamma, cfg.Btarget, cfg.Pmax, cfg.cap_scale, &n1_hi, &Bb);
    cfg.arena_words = (u64)(L > 1 ? L - 1 : 1) * (level_bits(n1_hi, gamma) / 64);
    FTRY(dev_alloc(sc.arena, cfg.arena_words * 8, st));
    cfg.arena = (u64 *)sc.arena.p;
    if (feed) FTRY(feed->ensure(N, st));
    FCUDA(cudaMemcpyAsync(meta, &hm, sizeof(hm), cudaMemcpyHostToDevice, st));
    if (!launch_mid(keys, N, meta, 0, cfg, st)) {
      *refused = true;
      goto fail;
    }
    {
      LaunchScope ls("tail", st);
      k_tail<<<1, kTailThreads, tail_smem_bytes(mcap, T), st>>>(meta, (int)L, cfg, mcap);
    }
    FCUDA(cudaGetLastError());
    FCUDA(cudaMemcpyAsync(&hm, meta, sizeof(hm), cudaMemcpyDeviceToHost, st));
    FCUDA(cudaStreamSynchronize(st));
  } else {
    size_bucketed(hm.lv[0], N, gamma, cfg.Pmin, cfg.Pmax, cfg.Btarget, cfg.cap_scale);
    hm.lv[0].off = 0;
    hm.lv[0].mode = LM_BUCKETED;
    const bool grouped = hm.lv[0].B > kGroupMinB;
    if (grouped && ceil_div(m0, 1ull << coarse_shift(m0)) > (u64)kWT) {
      *fallback_needed = true;
      sc.release(st);
      return MPHF_OK;
    }
    // Levels past the first are sized on the device by the last CTA of the
    // level before; their buffers come from a bound on |F_1| so that no host
    // round trip sits between the levels.  |F_1| (keys not alone in their bin
    // at level 0) has mean N - N (1 - 1/m_0)^(N-1) and a standard deviation
    // below sqrt(N); the bound adds 10 of those, and level1_bound covers the
    // buckets of any level that small.  A level that does not fit anyway
    // (duplicate-heavy input) is caught on the device and the build is redone
    // by the unbucketed path.
    u64 n1_hi = 0, Bb = 0;
    const u64 cap1 = level1_bound(N, gamma, cfg.Btarget, cfg.Pmax, cfg.cap_scale, &n1_hi, &Bb);
    const u64 m1_hi = level_bits(n1_hi, gamma);
    cfg.capX = hm.lv[0].B * hm.lv[0].cap;
    redo_small = grouped;
    if (grouped) {
      // room for the slabs of level 0 or of any smaller level.  A level's keys per
      // position may exceed level 0's (both sizes are rounded up to whole words)
      // but not 1 / gamma; the one step more is for the rounding of the mean
      auto slots = [&](unsigned shift) {
        return group_cap((double)(1ull << shift) / gamma, cfg.cap_scale) + 16;
      };
      cfg.capX = 0;
      for (unsigned cs = kGroupShift; cs <= coarse_shift(m0); cs++)
        cfg.capX = std::max(cfg.capX, ceil_div(m0, 1ull << cs) * slots(cs));
      FTRY(dev_alloc(sc.T, (u64)kBatchFine * 8 * slots(kGroupShift), st));
    }
    if (cfg.capX < cap1) cfg.capX = cap1;
    FTRY(dev_alloc(sc.X, cfg.capX * 8, st));
    FTRY(dev_alloc(sc.cnt, (kWMaxNb + kBatchFine) * 8, st));
    cfg.X = (u64 *)sc.X.p;
    cfg.cnt = (u64 *)sc.cnt.p;
    cfg.F_cap = n1_hi < T ? T : n1_hi;
    FTRY(dev_alloc(sc.F, cfg.F_cap * 8, st));
    cfg.F = (u64 *)sc.F.p;
    cfg.arena_words = (u64)(L > 1 ? L - 1 : 1) * (m1_hi / 64);
    FTRY(dev_alloc(sc.arena, cfg.arena_words * 8, st));
    cfg.arena = (u64 *)sc.arena.p;
    // level 1 has the most keys of the levels >= 1, and a smaller level never
    // takes more than Btarget buckets (its width shrinks first), so Bb bounds
    // them all; the split checks it and falls back if ever exceeded
    const unsigned nb1 = (unsigned)(Bb < kBmax ? Bb : kBmax);
    {
      // predicted number of bucketed levels
      double e = expect_next((double)N, gamma);
      D = 1;
      // (a level within 2% of k_mid's reach may turn out larger)
      auto mid = [&](double x) {
        return 1.02 * x <= (double)cfg.Tmid && gamma * 1.02 * x <= (double)cfg.mmid - 64.0;
      };
      while (e > (double)T && !mid(e) && D < (int)L) {
        e = expect_next(e, gamma);
        D++;
      }
    }
    FCUDA(cudaMemsetAsync(sc.cnt.p, 0, kBmax * 8, st));
    FCUDA(cudaMemcpyAsync(meta, &hm, sizeof(hm), cudaMemcpyHostToDevice, st));
    if (grouped) {
      if (feed) FTRY(feed->ensure(N, st));
      FTRY(grouped_levels(keys, N, cfg, meta, &hm, sc, &dlim, st));
      // the device-driven loop goes on from here
      FCUDA(cudaMemsetAsync(sc.cnt.p, 0, kBmax * 8, st));
      FCUDA(cudaMemcpyAsync(meta, &hm, sizeof(hm), cudaMemcpyHostToDevice, st));
      if (D < dlim) D = dlim;
    } else {
      // Level-0 split.  Keys still arriving from the host are split one chunk
      // per launch as each chunk lands (the buckets' counters only grow, so
      // the launches compose).
      const u64 pstep = feed && feed->chunk ? feed->chunk : N;
      for (u64 c0 = 0; c0 < N; c0 += pstep) {
        const u64 cn = N - c0 < pstep ? N - c0 : pstep;
        if (feed) FTRY(feed->ensure(c0 + cn, st));
        launch_split(keys + c0, cn, meta, 0, cfg, (unsigned)hm.lv[0].B, st);
      }
    }
    const unsigned ctas = (unsigned)sm_count() * 2;
    for (int round = 0; round < 64; round++) {
      for (; dlim < D && dlim < (int)L; dlim++) {
        if (dlim > 0) launch_split(nullptr, n1_hi, meta, dlim, cfg, nb1, st);
        LaunchScope ls("fill_compact", st);
        k_fill_compact<<<dlim == 0 && hm.lv[0].B < ctas ? (unsigned)hm.lv[0].B : ctas, kTT,
                         fill_smem(dlim == 0 ? hm.lv[0].P : cfg.Pmax), st>>>(meta, dlim, cfg);
      }
      if (cfg.Tmid && !launch_mid(nullptr, cfg.Tmid, meta, dlim, cfg, st)) {
        *refused = true;
        goto fail;
      }
      {
        LaunchScope ls("tail", st);
        k_tail<<<1, kTailThreads, tail_smem_bytes(mcap, T), st>>>(meta, cfg.Tmid ? (int)L : dlim,
                                                                  cfg, mcap);
      }
      FCUDA(cudaGetLastError());
      FCUDA(cudaMemcpyAsync(&hm, meta, sizeof(hm), cudaMemcpyDeviceToHost, st));
      FCUDA(cudaStreamSynchronize(st));
      if (hm.status || hm.tail_done || dlim >= (int)L) break;
      D = dlim + 2;
    }
  }
  if (N <= T) {
    FCUDA(cudaMemcpyAsync(&hm, meta, sizeof(hm), cudaMemcpyDeviceToHost, st));
    FCUDA(cudaStreamSynchronize(st));
  }
  if (hm.status & ST_OVERFLOW) {
    *fallback_needed = true;
    sc.release(st);
    return MPHF_OK;
  }
  if (hm.status & ST_DUPLICATE) {
    rc = MPHF_EDUPLICATE;
    goto fail;
  }
  if (hm.status || !hm.tail_done) {
    rc = hm.status & ST_TIMEOUT ? MPHF_ETIMEOUT : MPHF_EINTERNAL;
    goto fail;
  }
  {
    // handle: level metadata, A = A_0 || arena, rank, fallback
    redo_small = false;
    const uint32_t used = hm.levels_used;
    if (used < 1 || used > L) {
      rc = MPHF_EINTERNAL;
      goto fail;
    }
    h->L_used = used;
    for (uint32_t d = 0; d < used; d++) {
      h->n[d] = hm.lv[d].n;
      h->m[d] = hm.lv[d].m;
      h->off[d] = hm.lv[d].off;
    }
    const u64 n_fb = (used == L) ? hm.lv[L].n : 0;
    h->n[used] = n_fb;
    h->n_fb = n_fb;
    h->M = h->off[used - 1] + h->m[used - 1];
    h->n_rank = (h->M + MPHF_RANK_BLOCK - 1) / MPHF_RANK_BLOCK;
    u64 placed = 0;
    for (uint32_t d = 0; d < used; d++) placed += hm.lv[d].weight;
    if (placed + n_fb != N) {
      rc = MPHF_EINTERNAL;
      goto fail;
    }
    // A = A_0 || (A_1 A_2 ... in the arena), stored as sectors with their ranks
    FTRY(make_sectors(h, ASrc{(const u64 *)sc.A0.p, m0 / 64, (const u64 *)sc.arena.p, h->M / 64},
                      &meta->rank_total, st));
    unsigned *dflag = &meta->dup;
    if (n_fb) {
      if (hm.tail_done == 2) {
        {
          LaunchScope ls("unhash", st);
          k_unhash<<<grid_for(n_fb, 256 * 4, (unsigned)sm_count() * 8), 256, 0, st>>>(
              cfg.F, n_fb, level_seed(seed, L - 1));
        }
        FTRY(sort_fallback(cfg.F, n_fb, dflag, st));
      }
      FTRY(dev_alloc(h->fb, n_fb * 8, st));
      FCUDA(cudaMemcpyAsync(h->fb.p, cfg.F, n_fb * 8, cudaMemcpyDeviceToDevice, st));
    }
    FCUDA(cudaMemcpyAsync(&hm, meta, sizeof(hm), cudaMemcpyDeviceToHost, st));
    FCUDA(cudaStreamSynchronize(st));
    if (hm.dup) {
      rc = MPHF_EDUPLICATE;
      goto fail;
    }
    if (hm.rank_total != N - n_fb) {
      rc = MPHF_EINTERNAL;
      goto fail;
    }
  }
  sc.release(st);
  return MPHF_OK;

fail:
  cudaGetLastError();
  sc.release(st);
  cudaStreamSynchronize(st);
  if (rc == MPHF_ENOMEM && redo_small) {
    *fallback_needed = true;
    return MPHF_OK;
  }
  return rc;
#undef FTRY
#undef FCUDA
}

int fast_build(const u64 *keys, u64 N, double gamma, uint32_t L, u64 seed, cudaStream_t st,
               mphf_t *h, bool *fallback_needed, KeyFeed *feed) {
  bool refused = false;
  const int rc = fast_build_levels(keys, N, gamma, L, seed, st, h, fallback_needed, feed, true,
                                   &refused);
  if (!refused) return rc;
  return fast_build_levels(keys, N, gamma, L, seed, st, h, fallback_needed, feed, false, &refused);
}

}  // namespace bbh

// Test hooks (host arithmetic only, no device work): the bucketed level size
// the device picks for n keys, and the level-1 arena bound of an N-key build.
extern "C" int mphf_debug_size_level(uint64_t n, double gamma, uint64_t btarget, uint64_t *B,
                                     uint64_t *cap, uint64_t *P) {
  if (!B || !cap || !P || !(gamma >= 1.0) || btarget == 0) return MPHF_EINVAL;
  bbh::FLevel lv;
  memset(&lv, 0, sizeof(lv));
  bbh::size_bucketed(lv, n, gamma, 4096, bbh::kPmax, btarget, 1.0);
  *B = lv.B;
  *cap = lv.cap;
  *P = lv.P;
  return MPHF_OK;
}

extern "C" int mphf_debug_level1_bound(uint64_t N, double gamma, uint64_t btarget,
                                       uint64_t *n1_hi, uint64_t *capY, uint64_t *Bb) {
  if (!n1_hi || !capY || !Bb || !(gamma >= 1.0) || btarget == 0) return MPHF_EINVAL;
  bbh::u64 nh = 0, bb = 0;
  *capY = bbh::level1_bound(N, gamma, btarget, bbh::kPmax, 1.0, &nh, &bb);
  *n1_hi = nh;
  *Bb = bb;
  return MPHF_OK;
}

extern "C" int mphf_debug_mid(int polls, uint32_t ctas) {
  bbh::g_mid_ctas = ctas;
  bbh::g_mid_polls = polls < 0 ? bbh::kMidPolls : (unsigned)polls;
  return MPHF_OK;
}
