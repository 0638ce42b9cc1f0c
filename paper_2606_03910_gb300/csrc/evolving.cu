// The greedy of Algorithm 1 (Sec. V-A) with evolving decode caches: the LRU-managed
// KV-block caches of the simulator of Sec. VI-B.  Each arrival's prefix hits are taken
// against the caches as they are at that arrival, and a dispatch brings the request's
// chain into the chosen decode's cache as its most recently used blocks (from the last
// block to the first, so that block 0 is the most recent), evicting the least recently
// used blocks beyond the cache's capacity.
//
// State of one cache (a decode of a stream), in caller-owned memory:
//   recency log   2^log2_ring block hashes; every use of a block appends it at the next
//                 position (positions only grow; entry p sits at p mod 2^log2_ring)
//   hash table    2^log2_slots slots {hash, latest position of the hash in the log}
//   header        head (the oldest position still in the cache), tail (the next
//                 position), live blocks, occupied slots
// A block is cached iff its latest position is at least head, and a use zeroes the log
// entry it supersedes, so the non-zero entries of the window [head, tail) are exactly the
// cached blocks at their latest uses:
//   lookup    one probe of the table and a comparison with head;
//   use       append at tail, raise the slot's position (atomicMax, so a hash that occurs
//             twice in a chain keeps its later use) and zero the superseded entry;
//   evict     advance head past as many non-zero entries as blocks to evict (a coalesced
//             scan of the log, no lookups).
// The table keeps evicted hashes (with old positions) until the log or the table fills;
// then the cache is rebuilt in place: the non-zero entries are packed in order from head
// and the table is rebuilt from them.
//
// One CTA per stream walks the stream's events in order:
//   departure  the first thread of the last warp returns the request's tokens to its
//              decode's load.  It alone writes loads, so departures need no barrier of
//              their own: those of an arrival separate its writes from the others' reads;
//   arrival    warps take decodes and find the first miss of the chain by following the
//              runs the chain's blocks form in the log (64 or 128 blocks a step); threads
//              take decodes and score them exactly as netkv_schedule_streams does without
//              a workspace (base score + w_load * theta * load), then a block-wide
//              (score, index) argmin; every thread then uses its share of the chain's
//              blocks on the chosen cache, and the CTA evicts in chunks of two log entries
//              a thread with a block scan over their liveness.
#include <math.h>

#include "score.cuh"

namespace {

constexpr int kLruBlock = 1024;
constexpr uint64_t kMaxChain = 65535;
constexpr uint64_t kHeaderBytes = 64;
constexpr uint32_t kNoDecode = 0xffffffffu;

struct __align__(16) LruSlot {
  unsigned long long key;  // block hash; 0 marks an empty slot
  unsigned long long pos;  // latest log position of the hash; 0 = none
};

struct LruHeader {
  unsigned long long head, tail, live, n_keys;
};

struct LruGeom {
  uint32_t log2_slots, log2_ring;
  unsigned long long cap_blocks;   // blocks a cache keeps
  unsigned long long max_keys;     // occupied slots allowed before a rebuild
  unsigned long long cache_bytes;  // bytes of one cache's state
};

__host__ __device__ inline unsigned long long lru_cache_bytes(uint32_t ls, uint32_t lr) {
  return kHeaderBytes + (16ull << ls) + (8ull << lr);
}

__device__ __forceinline__ char* lru_base(void* state, const LruGeom& g, uint64_t c) {
  return reinterpret_cast<char*>(state) + c * g.cache_bytes;
}
__device__ __forceinline__ LruHeader* lru_header(void* state, const LruGeom& g, uint64_t c) {
  return reinterpret_cast<LruHeader*>(lru_base(state, g, c));
}
__device__ __forceinline__ LruSlot* lru_slots(void* state, const LruGeom& g, uint64_t c) {
  return reinterpret_cast<LruSlot*>(lru_base(state, g, c) + kHeaderBytes);
}
__device__ __forceinline__ unsigned long long* lru_ring(void* state, const LruGeom& g,
                                                        uint64_t c) {
  return reinterpret_cast<unsigned long long*>(lru_base(state, g, c) + kHeaderBytes +
                                               (16ull << g.log2_slots));
}

// Table and log entries change during a kernel (atomics, in-place rebuilds), so they are
// read with volatile loads, never through the read-only path.
__device__ __forceinline__ unsigned long long vload(const unsigned long long* p) {
  return *reinterpret_cast<const volatile unsigned long long*>(p);
}

__device__ __forceinline__ ulonglong2 vload_slot(const LruSlot* p) {
  return __ldcg(reinterpret_cast<const ulonglong2*>(p));
}

// Latest log position of `key` (non-zero) in a cache's table, by the whole warp (kFind slots
// per step); 0 when the key is absent.
template <int kFind>
__device__ __forceinline__ unsigned long long lru_find(const LruSlot* T, uint32_t ls,
                                                       unsigned long long key, uint32_t lane,
                                                       int* status) {
  const unsigned long long n = 1ull << ls;
  const unsigned long long home = home_slot(key, ls);
  for (unsigned long long seen = 0; seen < n; seen += kFind) {
    ulonglong2 s = make_ulonglong2(~key, 0ull);
    if (lane < kFind) s = vload_slot(T + ((home + seen + lane) & (n - 1)));
    const uint32_t end = __ballot_sync(0xffffffffu, lane < kFind && (s.x == key || s.x == 0ull));
    if (end) {  // the first of them that holds the key or nothing decides
      const uint32_t at = __ffs(end) - 1;
      const bool found = __shfl_sync(0xffffffffu, s.x == key, at);
      const unsigned long long pos = __shfl_sync(0xffffffffu, s.y, at);
      return found ? pos : 0ull;
    }
  }
  if (lane == 0) flag_status(status, NETKV_DEV_EFULL);
  return 0ull;
}

// The slot of `key` (non-zero), claimed when the key is absent (fresh: claimed here).  kWide
// slots are read at a time: a walk that waits for one chain's blocks reads two (1, 2 and 4:
// 5.12, 4.93 and 5.19 ms of 300 arrivals on each of 32 streams), an initial fill and the walk
// of many streams, bound by the sectors they touch, one.
template <int kWide>
__device__ __forceinline__ LruSlot* lru_claim(LruSlot* T, uint32_t ls, unsigned long long key,
                                              bool& fresh, int* status) {
  fresh = false;
  const unsigned long long mask = (1ull << ls) - 1;
  const unsigned long long home = home_slot(key, ls);
  for (unsigned long long i = 0; i <= mask; i += kWide) {
    unsigned long long k[kWide];
#pragma unroll
    for (int q = 0; q < kWide; ++q) k[q] = vload(&T[(home + i + q) & mask].key);
#pragma unroll
    for (int q = 0; q < kWide; ++q) {
      LruSlot* slot = &T[(home + i + q) & mask];
      if (k[q] == key) return slot;
      if (k[q] == 0ull) {
        const unsigned long long prev = atomicCAS(&slot->key, 0ull, key);
        if (prev == 0ull) {
          fresh = true;
          return slot;
        }
        if (prev == key) return slot;
      }
    }
  }
  flag_status(status, NETKV_DEV_EFULL);
  return nullptr;
}

// Exclusive prefix count of `own` per thread over a CTA of BLOCK threads; the total goes to
// every thread.  Contains two block barriers.
template <int BLOCK>
__device__ __forceinline__ uint32_t block_count(uint32_t own, uint32_t* warp_buf, uint32_t& total) {
  constexpr uint32_t NW = BLOCK / 32;
  const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t in = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, in, o);
    if (lane >= (uint32_t)o) in += y;
  }
  if (lane == 31) warp_buf[wid] = in;
  __syncthreads();
  const uint32_t v = lane < NW ? warp_buf[lane] : 0u;
  const uint32_t before = __reduce_add_sync(0xffffffffu, lane < wid ? v : 0u);
  total = __reduce_add_sync(0xffffffffu, v);
  __syncthreads();
  return before + in - own;
}

// Record that log position p (already holding `key`) is the latest use of the key: raise
// the slot's position and zero the superseded log entry, which is p itself when a later
// use of the key in the same pass got there first, else the key's previous entry when it
// lies in the log window [head, tail).  So the non-zero entries of the window are exactly
// the cached blocks, each at its latest use.  Counts claimed slots and keys that were not
// cached before.
template <int kWide>
__device__ __forceinline__ void lru_use(LruSlot* T, unsigned long long* ring, const LruGeom& g,
                                        unsigned long long key, unsigned long long p,
                                        unsigned long long head, uint32_t& fresh_cnt,
                                        uint32_t& live_cnt, int* status) {
  const unsigned long long qmask = (1ull << g.log2_ring) - 1;
  bool fresh;
  LruSlot* slot = lru_claim<kWide>(T, g.log2_slots, key, fresh, status);
  if (!slot) {  // not indexed (a full table, flagged): the entry does not count as cached
    ring[p & qmask] = 0ull;
    return;
  }
  const unsigned long long old = atomicMax(&slot->pos, p);
  fresh_cnt += fresh;
  if (old > p) {
    ring[p & qmask] = 0ull;
  } else if (old >= head) {
    ring[old & qmask] = 0ull;
  } else {
    ++live_cnt;
  }
}

// A CTA's counts of lru_use into shared memory: one addition per warp.
__device__ __forceinline__ void add_counts(uint32_t fresh, uint32_t live, unsigned int* s_fresh,
                                           unsigned int* s_live) {
  fresh = __reduce_add_sync(0xffffffffu, fresh);
  live = __reduce_add_sync(0xffffffffu, live);
  if ((threadIdx.x & 31) == 0) {
    if (fresh) atomicAdd(s_fresh, fresh);
    if (live) atomicAdd(s_live, live);
  }
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// Leading chain blocks cached in one cache: the first miss among blocks [0, n), found by
// one warp.  The blocks of a chain that entered the cache together sit in the log as one
// run in reverse order (block j at the run's start position minus j), so the warp looks a
// block up in the table once and then compares 32 U chain blocks with the 32 U log entries
// below its position per step (coalesced), looking up again only where chain and log part.
// A log entry in the window that holds the block's hash is its latest use (the others
// are zero), so a match there is a cached block.
template <int U, int kFind>
__device__ __forceinline__ uint32_t lru_match(const LruSlot* T, const unsigned long long* ring,
                                              const LruGeom& g, unsigned long long head,
                                              const uint64_t* __restrict__ chain, uint32_t n,
                                              uint32_t lane, int* status) {
  const unsigned long long qmask = (1ull << g.log2_ring) - 1;
  uint32_t p = 0;
  unsigned long long rp = 0;  // log position of block p within the current run
  bool in_run = false;
  while (p < n) {
    const bool looked_up = !in_run;
    if (!in_run) {  // look block p up in the table
      const unsigned long long key = __ldg(chain + p);
      const unsigned long long pos =
          key != 0ull ? lru_find<kFind>(T, g.log2_slots, key, lane, status) : 0ull;
      if (pos == 0ull || pos < head) return p;  // absent or evicted
      rp = pos;
      in_run = true;
      // the log entries of the next steps into L2, a line a lane
      const unsigned long long ahead = 32ull * U + 16ull * lane;
      if (p + ahead < n && ahead <= rp - head) prefetch_l2(ring + ((rp - ahead) & qmask));
    }
    unsigned long long ck[U], rk[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t o = 32 * u + lane;
      ck[u] = 0ull;
      rk[u] = 1ull;
      if (p + o < n && rp >= head && (unsigned long long)o <= rp - head) {
        ck[u] = __ldg(chain + p + o);
        rk[u] = vload(ring + ((rp - o) & qmask));
      }
    }
    uint32_t lead = 32u * U;
#pragma unroll
    for (int u = U - 1; u >= 0; --u) {
      const uint32_t part = ~__ballot_sync(0xffffffffu, ck[u] != 0ull && ck[u] == rk[u]);
      if (part) lead = 32u * u + (uint32_t)(__ffs(part) - 1);
    }
    if (lead == 0) {
      if (looked_up) {  // the table's latest position does not hold the hash: inconsistent
        if (lane == 0) flag_status(status, NETKV_DEV_EFULL);
        return p;
      }
      in_run = false;  // the run ended with the last step: look block p up
      continue;
    }
    p += lead;
    rp -= lead;
    if (lead < 32u * U) in_run = false;
  }
  return n;
}

// (score, index) order with the runner-up carried along: lower score first, then lower
// decode rank (Algorithm 1 line 13).
__device__ __forceinline__ void take(float& b, uint32_t& i, float& s, float b2, uint32_t i2,
                                     float s2) {
  const bool other = (b2 < b) || (b2 == b && i2 < i);
  if (other) {
    s = fminf(s2, b);
    b = b2;
    i = i2;
  } else {
    s = fminf(s, b2);
  }
}
__device__ __forceinline__ void warp_take(float& b, uint32_t& i, float& s) {
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const float b2 = __shfl_xor_sync(0xffffffffu, b, o);
    const uint32_t i2 = __shfl_xor_sync(0xffffffffu, i, o);
    const float s2 = __shfl_xor_sync(0xffffffffu, s, o);
    take(b, i, s, b2, i2, s2);
  }
}

// Evict the `excess` least recently used blocks of a cache: advance head past that many
// non-zero log entries (a coalesced scan of the log, two entries a thread).  CTA-wide.
template <int BLOCK>
__device__ void lru_evict(const unsigned long long* ring, const LruGeom& g,
                          unsigned long long& head, unsigned long long tail,
                          unsigned long long excess, uint32_t* warp_buf,
                          unsigned long long* s_newhead, int* status) {
  const unsigned long long qmask = (1ull << g.log2_ring) - 1;
  unsigned long long p = head;
  while (excess > 0) {
    if (p >= tail) {  // fewer cached blocks than the header counts: an inconsistent state
      if (threadIdx.x == 0) flag_status(status, NETKV_DEV_EFULL);
      break;
    }
    const unsigned long long i = p + 2 * threadIdx.x;
    const bool live0 = i < tail && vload(ring + (i & qmask)) != 0ull;
    const bool live1 = i + 1 < tail && vload(ring + ((i + 1) & qmask)) != 0ull;
    uint32_t total;
    const uint32_t before =
        block_count<BLOCK>((live0 ? 1u : 0u) + (live1 ? 1u : 0u), warp_buf, total);
    if ((unsigned long long)total >= excess) {
      if (live0 && before + 1 == excess) *s_newhead = i + 1;
      if (live1 && before + (live0 ? 2 : 1) == excess) *s_newhead = i + 2;
      __syncthreads();
      p = *s_newhead;
      __syncthreads();
      excess = 0;
    } else {
      excess -= total;
      p += 2 * BLOCK;
    }
  }
  head = p;
}

// Rebuild a cache in place: pack the non-zero log entries of [head, tail) in order from
// head, then clear the table and insert them at their new positions.  Returns the number
// kept (the cached blocks).  CTA-wide.
template <int BLOCK>
__device__ unsigned long long lru_rebuild(LruSlot* T, unsigned long long* ring, const LruGeom& g,
                                          unsigned long long head, unsigned long long tail,
                                          uint32_t* warp_buf, int* status) {
  const unsigned long long qmask = (1ull << g.log2_ring) - 1;
  unsigned long long kept = 0;
  for (unsigned long long p = head; p < tail; p += BLOCK) {
    const unsigned long long i = p + threadIdx.x;
    const unsigned long long key = i < tail ? vload(ring + (i & qmask)) : 0ull;
    uint32_t total;
    const uint32_t before = block_count<BLOCK>(key != 0ull ? 1u : 0u, warp_buf, total);  // reads done
    // the write position never passes the entry's own: entries are only moved down
    if (key != 0ull) ring[(head + kept + before) & qmask] = key;
    kept += total;
    __syncthreads();
  }
  const unsigned long long n_slots = 1ull << g.log2_slots;
  for (unsigned long long s = threadIdx.x; s < n_slots; s += BLOCK)
    reinterpret_cast<ulonglong2*>(T)[s] = make_ulonglong2(0ull, 0ull);
  __syncthreads();
  for (unsigned long long i = threadIdx.x; i < kept; i += BLOCK) {
    const unsigned long long key = vload(ring + ((head + i) & qmask));
    bool fresh;
    LruSlot* slot = lru_claim<4>(T, g.log2_slots, key, fresh, status);
    if (slot) atomicMax(&slot->pos, head + i);
  }
  __syncthreads();
  return kept;
}

// Initial state of every cache from its key list (most recently used block first): entry
// j of a list of K blocks is used at position K - j, so the list's first block is the
// most recent.  One CTA per cache.
__global__ void __launch_bounds__(kLruBlock) lru_init_kernel(void* state, LruGeom g,
                                                            uint64_t n_caches,
                                                            const uint64_t* __restrict__ keys,
                                                            const uint64_t* __restrict__ key_off,
                                                            int* status) {
  __shared__ unsigned int s_fresh, s_live;
  const unsigned long long qmask = (1ull << g.log2_ring) - 1;
  const unsigned long long n_slots = 1ull << g.log2_slots;
  for (uint64_t c = blockIdx.x; c < n_caches; c += gridDim.x) {
    LruSlot* T = lru_slots(state, g, c);
    unsigned long long* ring = lru_ring(state, g, c);
    for (unsigned long long s = threadIdx.x; s < n_slots; s += kLruBlock)
      reinterpret_cast<ulonglong2*>(T)[s] = make_ulonglong2(0ull, 0ull);
    if (threadIdx.x == 0) {
      s_fresh = 0;
      s_live = 0;
    }
    __syncthreads();
    uint64_t beg = 0, K = 0;
    if (keys) {
      beg = __ldg(key_off + c);
      const uint64_t end = __ldg(key_off + c + 1);
      if (end < beg) {
        if (threadIdx.x == 0) flag_status(status, NETKV_DEV_ERANGE);
      } else {
        K = end - beg;
      }
      if (K > g.cap_blocks) {  // a list longer than the capacity: keep its first entries
        if (threadIdx.x == 0) flag_status(status, NETKV_DEV_ERANGE);
        K = g.cap_blocks;
      }
    }
    for (uint64_t j = threadIdx.x; j < K; j += kLruBlock) {
      const unsigned long long key = __ldg(keys + beg + j);
      ring[(K - j) & qmask] = key;
      if (key == 0ull) flag_status(status, NETKV_DEV_EDOMAIN);
    }
    __syncthreads();  // every entry is written before any is zeroed as superseded
    uint32_t fresh = 0, live = 0;
    for (uint64_t j = threadIdx.x; j < K; j += kLruBlock) {
      const unsigned long long key = __ldg(keys + beg + j);
      if (key != 0ull) lru_use<1>(T, ring, g, key, K - j, 1ull, fresh, live, status);
    }
    add_counts(fresh, live, &s_fresh, &s_live);
    __syncthreads();
    if (threadIdx.x == 0) {
      LruHeader* h = lru_header(state, g, c);
      h->head = 1;
      h->tail = K + 1;
      h->live = s_live;
      h->n_keys = s_fresh;
    }
    __syncthreads();
  }
}

// Every cache's blocks from the most to the least recently used: out[c][0 .. len[c]).
__global__ void __launch_bounds__(kLruBlock) lru_export_kernel(const void* state, LruGeom g,
                                                              uint64_t n_caches,
                                                              unsigned long long* out,
                                                              unsigned long long* out_len,
                                                              int* status) {
  __shared__ uint32_t warp_buf[kLruBlock / 32];
  const unsigned long long qmask = (1ull << g.log2_ring) - 1;
  void* st = const_cast<void*>(state);
  for (uint64_t c = blockIdx.x; c < n_caches; c += gridDim.x) {
    const LruHeader* h = lru_header(st, g, c);
    const unsigned long long head = vload(&h->head), tail = vload(&h->tail);
    const LruSlot* T = lru_slots(st, g, c);
    const unsigned long long* ring = lru_ring(st, g, c);
    unsigned long long* o_list = out + c * g.cap_blocks;
    unsigned long long w = 0;
    constexpr uint32_t kEach = 4;  // consecutive entries of a thread, newest first
    for (unsigned long long top = tail; top > head;) {
      const unsigned long long left = top - head;
      const unsigned long long chunk = left < kEach * kLruBlock ? left : kEach * kLruBlock;
      unsigned long long key[kEach];
      uint32_t n = 0;
#pragma unroll
      for (uint32_t u = 0; u < kEach; ++u) {
        const uint32_t o = kEach * threadIdx.x + u;
        key[u] = o < chunk ? vload(ring + ((top - 1 - o) & qmask)) : 0ull;
        n += key[u] != 0ull;  // the window's non-zero entries are the cached blocks
      }
      uint32_t total;
      unsigned long long at = w + block_count<kLruBlock>(n, warp_buf, total);
#pragma unroll
      for (uint32_t u = 0; u < kEach; ++u) {
        if (key[u] == 0ull) continue;
        if (at < g.cap_blocks) o_list[at] = key[u];
        ++at;
      }
      w += total;
      top -= chunk;
    }
    if (threadIdx.x == 0) {
      if (w > g.cap_blocks) flag_status(status, NETKV_DEV_EFULL);
      out_len[c] = w < g.cap_blocks ? w : g.cap_blocks;
    }
    __syncthreads();
  }
}

// One CTA of BLOCK threads per stream, kResident CTAs an SM.  Bound by the dependent round
// trips of an arrival (look-up and log comparison, claims and atomics of the chain's blocks,
// the eviction's scan), so every phase spreads over as many threads as the streams leave room
// for, and departures and the scores of small pools are taken by the last warp, whose loads
// overlap the others' match.  The wide forms read the next event's fields and fetch its chain
// into L2 an event ahead and read several slots at once; the narrow ones, whose SMs other
// streams keep busy, do neither, for fewer registers and sectors (760 streams x 60 arrivals at
// 5 CTAs an SM: 1,447 us, reading ahead 1,579).  32 streams x 300 arrivals on 8
// decodes of 60,000 blocks: 16 us an arrival, about 4 of them the match, 5 the chain's slots,
// 4 the eviction and the counts before it, 2 the scores; 35 us with 256 threads and 32 blocks
// a step (512 threads: 17).
template <int BLOCK, int kResident>
__global__ void __launch_bounds__(BLOCK, kResident) evolving_kernel(
    TopoArgs t, uint32_t n_streams, const netkv_weights* __restrict__ W, uint32_t R,
    const uint32_t* __restrict__ len, const uint32_t* __restrict__ prefill,
    const uint32_t* __restrict__ snap, const float* __restrict__ UB, uint32_t n_snap,
    const uint64_t* __restrict__ chains, const uint64_t* __restrict__ chain_off,
    const uint32_t* __restrict__ events, const uint64_t* __restrict__ event_off, void* state,
    LruGeom g, const int64_t* __restrict__ load_init, int32_t* dec, float* __restrict__ best,
    float* __restrict__ second, uint16_t* __restrict__ M, int64_t* __restrict__ load_final,
    int* status) {
  constexpr int NW = BLOCK / 32;
  constexpr bool kAhead = BLOCK >= 512;      // the next event is read ahead
  constexpr int kFind = BLOCK >= 512 ? 4 : 1;   // slots of a look-up read at a time
  constexpr int kClaim = BLOCK >= 512 ? 2 : 1;  // and of a claim
  constexpr int kStep = kResident < 6 ? 4 : 2;  // 32 chain blocks each, compared at a time
  constexpr uint32_t kNoEvent = 0xffffffffu;
  extern __shared__ __align__(16) unsigned char evo_smem[];
  __shared__ uint32_t warp_buf[NW];
  __shared__ float s_b[NW], s_s[NW];
  __shared__ uint32_t s_i[NW];
  __shared__ int32_t s_dstar;
  __shared__ unsigned int s_cnt[2];  // fresh slots, newly cached blocks
  __shared__ unsigned long long s_newhead;
  const uint32_t D = t.D, N = t.N;
  unsigned long long* s_head = reinterpret_cast<unsigned long long*>(evo_smem);
  unsigned long long* s_tail = s_head + D;
  unsigned long long* s_live = s_tail + D;
  unsigned long long* s_keys = s_live + D;
  long long* s_load = reinterpret_cast<long long*>(s_keys + D);
  uint32_t* s_m = reinterpret_cast<uint32_t*>(s_load + D);
  const uint32_t stream = blockIdx.x;
  if (stream >= n_streams) return;
  const uint32_t tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const unsigned long long qmask = (1ull << g.log2_ring) - 1;
  const unsigned long long Q = 1ull << g.log2_ring;
  const uint64_t c0_cache = (uint64_t)stream * D;
  for (uint32_t d = tid; d < D; d += BLOCK) {
    const LruHeader* h = lru_header(state, g, c0_cache + d);
    s_head[d] = vload(&h->head);
    s_tail[d] = vload(&h->tail);
    s_live[d] = vload(&h->live);
    s_keys[d] = vload(&h->n_keys);
    s_load[d] = load_init ? load_init[c0_cache + d] : 0;
  }
  __syncthreads();
  const netkv_weights w = W[stream];
  const float4 lat = make_float4(t.lat[0], t.lat[1], t.lat[2], t.lat[3]);
  const float inf = __int_as_float(0x7f800000);
  const uint64_t e0 = event_off[stream], e1 = event_off[stream + 1];

  // the next event's code and fields (zeros for what it has not)
  struct Fields {
    uint32_t code, l, pr, k;
    uint64_t c0, c1;
  };
  auto fields = [&](uint64_t e) -> Fields {
    Fields f = {kNoEvent, 0u, 0u, 0u, 0ull, 0ull};
    if (e >= e1) return f;
    f.code = __ldg(events + e);
    const uint32_t r = f.code & 0x7fffffffu;
    if (r >= R) return f;
    f.l = __ldg(len + r);
    if (f.code >> 31) return f;
    f.pr = __ldg(prefill + r);
    f.k = __ldg(snap + r);
    f.c0 = __ldg(chain_off + r);
    f.c1 = __ldg(chain_off + r + 1);
    return f;
  };
  Fields nf;
  if (kAhead) nf = fields(e0);
  for (uint64_t e = e0; e < e1; ++e) {
    const Fields f = kAhead ? nf : fields(e);
    if (kAhead) nf = fields(e + 1);
    const uint32_t code = f.code;
    const uint32_t r = code & 0x7fffffffu;
    if (r >= R) {
      if (tid == 0) flag_status(status, NETKV_DEV_ERANGE);
      continue;
    }
    if (code >> 31) {  // departure: the last warp's first thread returns the tokens
      if (tid == BLOCK - 32) {
        const int32_t dd = *reinterpret_cast<const volatile int32_t*>(dec + r);
        if (dd >= 0 && (uint32_t)dd < D) s_load[dd] -= (long long)f.l;
      }
      continue;
    }
    const uint32_t l = f.l, pr = f.pr, k = f.k;
    const uint64_t c0 = f.c0, c1 = f.c1;
    if (pr >= t.P || k >= n_snap || l == 0 || c1 < c0) {
      if (tid == 0) {
        flag_status(status, l == 0 ? NETKV_DEV_EDOMAIN : NETKV_DEV_ERANGE);
        best[r] = inf;
        second[r] = inf;
        dec[r] = -1;
      }
      for (uint32_t d = tid; d < D; d += BLOCK) M[(uint64_t)r * D + d] = 0;
      __syncthreads();
      continue;
    }
    uint64_t n = c1 - c0;
    if (n > kMaxChain) {
      if (tid == 0) flag_status(status, NETKV_DEV_EDOMAIN);
      n = kMaxChain;
    }
    const uint64_t* chain = chains + c0;

    // the scoring warps read what a score needs besides the hits before the match: all of
    // them, or for pools of at most 32 decodes the last warp alone
    const bool one_warp = D <= 32;
    const uint32_t sd = one_warp ? (wid == NW - 1 ? lane : D) : tid;  // its first decode
    const uint32_t pinst = __ldg(t.pre + pr);
    const float* ub_row = UB + (uint64_t)k * N * 4;
    const uint4 lp = __ldg(t.links + pinst);
    float ubp0 = 0.f, ubd0 = 0.f, lat0 = 0.f;
    if (sd < D) {
      const float4 ubp = __ldg(reinterpret_cast<const float4*>(UB) + (uint64_t)k * N + pinst);
      const uint4 ld = __ldg(t.links + __ldg(t.dec + sd));
      const int tau = tier_of(lp, ld);
      ubp0 = pick4(ubp, tau);
      lat0 = pick4(lat, tau);
      ubd0 = __ldg(ub_row + (uint64_t)ld.x * 4 + tau);
      if (one_warp) asm volatile("" : "+f"(ubp0), "+f"(ubd0));  // not read after the barrier
    }
    // the next arrival's chain into L2, a line a thread
    if (kAhead && !(nf.code >> 31) && nf.c1 > nf.c0) {
      const uint64_t at = (uint64_t)tid * 16;
      if (at < nf.c1 - nf.c0) prefetch_l2(chains + nf.c0 + at);
    }

    // hits against the caches as they are now (Sec. III-B first-miss scan)
    for (uint32_t d = wid; d < D; d += NW) {
      const uint32_t m = lru_match<kStep, kFind>(
          lru_slots(state, g, c0_cache + d), lru_ring(state, g, c0_cache + d), g, s_head[d], chain,
          (uint32_t)n, lane, status);
      if (lane == 0) {
        s_m[d] = m;
        M[(uint64_t)r * D + d] = (uint16_t)m;
      }
    }
    if (tid == 0) {
      s_cnt[0] = 0;
      s_cnt[1] = 0;
    }
    __syncthreads();

    // scores over the feasible decodes and the lowest-index argmin (lines 1-13)
    float b = inf, s2 = inf;
    uint32_t bi = kNoDecode;
    if (!one_warp || wid == NW - 1) {
      for (uint32_t d = sd; d < D; d += BLOCK) {
        float up = ubp0, ud = ubd0, la = lat0;
        if (d != sd) {
          const uint4 ld = __ldg(t.links + __ldg(t.dec + d));
          const int tau = tier_of(lp, ld);
          up = __ldg(ub_row + (uint64_t)pinst * 4 + tau);
          la = pick4(lat, tau);
          ud = __ldg(ub_row + (uint64_t)ld.x * 4 + tau);
        }
        const long long load = s_load[d];
        if (load + (long long)l <= w.cap_tokens) {
          const float sc = base_score(w, l, s_m[d], up, ud, la, status) +
                           w.w_load * (w.theta_s_per_token * (float)load);
          take(b, bi, s2, sc, d, inf);
        }
      }
      warp_take(b, bi, s2);
    }
    if (!one_warp) {
      if (lane == 0) {
        s_b[wid] = b;
        s_i[wid] = bi;
        s_s[wid] = s2;
      }
      __syncthreads();
      if (wid == NW - 1) {
        b = lane < (uint32_t)NW ? s_b[lane] : inf;
        bi = lane < (uint32_t)NW ? s_i[lane] : kNoDecode;
        s2 = lane < (uint32_t)NW ? s_s[lane] : inf;
        warp_take(b, bi, s2);
      }
    }
    if (tid == BLOCK - 32) {  // the thread that takes departures
      const int32_t d = bi == kNoDecode ? -1 : (int32_t)bi;
      dec[r] = d;
      best[r] = b;
      second[r] = s2;
      if (d >= 0) s_load[d] += (long long)l;
      s_dstar = d;
    }
    __syncthreads();
    const int32_t dstar = s_dstar;
    if (dstar < 0) continue;

    // the chain enters the chosen cache as its most recently used blocks
    const uint64_t cc = c0_cache + (uint32_t)dstar;
    LruSlot* T = lru_slots(state, g, cc);
    unsigned long long* ring = lru_ring(state, g, cc);
    if (s_tail[dstar] - s_head[dstar] + n > Q || s_keys[dstar] + n > g.max_keys) {
      const unsigned long long kept = lru_rebuild<BLOCK>(T, ring, g, s_head[dstar],
                                                         s_tail[dstar], warp_buf, status);
      if (tid == 0) {
        s_tail[dstar] = s_head[dstar] + kept;
        s_keys[dstar] = kept;
        s_live[dstar] = kept;
      }
      __syncthreads();
    }
    const unsigned long long P0 = s_tail[dstar], head = s_head[dstar];
    // what the eviction will scan (as many entries as the chain has blocks, if none is
    // cached), a line a thread
    if (16ull * tid < n && head + 16ull * tid < P0) prefetch_l2(ring + ((head + 16ull * tid) & qmask));
    for (uint64_t j = tid; j < n; j += BLOCK) {  // block j is used at P0 + n - 1 - j
      const unsigned long long key = __ldg(chain + j);
      ring[(P0 + (n - 1 - j)) & qmask] = key;
      if (key == 0ull) flag_status(status, NETKV_DEV_EDOMAIN);
    }
    __syncthreads();  // every entry is written before any is zeroed as superseded
    uint32_t fresh = 0, newly = 0;
    for (uint64_t j = tid; j < n; j += BLOCK) {
      const unsigned long long key = __ldg(chain + j);
      if (key != 0ull) lru_use<kClaim>(T, ring, g, key, P0 + (n - 1 - j), head, fresh, newly, status);
    }
    add_counts(fresh, newly, &s_cnt[0], &s_cnt[1]);
    __syncthreads();
    const unsigned long long tail = P0 + n;
    const unsigned long long live = s_live[dstar] + s_cnt[1];
    unsigned long long hd = head;
    if (live > g.cap_blocks)
      lru_evict<BLOCK>(ring, g, hd, tail, live - g.cap_blocks, warp_buf, &s_newhead, status);
    __syncthreads();  // every thread has read the counts that decide whether to evict
    if (tid == 0) {
      s_head[dstar] = hd;
      s_live[dstar] = live < g.cap_blocks ? live : g.cap_blocks;
      s_tail[dstar] = tail;
      s_keys[dstar] += s_cnt[0];
    }
    __syncthreads();
  }
  __syncthreads();  // the last departures are in s_load
  for (uint32_t d = tid; d < D; d += BLOCK) {
    LruHeader* h = lru_header(state, g, c0_cache + d);
    h->head = s_head[d];
    h->tail = s_tail[d];
    h->live = s_live[d];
    h->n_keys = s_keys[d];
    load_final[c0_cache + d] = s_load[d];
  }
}

bool lru_geom(const netkv_lru_config* cfg, LruGeom& g) {
  if (!cfg || cfg->cap_blocks < 1 || cfg->log2_slots < 4 || cfg->log2_slots > 31 ||
      cfg->log2_ring < 4 || cfg->log2_ring > 40)
    return false;
  g.log2_slots = cfg->log2_slots;
  g.log2_ring = cfg->log2_ring;
  g.cap_blocks = cfg->cap_blocks;
  g.max_keys = (3ull << cfg->log2_slots) / 4;
  g.cache_bytes = lru_cache_bytes(cfg->log2_slots, cfg->log2_ring);
  // after a rebuild the cache holds at most cap_blocks entries, and one chain must fit
  if ((1ull << cfg->log2_ring) < cfg->cap_blocks + kMaxChain + 1) return false;
  if (g.max_keys < cfg->cap_blocks + kMaxChain) return false;
  return true;
}

unsigned cache_grid(uint64_t n_caches) {
  return (unsigned)(n_caches < (1u << 20) ? n_caches : (1u << 20));
}

}  // namespace

extern "C" size_t netkv_lru_state_bytes(uint64_t n_caches, const netkv_lru_config* cfg) {
  LruGeom g;
  if (!lru_geom(cfg, g)) return 0;
  return (size_t)(n_caches * g.cache_bytes);
}

extern "C" netkv_status netkv_lru_init(void* d_state, size_t state_bytes, uint64_t n_caches,
                                       const netkv_lru_config* cfg, const uint64_t* d_keys,
                                       const uint64_t* d_key_off, int* d_status,
                                       netkv_stream_t stream) {
  LruGeom g;
  if (!d_state || !lru_geom(cfg, g) || (d_keys && !d_key_off)) return NETKV_EINVAL;
  if (state_bytes / g.cache_bytes < n_caches) return NETKV_EINVAL;
  if (!aligned_to(d_state, 16) || (d_keys && !aligned_to(d_keys, 8)) ||
      (d_key_off && !aligned_to(d_key_off, 8)))
    return NETKV_EINVAL;
  if (n_caches == 0) return NETKV_OK;
  lru_init_kernel<<<cache_grid(n_caches), kLruBlock, 0, (cudaStream_t)stream>>>(
      d_state, g, n_caches, d_keys, d_key_off, d_status);
  return netkv_launch_status();
}

extern "C" netkv_status netkv_lru_export(const void* d_state, size_t state_bytes,
                                         uint64_t n_caches, const netkv_lru_config* cfg,
                                         uint64_t* d_keys_out, uint64_t* d_len_out, int* d_status,
                                         netkv_stream_t stream) {
  LruGeom g;
  if (!d_state || !d_keys_out || !d_len_out || !lru_geom(cfg, g)) return NETKV_EINVAL;
  if (state_bytes / g.cache_bytes < n_caches) return NETKV_EINVAL;
  if (!aligned_to(d_state, 16) || !aligned_to(d_keys_out, 8) || !aligned_to(d_len_out, 8))
    return NETKV_EINVAL;
  if (n_caches == 0) return NETKV_OK;
  lru_export_kernel<<<cache_grid(n_caches), kLruBlock, 0, (cudaStream_t)stream>>>(
      d_state, g, n_caches, reinterpret_cast<unsigned long long*>(d_keys_out),
      reinterpret_cast<unsigned long long*>(d_len_out), d_status);
  return netkv_launch_status();
}

extern "C" netkv_status netkv_schedule_streams_evolving(
    netkv_topology_t topo, uint32_t n_streams, const netkv_weights* d_w, uint32_t R,
    const uint32_t* d_len, const uint32_t* d_prefill, const uint32_t* d_snap, const float* d_UB,
    uint32_t n_snap, const uint64_t* d_chains, const uint64_t* d_chain_off,
    const uint32_t* d_events, const uint64_t* d_event_off, void* d_state, size_t state_bytes,
    const netkv_lru_config* cfg, const int64_t* d_load_init, int32_t* d_dec, float* d_best,
    float* d_second, uint16_t* d_M, int64_t* d_load_final, int* d_status,
    netkv_stream_t stream) {
  LruGeom g;
  if (!topo || !d_w || !d_event_off || !d_load_final || !d_state || !lru_geom(cfg, g))
    return NETKV_EINVAL;
  if (n_streams == 0) return NETKV_OK;
  if (n_streams > 0x7fffffffu) return NETKV_EINVAL;
  if (R > 0 && (!d_len || !d_prefill || !d_snap || !d_UB || !d_chains || !d_chain_off ||
                !d_events || !d_dec || !d_best || !d_second || !d_M))
    return NETKV_EINVAL;
  if (!aligned_to(d_w, 8) || !aligned_to(d_UB, 16) || !aligned_to(d_event_off, 8) ||
      !aligned_to(d_load_final, 8) || !aligned_to(d_state, 16) ||
      (d_load_init && !aligned_to(d_load_init, 8)) || (d_chains && !aligned_to(d_chains, 8)) ||
      (d_chain_off && !aligned_to(d_chain_off, 8)) || (d_M && !aligned_to(d_M, 2)))
    return NETKV_EINVAL;
  const TopoArgs t = topo_args(topo);
  if (t.D > 1024) return NETKV_EINVAL;
  if (state_bytes / g.cache_bytes < (uint64_t)n_streams * t.D) return NETKV_EINVAL;
  const size_t smem = (size_t)t.D * (4 * 8 + 8 + 4);
  int dev = 0, sms = 0;
  NETKV_CUDA_TRY(cudaGetDevice(&dev));
  NETKV_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
#define NETKV_EVOLVE(BLOCK, RESIDENT)                                                          \
  evolving_kernel<BLOCK, RESIDENT><<<n_streams, BLOCK, smem, (cudaStream_t)stream>>>(          \
      t, n_streams, d_w, R, d_len, d_prefill, d_snap, d_UB, n_snap, d_chains, d_chain_off,     \
      d_events, d_event_off, d_state, g, d_load_init, d_dec, d_best, d_second, d_M,            \
      d_load_final, d_status)
  // As many threads per stream as keep every stream resident: 1, 2, 4 and 6 CTAs an SM by the
  // launch bounds.  60 arrivals of 4,096 tokens a stream on 8 decodes (us; 1,024 threads / 512 /
  // 256 by 4 / 256 by 6): 152 streams 761 / 778 / 948 / 1,023, 153 1,244 / 773 / 922 / -, 304
  // 1,531 / 938 / 1,130 / 1,229, 456 2,166 / 1,536 / 1,207 / 1,286, 608 2,852 / 1,706 / 1,293 /
  // 1,361, 760 3,527 / 2,276 / 1,861 / 1,486, 1,024 4,765 / 2,941 / 2,043 / 2,217, 1,824 8,235 /
  // 4,661 / 3,186 / 2,948.
  const uint32_t per_sm = (n_streams + (uint32_t)sms - 1) / (uint32_t)sms;
  if (per_sm <= 1) NETKV_EVOLVE(1024, 1);
  else if (per_sm <= 2) NETKV_EVOLVE(512, 2);
  else if (per_sm <= 4) NETKV_EVOLVE(256, 4);
  else NETKV_EVOLVE(256, 6);
#undef NETKV_EVOLVE
  return netkv_launch_status();
}
