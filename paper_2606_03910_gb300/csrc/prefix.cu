// Decode caches K_d and the block-level prefix hit of Sec. III-B:
// M[r][d] = |LCP_block(h_r, K_d)|, the number of leading blocks of request r's hash chain
// that are all cached on decode d.
//
// Cache index.  The caches of a table set are indexed per group of up to 64 decodes:
//   run keys    the group's distinct cached hashes in the order the key lists give them
//               (decode by decode, first appearance);
//   run masks   beside each run key, the mask of the group's decodes that cache it, in
//               1, 2, 4 or 8 bytes by the pool's size;
//   hash table  open addressing, 16-byte slots {hash, position in the run array}.
// Caches are filled with whole prefixes of chains, so a cached prefix sits in the run
// array as a contiguous run in chain order.
// The build numbers the distinct hashes of an index by their first position in its lists
// (see "Cache build" below).
//
// Match.  One warp per (request, decode group).  The warp looks up the block at the
// current position in the hash table (one random access), then compares the chain with
// the run keys from that position on, 128 blocks per step (coalesced loads of chain, key
// and mask bytes): every block that equals the next run key is cached exactly on the
// decodes of that position's mask.  A step whose blocks all match and are cached on every
// live decode costs one vote; otherwise ballots find each decode's first missing block.
// Where chain and run part, the next block is looked up in the hash table again; a block
// absent from the table is missing on every decode.  The answer never depends on the run
// order (any key order is exact); the order only decides how many lookups a chain needs.
// A decode leaves once its first miss is known and the warp stops when every decode of the
// group has missed.
//   match_kernel: pools of one decode group (D <= 64), and any pool without a workspace.
//
// Prefix sharing.  Requests that share leading blocks have the same membership answers on
// those blocks, so for pools of several groups, whose every group would read the chain
// again, a match with a workspace runs in three steps:
//   group_scan_kernel: every chain is followed through the run keys of its set's first
//     index (no masks), which gives how many of its blocks that group caches at all.
//     Requests are grouped by (table set, first block hash) in an open-addressing table, and
//     each group's leader is the chain with the most such blocks (then the longest, then the
//     lowest index): the one whose cached prefix the others' are prefixes of.
//   group_resolve_kernel: leaders go to a compact list; a member r with leader L gets
//     lcp = |common prefix of h_r and h_L| from the runs that both chains followed, without
//     reading them again (exactly, unless both left the same last run at the same block).
//   match_leaders_kernel: leaders (and ungrouped requests) run the full match, one task
//     per (leader, decode group) taken in order from a counter.
//   match_members_wide_kernel: one warp per member.  For a decode with M_L[d] < lcp the
//     first missing block of L lies inside the common prefix, so M_r[d] = M_L[d] exactly;
//     otherwise blocks [0, lcp) are all cached.  So the member's row is min(M_L, lcp)
//     elementwise, and block lcp is probed only in the groups where a leader hit reaches
//     lcp, up to 32 groups at a time.  The result equals the full match whatever the
//     grouping.
#include <algorithm>
#include <type_traits>

#include "cache_index.cuh"

namespace {

constexpr int kBuildBlock = 1024;
constexpr int kMatchBlock = 256;
constexpr int kDirectBlock = 64;
constexpr uint32_t kNoRun = 0xffffffffu;  // no run position (they are at most 2^31)
// Exclusive scan of one flag per thread over a 1024-thread block; returns the prefix and
// writes the block total to *total (shared).
__device__ __forceinline__ uint32_t block_scan(uint32_t flag, uint32_t* warp_sums,
                                               uint32_t* total) {
  const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t b = __ballot_sync(0xffffffffu, flag);
  const uint32_t in_warp = __popc(b & ((1u << lane) - 1));
  if (lane == 0) warp_sums[wid] = __popc(b);
  __syncthreads();
  if (wid == 0) {
    const uint32_t v = warp_sums[lane];
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= (uint32_t)o) x += y;
    }
    warp_sums[lane] = x - v;  // exclusive
    if (lane == 31) *total = x;
  }
  __syncthreads();
  return warp_sums[wid] + in_warp;
}

// ---- Cache build -------------------------------------------------------------------
// The lists of an index's decodes, one after another, are its elements 0 .. T - 1.  A hash's
// run position is the number of distinct hashes that appear before it, so cached prefixes
// stay contiguous.  Every pass is parallel over the elements or slots of all indices:
//   insert  each element claims its hash's slot and keeps the first position there
//           (atomicMax on its complement, since a cleared slot holds 0), unless it is seen
//           to repeat an earlier element: a warp looks one hash up and follows the list
//           from its first position;
//   mark    each occupied slot sets the bit of its first position in a bitmap of T bits,
//           which borrows the index's run masks;
//   count   one block per index: how many bits are set before every 256 of them, at the
//           end of the index's run keys, and the number of distinct hashes n;
//   place   each occupied slot takes its position's rank as its run position and writes
//           its run key;
//   wipe    the bitmap and the counts are cleared;
//   masks   each element adds its decode's bit to its hash's run mask; a warp looks one
//           hash up and follows the run for the next ones.
// Bound by random accesses to the slots (one sector per lane and probe), which stay in L2
// where the blocks in flight cover few indices: kPartsMax blocks per index keep them so.
// 256 decodes of 50,000 keys (4 indices, 12.8 M elements): 0.28 ms, insert 0.125 and masks
// 0.060 of it; one block per index walking its lists in chunks of 1,024 took 14.85 ms.
// An index whose lists are too long for the borrowed memory (T over 8 bits per mask byte,
// lists that repeat hashes many times) or whose table is nearly full is built by
// build_serial_kernel instead: one block walks the lists in chunks.  So are all indices of a
// call on small ones (serial_build), where seven launches or the passes over the slots cost more.
struct GroupLists {
  uint64_t pre[kGroup + 1];  // elements before each decode's list
  uint64_t beg[kGroup];      // where the list starts in the keys
  bool in_order;             // the lists follow one another in the keys
};
constexpr int kPassBlock = 256;
constexpr uint32_t kPartsMax = 512;

struct BuildArgs {
  void* index;
  uint64_t n_index;
  uint32_t D, log2_cap, parts;
  const uint64_t* keys;
  const uint64_t* key_off;
  int* status;
};

// The lists of index idx, by the whole block; ends with a barrier.
__device__ __forceinline__ void load_lists(GroupLists& L, const BuildArgs& a, uint64_t idx,
                                           bool report) {
  const uint32_t n_dgroups = (a.D + kGroup - 1) / kGroup;
  const uint64_t g = idx / n_dgroups;
  const uint32_t q0 = (uint32_t)(idx - g * n_dgroups) * kGroup;
  const uint32_t ng = min(kGroup, a.D - q0);
  __syncthreads();  // the lists of the index before are no longer read
  if (threadIdx.x < 32) {
    const uint32_t lane = threadIdx.x;
    uint64_t len[2];
    bool bad = false;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t j = 2 * lane + h;
      len[h] = 0;
      if (j < ng) {
        const uint64_t t = g * a.D + q0 + j;
        const uint64_t beg = __ldg(a.key_off + t), end = __ldg(a.key_off + t + 1);
        if (end >= beg) len[h] = end - beg;
        else bad = true;
        L.beg[j] = beg;
      }
    }
    if (bad && report) flag_status(a.status, NETKV_DEV_ERANGE);
    const bool any_bad = __any_sync(0xffffffffu, bad);
    uint64_t x = len[0] + len[1];
    const uint64_t own = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= (uint32_t)o) x += y;
    }
    L.pre[2 * lane] = x - own;
    L.pre[2 * lane + 1] = x - own + len[0];
    if (lane == 31) L.pre[kGroup] = x;
    if (lane == 0) L.in_order = !any_bad;
  }
  __syncthreads();
}

// Words of the counts of an index: one per 256 elements, then n; they end the run keys.
__device__ __forceinline__ uint64_t count_words(uint64_t T) { return (T + 255) / 256 + 1; }
__device__ __forceinline__ uint32_t* build_counts(const IndexView& v, uint64_t cap, uint64_t T) {
  return reinterpret_cast<uint32_t*>(v.keys + cap) - count_words(T);
}
// Whether the bitmap fits the masks, and the counts the run keys.
__device__ __forceinline__ bool lists_fit(uint64_t T, uint64_t cap, uint32_t mask_bytes) {
  return T <= 8u * mask_bytes * cap && count_words(T) <= 2 * cap;
}
__device__ __forceinline__ bool counts_fit(uint64_t n, uint64_t T, uint64_t cap) {
  return 2 * n + count_words(T) <= 2 * cap;
}

__global__ void __launch_bounds__(kPassBlock) build_insert_kernel(BuildArgs a) {
  __shared__ GroupLists L;
  const uint64_t cap = 1ull << a.log2_cap, mask = cap - 1;
  const uint32_t mb = mask_bytes_of(a.D), lane = threadIdx.x & 31;
  constexpr uint32_t kRow = 64;
  for (uint64_t b = blockIdx.x; b < a.n_index * a.parts; b += gridDim.x) {
    const uint64_t idx = b / a.parts;
    const uint32_t part = (uint32_t)(b - idx * a.parts);
    load_lists(L, a, idx, part == 0);
    const uint64_t T = L.pre[kGroup];
    if (!lists_fit(T, cap, mb)) continue;
    IndexSlot* hash = index_view(a.index, idx, a.log2_cap, mb).hash;
    // the key of element e, e < T
    auto key_of = [&](uint64_t e) -> unsigned long long {
      if (L.in_order) return __ldg(a.keys + L.beg[0] + e);
      uint32_t d = 0;
      while (e >= L.pre[d + 1]) ++d;
      return __ldg(a.keys + L.beg[d] + (e - L.pre[d]));
    };
    // warps take kRow consecutive elements; the warps of all blocks pass over the lists
    // together, so that most elements meet an earlier list's entries in the table (rows of
    // 32, 64, 128 and 256 elements: 135, 125, 126 and 132 us)
    for (uint64_t row = (uint64_t)part * (kPassBlock / 32) + (threadIdx.x >> 5); row * kRow < T;
         row += (uint64_t)a.parts * (kPassBlock / 32)) {
      uint64_t f = kNotFound;  // an earlier element that may equal lane 0's
      for (uint64_t e0 = row * kRow; e0 < min(T, (row + 1) * kRow); e0 += 32) {
        const uint64_t e = e0 + lane;
        const unsigned long long key = e < T ? key_of(e) : 0ull;
        if (e < T && key == 0ull) flag_status(a.status, NETKV_DEV_EDOMAIN);
        if (f == kNotFound) {
          if (lane == 0 && key != 0ull) {
            uint64_t slot = home_slot(key, a.log2_cap);
            for (uint64_t step = 0; step < cap; ++step) {
              const ulonglong2 s = __ldcg(reinterpret_cast<const ulonglong2*>(hash + slot));
              if (s.x == key && s.y != 0ull) f = ~s.y;
              if (s.x == key || s.x == 0ull) break;
              slot = (slot + 1) & mask;
            }
          }
          f = __shfl_sync(0xffffffffu, f, 0);
        }
        // an element that repeats an earlier one needs no slot: the earlier one, or the
        // first of its kind, takes care of it
        const bool repeat = f < e0 && key != 0ull && key_of(f + lane) == key;
        if (key != 0ull && !repeat) {
          uint64_t slot = home_slot(key, a.log2_cap);
          bool placed = false;
          for (uint64_t step = 0; step < cap; ++step) {
            const ulonglong2 s = __ldcg(reinterpret_cast<const ulonglong2*>(hash + slot));
            unsigned long long k = s.x;
            if (k == 0ull) {
              const unsigned long long prev = atomicCAS(&hash[slot].key, 0ull, key);
              k = prev == 0ull ? key : prev;
            }
            if (k == key) {
              if (s.x != key || s.y < ~e) atomicMax(&hash[slot].pos, (unsigned long long)~e);
              placed = true;
              break;
            }
            slot = (slot + 1) & mask;
          }
          if (!placed) flag_status(a.status, NETKV_DEV_EFULL);
        }
        f = __ballot_sync(0xffffffffu, repeat) >> 31 ? f + 32 : kNotFound;
      }
    }
  }
}

__global__ void __launch_bounds__(kPassBlock) build_mark_kernel(BuildArgs a) {
  __shared__ GroupLists L;
  const uint64_t cap = 1ull << a.log2_cap;
  const uint32_t mb = mask_bytes_of(a.D);
  for (uint64_t b = blockIdx.x; b < a.n_index * a.parts; b += gridDim.x) {
    const uint64_t idx = b / a.parts;
    const uint32_t part = (uint32_t)(b - idx * a.parts);
    load_lists(L, a, idx, false);
    if (!lists_fit(L.pre[kGroup], cap, mb)) continue;
    const IndexView v = index_view(a.index, idx, a.log2_cap, mb);
    uint32_t* bits = reinterpret_cast<uint32_t*>(v.masks);
    for (uint64_t s = (uint64_t)part * kPassBlock + threadIdx.x; s < cap;
         s += (uint64_t)a.parts * kPassBlock) {
      const ulonglong2 x = __ldcg(reinterpret_cast<const ulonglong2*>(v.hash + s));
      if (x.x != 0ull) atomicOr(bits + (~x.y >> 5), 1u << (uint32_t)(~x.y & 31u));
    }
  }
}

// Bits set in the 256-bit group i of a bitmap.  The bitmap starts on a 16-byte boundary, and
// its last group lies inside the index: masks and padding, cleared past the last element.
__device__ __forceinline__ uint32_t bits_of(const uint4* __restrict__ bits, uint64_t i) {
  const uint4 x = __ldcg(bits + 2 * i), y = __ldcg(bits + 2 * i + 1);
  return __popc(x.x) + __popc(x.y) + __popc(x.z) + __popc(x.w) + __popc(y.x) + __popc(y.y) +
         __popc(y.z) + __popc(y.w);
}

__global__ void __launch_bounds__(kBuildBlock) build_count_kernel(BuildArgs a) {
  __shared__ GroupLists L;
  __shared__ uint32_t warp_sums[2][32];
  const uint64_t cap = 1ull << a.log2_cap;
  const uint32_t mb = mask_bytes_of(a.D), lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (uint64_t idx = blockIdx.x; idx < a.n_index; idx += gridDim.x) {
    load_lists(L, a, idx, false);
    const uint64_t T = L.pre[kGroup];
    if (!lists_fit(T, cap, mb)) continue;
    const IndexView v = index_view(a.index, idx, a.log2_cap, mb);
    uint32_t* counts = build_counts(v, cap, T);
    const uint4* bits = reinterpret_cast<const uint4*>(v.masks);
    const uint64_t groups = (T + 255) / 256;
    uint32_t before = 0;  // bits of the chunks before; n < 2^32 (at most 2^31 slots)
    uint32_t parity = 0;
    uint32_t next = threadIdx.x < groups ? bits_of(bits, threadIdx.x) : 0u;
    for (uint64_t c = 0; c < groups; c += kBuildBlock) {
      const uint32_t own = next;
      const uint64_t i = c + threadIdx.x, in_next = i + kBuildBlock;
      next = in_next < groups ? bits_of(bits, in_next) : 0u;
      uint32_t in = own;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, in, o);
        if (lane >= (uint32_t)o) in += y;
      }
      if (lane == 31) warp_sums[parity][wid] = in;
      __syncthreads();  // one barrier a chunk: the sums are double-buffered
      const uint32_t w = warp_sums[parity][lane];
      const uint32_t below = __reduce_add_sync(0xffffffffu, lane < wid ? w : 0u);
      if (i < groups) counts[i] = before + below + in - own;
      before += __reduce_add_sync(0xffffffffu, w);
      parity ^= 1u;
    }
    if (threadIdx.x == 0) counts[groups] = before;
  }
}

__global__ void __launch_bounds__(kPassBlock) build_place_kernel(BuildArgs a) {
  __shared__ GroupLists L;
  const uint64_t cap = 1ull << a.log2_cap;
  const uint32_t mb = mask_bytes_of(a.D);
  for (uint64_t b = blockIdx.x; b < a.n_index * a.parts; b += gridDim.x) {
    const uint64_t idx = b / a.parts;
    const uint32_t part = (uint32_t)(b - idx * a.parts);
    load_lists(L, a, idx, false);
    const uint64_t T = L.pre[kGroup];
    if (!lists_fit(T, cap, mb)) continue;
    const IndexView v = index_view(a.index, idx, a.log2_cap, mb);
    const uint32_t* counts = build_counts(v, cap, T);
    if (!counts_fit(__ldcg(counts + (T + 255) / 256), T, cap)) continue;
    const uint4* bits = reinterpret_cast<const uint4*>(v.masks);
    for (uint64_t s = (uint64_t)part * kPassBlock + threadIdx.x; s < cap;
         s += (uint64_t)a.parts * kPassBlock) {
      const ulonglong2 x = __ldcg(reinterpret_cast<const ulonglong2*>(v.hash + s));
      if (x.x == 0ull) continue;
      const uint64_t e = ~x.y;
      uint32_t rank = __ldcg(counts + (e >> 8));
      const uint4 lo = __ldcg(bits + (e >> 8) * 2), hi = __ldcg(bits + (e >> 8) * 2 + 1);
      const uint32_t word[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
      const uint32_t w = (uint32_t)(e >> 5) & 7u;  // the element's word in its group
      const uint32_t below = (1u << (uint32_t)(e & 31u)) - 1u;
#pragma unroll
      for (uint32_t j = 0; j < 8; ++j)
        rank += __popc(word[j] & (j < w ? ~0u : j == w ? below : 0u));
      v.hash[s].pos = rank;
      v.keys[rank] = x.x;
    }
  }
}

__global__ void __launch_bounds__(kPassBlock) build_wipe_kernel(BuildArgs a) {
  __shared__ GroupLists L;
  const uint64_t cap = 1ull << a.log2_cap;
  const uint32_t mb = mask_bytes_of(a.D);
  for (uint64_t b = blockIdx.x; b < a.n_index * a.parts; b += gridDim.x) {
    const uint64_t idx = b / a.parts;
    const uint32_t part = (uint32_t)(b - idx * a.parts);
    load_lists(L, a, idx, false);
    const uint64_t T = L.pre[kGroup];
    if (!lists_fit(T, cap, mb)) continue;
    const IndexView v = index_view(a.index, idx, a.log2_cap, mb);
    uint32_t* counts = build_counts(v, cap, T);
    // another block may have cleared n already: 0 fits, and only an index that fits is
    // cleared
    if (!counts_fit(__ldcg(counts + (T + 255) / 256), T, cap)) continue;
    uint32_t* bits = reinterpret_cast<uint32_t*>(v.masks);
    const uint64_t words = (T + 31) / 32, all = words + count_words(T);
    for (uint64_t i = (uint64_t)part * kPassBlock + threadIdx.x; i < all;
         i += (uint64_t)a.parts * kPassBlock) {
      if (i < words) bits[i] = 0u;
      else counts[i - words] = 0u;
    }
  }
}

__global__ void __launch_bounds__(kPassBlock) build_masks_kernel(BuildArgs a) {
  __shared__ GroupLists L;
  const uint64_t cap = 1ull << a.log2_cap;
  const uint32_t mb = mask_bytes_of(a.D), lane = threadIdx.x & 31;
  constexpr uint32_t kRow = 256;  // consecutive elements a warp takes at a time
  for (uint64_t b = blockIdx.x; b < a.n_index * a.parts; b += gridDim.x) {
    const uint64_t idx = b / a.parts;
    const uint32_t part = (uint32_t)(b - idx * a.parts);
    load_lists(L, a, idx, false);
    const uint64_t T = L.pre[kGroup];
    if (!lists_fit(T, cap, mb)) continue;
    const IndexView v = index_view(a.index, idx, a.log2_cap, mb);
    if (__ldcg(build_counts(v, cap, T) + (T + 255) / 256) != 0u) continue;  // not cleared: serial
    uint32_t d = 0;
    const uint64_t n_warps = (uint64_t)a.parts * (kPassBlock / 32);
    for (uint64_t row = (uint64_t)part * (kPassBlock / 32) + (threadIdx.x >> 5);
         row * kRow < T; row += n_warps) {
      unsigned long long next = kNotFound;  // run position that lane 0's element may have
      for (uint64_t e0 = row * kRow; e0 < min(T, (row + 1) * kRow); e0 += 32) {
        const uint64_t e = e0 + lane;
        unsigned long long key = 0ull;
        if (e < T) {
          while (e >= L.pre[d + 1]) ++d;
          key = __ldcs(a.keys + L.beg[d] + (e - L.pre[d]));
        }
        if (next == kNotFound) {
          if (lane == 0 && key != 0ull) next = lookup(v.hash, key, a.log2_cap, a.status);
          next = __shfl_sync(0xffffffffu, next, 0);
        }
        unsigned long long pos = kNotFound;
        if (key != 0ull) {
          const unsigned long long at = next + lane;  // kNotFound + lane wraps: checked below
          if (next != kNotFound && at < cap && __ldg(v.keys + at) == key) pos = at;
          else pos = lookup(v.hash, key, a.log2_cap, a.status);
        }
        if (pos != kNotFound) run_mask_or(v, pos, 1ull << d);
        next = __shfl_sync(0xffffffffu, pos, 31);
        if (next != kNotFound) ++next;
      }
    }
  }
}

// The indices that the passes above left out, or all (kAll: no pass has run): one block each, the
// lists walked in order in chunks; new hashes are claimed by atomicCAS and numbered by a block
// scan.  Where a chunk repeats a hash that is new in it, another thread than the first may have
// claimed it: such an index (lists seldom repeat a hash) is built again, numbering every chunk
// by first elements, by a call out of line, so that the common path keeps its 32 registers.
constexpr unsigned long long kTentative = 1ull << 63;  // above every run position

// The lists of one index into it (cleared); kExact: by first elements in a chunk, else whether a
// chunk repeated a hash that was new in it goes to *repeated (shared).
template <bool kExact>
__device__ __forceinline__ void build_lists(const BuildArgs& a, uint64_t idx, uint32_t* warp_sums,
                                            uint32_t* chunk_new, int* repeated) {
  const uint32_t cap = 1u << a.log2_cap;  // at most 2^31
  const uint32_t n_dgroups = (a.D + kGroup - 1) / kGroup;
  const uint64_t g = idx / n_dgroups;
  const uint32_t q0 = (uint32_t)(idx - g * n_dgroups) * kGroup;
  const uint32_t ng = min(kGroup, a.D - q0);
  const uint64_t* off = a.key_off + g * a.D + q0;
  const IndexView v = index_view(a.index, idx, a.log2_cap, mask_bytes_of(a.D));
  IndexSlot* hash = v.hash;
  uint32_t run_len = 0;  // same value in every thread
  for (uint32_t d = 0; d < ng; ++d) {
    const uint64_t beg = __ldg(off + d), end = __ldg(off + d + 1);
    if (end < beg && threadIdx.x == 0) flag_status(a.status, NETKV_DEV_ERANGE);
    const unsigned long long bit = 1ull << d;
    for (uint64_t c = beg; c < end; c += kBuildBlock) {
      const uint64_t j = c + threadIdx.x;
      unsigned long long key = j < end ? __ldg(a.keys + j) : 0ull;
      if (j < end && key == 0ull) flag_status(a.status, NETKV_DEV_EDOMAIN);
      bool is_new = false, placed = false;
      uint32_t slot = 0;
      if (key != 0ull) {
        slot = (uint32_t)home_slot(key, a.log2_cap);
        for (uint32_t step = 0; step < cap; ++step) {
          const unsigned long long prev = atomicCAS(&hash[slot].key, 0ull, key);
          if (prev == 0ull || prev == key) {
            is_new = prev == 0ull;
            placed = true;
            break;
          }
          slot = (slot + 1) & (cap - 1);
        }
        if (!placed) flag_status(a.status, NETKV_DEV_EFULL);
      }
      if (kExact) {  // of the elements that share a hash new in this chunk, the first counts
        const unsigned long long own = kTentative | (kBuildBlock - 1 - threadIdx.x);
        if (is_new) atomicMax(&hash[slot].pos, own);
        __syncthreads();
        const bool again =
            placed && !is_new && *((volatile unsigned long long*)&hash[slot].pos) >= kTentative;
        if (again) atomicMax(&hash[slot].pos, own);
        __syncthreads();
        is_new = (is_new || again) && *((volatile unsigned long long*)&hash[slot].pos) == own;
      }
      const uint32_t pos = run_len + block_scan(is_new ? 1u : 0u, warp_sums, chunk_new);
      if (is_new) {
        hash[slot].pos = pos;
        v.keys[pos] = key;
        run_mask_or(v, pos, bit);  // masks share 32-bit words: set by atomics only
      }
      __syncthreads();
      if (placed && !is_new) {
        const uint64_t p = *((volatile unsigned long long*)&hash[slot].pos);
        run_mask_or(v, p, bit);
        if (!kExact && p >= run_len) *repeated = 1;
      }
      run_len += *chunk_new;
      __syncthreads();
    }
  }
}

__device__ __forceinline__ void clear_index(const BuildArgs& a, uint64_t idx) {
  const uint32_t mb = mask_bytes_of(a.D);
  uint4* w = reinterpret_cast<uint4*>(index_view(a.index, idx, a.log2_cap, mb).hash);
  for (uint64_t i = threadIdx.x; i < index_stride(a.log2_cap, mb) / 16; i += kBuildBlock)
    w[i] = make_uint4(0u, 0u, 0u, 0u);
}

__device__ __noinline__ void rebuild_exact(const BuildArgs& a, uint64_t idx, uint32_t* warp_sums,
                                           uint32_t* chunk_new) {
  clear_index(a, idx);
  __syncthreads();
  build_lists<true>(a, idx, warp_sums, chunk_new, nullptr);
}

template <bool kAll>
__global__ void __launch_bounds__(kBuildBlock, 2) build_serial_kernel(
    const __grid_constant__ BuildArgs a) {
  __shared__ uint32_t warp_sums[32];
  __shared__ uint32_t chunk_new;
  __shared__ int repeated;
  for (uint64_t idx = blockIdx.x; idx < a.n_index; idx += gridDim.x) {
    if (!kAll) {
      __shared__ GroupLists L;
      load_lists(L, a, idx, false);
      const uint64_t cap = 1ull << a.log2_cap, T = L.pre[kGroup];
      const uint32_t mb = mask_bytes_of(a.D);
      if (lists_fit(T, cap, mb)) {
        const IndexView v = index_view(a.index, idx, a.log2_cap, mb);
        if (__ldcg(build_counts(v, cap, T) + (T + 255) / 256) == 0u) continue;  // built
        __syncthreads();      // every thread has read the count
        clear_index(a, idx);  // the table was nearly full: start over
      }
    }
    if (threadIdx.x == 0) repeated = 0;
    __syncthreads();
    build_lists<false>(a, idx, warp_sums, &chunk_new, &repeated);
    if (repeated) rebuild_exact(a, idx, warp_sums, &chunk_new);
    __syncthreads();  // every thread has read `repeated`
  }
}

__device__ __forceinline__ int32_t find_set(const uint32_t* __restrict__ set_off, uint32_t n_sets,
                                            uint32_t r) {
  if (!set_off) return 0;
  if (r < __ldg(set_off) || r >= __ldg(set_off + n_sets)) return -1;
  uint32_t lo = 0, hi = n_sets;  // invariant: set_off[lo] <= r < set_off[hi]
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (__ldg(set_off + mid) <= r) lo = mid; else hi = mid;
  }
  return (int32_t)lo;
}

// Per-lane results of one decode group: lane j holds decodes j and j + 32.
struct GroupHits {
  uint32_t lo, hi;
};

__device__ __forceinline__ void set_hit(GroupHits& h, uint32_t lane, uint32_t j, uint32_t v) {
  if (j == lane) h.lo = v;
  if (j == lane + 32) h.hi = v;
}

// Every decode in `alive` misses at position v.
__device__ __forceinline__ void miss_all(GroupHits& h, uint32_t lane, unsigned long long alive,
                                         uint32_t v) {
  if ((alive >> lane) & 1ull) h.lo = v;
  if ((alive >> (lane + 32)) & 1ull) h.hi = v;
}

// Run position of `key` (non-zero) in one index, or kNotFound, by the whole warp: four
// consecutive slots (two sectors) per step, so that most probes take one round trip.
__device__ __forceinline__ unsigned long long lookup_warp(const IndexSlot* __restrict__ hash,
                                                          uint64_t key, uint32_t log2_cap,
                                                          uint32_t lane, int* status) {
  const uint64_t cap = 1ull << log2_cap;
  const uint64_t home = home_slot(key, log2_cap);
  for (uint64_t seen = 0; seen < cap; seen += 4) {
    ulonglong2 s = make_ulonglong2(~key, 0ull);
    if (lane < 4)
      s = __ldg(reinterpret_cast<const ulonglong2*>(hash + ((home + seen + lane) & (cap - 1))));
    const uint32_t end = __ballot_sync(0xffffffffu, lane < 4 && (s.x == key || s.x == 0ull));
    if (end) {  // the first of the four that holds the key or nothing decides
      const uint32_t at = __ffs(end) - 1;
      const bool found = __shfl_sync(0xffffffffu, s.x == key, at);
      const unsigned long long pos = __shfl_sync(0xffffffffu, s.y, at);
      return found ? pos : kNotFound;
    }
  }
  if (lane == 0) flag_status(status, NETKV_DEV_EFULL);
  return kNotFound;
}

template <int kMB>  // masks of at most 32 decodes are reduced as one word
using DecodeMask = std::conditional_t<kMB == 8, unsigned long long, uint32_t>;

// OR of one mask over the warp.
template <typename Mask>
__device__ __forceinline__ Mask warp_or(Mask m) {
  Mask a = __reduce_or_sync(0xffffffffu, (uint32_t)m);
  if (sizeof(Mask) == 8)
    a |= (Mask)((uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)((uint64_t)m >> 32)) << 32);
  return a;
}

// The decodes of nm[u] miss block p + 32 u + lane: the first miss of each counts, and the
// decode leaves `alive`.  A few decodes take a vote each per 32 blocks; more are settled by the
// blocks where some decode misses first (a prefix OR over the lanes), of which there are at most
// as many.  32,000 requests on 64 decodes whose hits end within 16 blocks: 59 us, 161 with votes
// over all blocks, 105 with votes over the 32 of the miss.  Up to 8 that miss in one step vote
// over all its blocks: 57 us from 3 up instead, but 24 streams of 4 requests on 42 decodes 20.8
// -> 21.4.
constexpr int kVotes = 6;
template <bool kMany, int N, typename Mask>
__device__ __forceinline__ void settle(const Mask (&nm)[N], uint32_t p, GroupHits& h, Mask& alive,
                                       uint32_t lane) {
  Mask m = nm[0];
#pragma unroll
  for (int u = 1; u < N; ++u) m |= nm[u];
  Mask a = warp_or(m);
  if (!a) return;  // usually
  if (!kMany || (N > 1 && __popcll((unsigned long long)a) <= 8)) {  // over all blocks at once
    alive &= ~a;
    while (a) {
      const uint32_t j = __ffsll((long long)a) - 1;
      a &= a - 1;
      uint32_t first = 0;
#pragma unroll
      for (int u = N - 1; u >= 0; --u) {
        const uint32_t miss = __ballot_sync(0xffffffffu, (uint32_t)(nm[u] >> j) & 1u);
        if (miss) first = 32u * u + (uint32_t)(__ffs(miss) - 1);
      }
      set_hit(h, lane, j, p + first);
    }
    return;
  }
#pragma unroll
  for (int u = 0; u < N; ++u) {
    const Mask own = (Mask)(nm[u] & alive);
    if (N > 1) {
      if (!__any_sync(0xffffffffu, own != 0)) continue;
      a = warp_or(own);
    }
    alive &= ~a;
    if (__popcll((unsigned long long)a) <= kVotes) {
      while (a) {
        const uint32_t j = __ffsll((long long)a) - 1;
        a &= a - 1;
        const uint32_t miss = __ballot_sync(0xffffffffu, (uint32_t)(own >> j) & 1u);
        set_hit(h, lane, j, p + 32u * u + (uint32_t)(__ffs(miss) - 1));
      }
      continue;
    }
    Mask in = own;  // the decodes that miss at this block or one before
#pragma unroll
    for (uint32_t o = 1; o < 32; o <<= 1) {
      const Mask y = __shfl_up_sync(0xffffffffu, in, o);
      if (lane >= o) in |= y;
    }
    const Mask up = __shfl_up_sync(0xffffffffu, in, 1);
    const Mask first = (Mask)(own & ~(lane ? up : (Mask)0));
    uint32_t at = __ballot_sync(0xffffffffu, first != 0);
    while (at) {
      const uint32_t l = __ffs(at) - 1;
      at &= at - 1;
      miss_all(h, lane, __shfl_sync(0xffffffffu, first, l), p + 32u * u + l);
    }
  }
}

// Where the lists are not in chain order: blocks from p on looked up 32 at a time, side by
// side, until the scan is done (p = n) or a run can be followed again from `run`.  A position
// counts only where the run array holds the block's hash, as when a run is followed.  Out of
// line, with its state by value, so that the common path keeps its registers.
template <int kMB>
struct SideScan {
  GroupHits h;
  DecodeMask<kMB> alive;
  uint32_t p, run;
};
template <int kMB>
__device__ __noinline__ SideScan<kMB> scan_side_by_side(const IndexSlot* __restrict__ hash,
                                                        const unsigned long long* __restrict__ keys,
                                                        const unsigned char* __restrict__ masks,
                                                        const uint64_t* __restrict__ chain,
                                                        uint32_t n, uint32_t log2_cap,
                                                        SideScan<kMB> s, int* status) {
  using Mask = DecodeMask<kMB>;
  const uint32_t lane = threadIdx.x & 31;
  IndexView ix;
  ix.masks = const_cast<unsigned char*>(masks);
  while (s.p < n && s.alive) {
    const uint32_t i = s.p + lane;
    const uint64_t key = i < n ? __ldcs(chain + i) : 0ull;
    unsigned long long pos = key != 0ull ? lookup(hash, key, log2_cap, status) : kNotFound;
    const bool corrupt = pos != kNotFound && (pos >> log2_cap || __ldg(keys + pos) != key);
    if (corrupt) pos = kNotFound;
    const uint32_t ok = __ballot_sync(0xffffffffu, pos != kNotFound);
    const uint32_t lead = ~ok ? (uint32_t)(__ffs(~ok) - 1) : 32u;
    const Mask nm[1] = {lane < lead ? (Mask)(s.alive & ~(Mask)run_mask<kMB>(ix, pos)) : (Mask)0};
    settle<(kMB > 2)>(nm, s.p, s.h, s.alive, lane);
    if (lead < 32u) {
      if (s.p + lead < n) {  // block p + lead is absent from every cache of the group
        if (lane == lead && s.alive && (corrupt || key == 0ull))
          flag_status(status, corrupt ? NETKV_DEV_EFULL : NETKV_DEV_EDOMAIN);
        miss_all(s.h, lane, s.alive, s.p + lead);
      }
      s.p = n;
      return s;
    }
    s.p += 32;
    const unsigned long long before = __shfl_up_sync(0xffffffffu, pos, 1);
    const uint32_t follows = __ballot_sync(0xffffffffu, lane > 0 && pos == before + 1);
    if (__popc(follows) >= 16) {  // in order here
      s.run = (uint32_t)__shfl_sync(0xffffffffu, pos, 31) + 1;
      return s;
    }
  }
  s.p = n;
  return s;
}

// First-miss scan of blocks [start, n) of one chain for the `alive` decodes of a group; n is at
// most 65,535.  Decodes found missing at position p get p; decodes never missing keep their
// value.  start_pos: the run position of block `start` when the caller has already looked it up.
// kMB: the run masks' width.  U: a step compares 32 * U chain blocks with the run; a wide step
// has more loads in flight per warp, but reads up to 32 * U - 1 blocks past the last one needed.
// Where a looked-up block's run ends at once (lists that are not in chain order) the next 32
// blocks are looked up side by side.  (Two runs of fewer than 32 blocks in a row taken for lists
// out of order: pieces of 4 blocks 2,105 -> 592 us, but lists of a dozen decodes in order, whose
// depths lie that close, 13.1 -> 16.1.)
template <int U, int kMB>
__device__ __forceinline__ void scan_chain(const IndexView& ix, uint32_t log2_cap,
                                           const uint64_t* __restrict__ chain, uint32_t start,
                                           uint32_t n, unsigned long long alive_decodes,
                                           GroupHits& h, uint32_t lane, int* status,
                                           unsigned long long start_pos = kNotFound) {
  using Mask = DecodeMask<kMB>;
  const uint32_t cap = 1u << log2_cap;  // at most 2^31
  Mask alive = (Mask)alive_decodes;
  uint32_t p = start;
  uint32_t run = (uint32_t)min(start_pos, (unsigned long long)cap);  // block p's run position
  bool in_run = start_pos != kNotFound, looked_up = in_run;
  while (p < n && alive) {
    if (!in_run) {
      const uint64_t key = __ldg(chain + p);
      unsigned long long pos = kNotFound;
      if (key != 0ull) pos = lookup_warp(ix.hash, key, log2_cap, lane, status);
      else if (lane == 0) flag_status(status, NETKV_DEV_EDOMAIN);
      if (pos == kNotFound) {  // absent from every cache of the group
        miss_all(h, lane, alive, p);
        return;
      }
      run = (uint32_t)min(pos, (unsigned long long)cap);
      looked_up = true;
    }
    // blocks p .. p + 32 U - 1 against the run: as long as whole steps match and no live
    // decode misses, a step costs its loads, the comparisons and one vote
    unsigned long long ck[U], rk[U];
    Mask rm[U];
    for (;;) {
      const bool whole = p + 32u * U <= n && run + 32u * U <= cap;
      const uint64_t* cp = chain + p + lane;
      const unsigned long long* kp = ix.keys + run + lane;
      if (whole) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          ck[u] = __ldcs(cp + 32 * u);
          rk[u] = __ldg(kp + 32 * u);
          rm[u] = (Mask)run_mask<kMB>(ix, run + lane + 32 * u);
        }
      } else {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          ck[u] = rk[u] = 0ull;
          rm[u] = 0;
          if (p + 32 * u + lane < n) {
            ck[u] = __ldcs(cp + 32 * u);
            if (run + 32 * u + lane < cap) {
              rk[u] = __ldg(kp + 32 * u);
              rm[u] = (Mask)run_mask<kMB>(ix, run + lane + 32 * u);
            }
          }
        }
      }
      bool same = true;
      Mask all = rm[0];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        same &= ck[u] == rk[u] && ck[u] != 0ull;
        all &= rm[u];
      }
      if (!whole || !__all_sync(0xffffffffu, same && !(alive & ~all))) break;
      p += 32u * U;
      run += 32u * U;
      looked_up = false;
    }
    uint32_t lead = 32u * U;  // leading blocks that match
#pragma unroll
    for (int u = U - 1; u >= 0; --u) {
      const uint32_t part = ~__ballot_sync(0xffffffffu, ck[u] != 0ull && rk[u] == ck[u]);
      if (part) lead = 32u * u + (uint32_t)(__ffs(part) - 1);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      rm[u] = 32u * u + lane < lead ? (Mask)(alive & ~rm[u]) : (Mask)0;
    settle<(kMB > 2)>(rm, p, h, alive, lane);
    if (lead == 0 && looked_up) {
      // the run entry the table points to does not hold the key: a corrupted index.
      // Report it and count the block as missing, so the walk always advances.
      if (lane == 0) flag_status(status, NETKV_DEV_EFULL);
      miss_all(h, lane, alive, p);
      return;
    }
    const bool out_of_order = looked_up && lead < 3;
    looked_up = false;
    p += lead;
    run += lead;
    in_run = lead == 32u * U;  // else the run parts here: look the next block up
    if (out_of_order) {
      const SideScan<kMB> s = scan_side_by_side<kMB>(ix.hash, ix.keys, ix.masks, chain, n,
                                                     log2_cap, SideScan<kMB>{h, alive, p, run},
                                                     status);
      h = s.h;
      alive = s.alive;
      p = s.p;
      run = s.run;
      in_run = true;
    }
  }
}

// Group key of a request: its table set and first block hash, never zero.
__device__ __forceinline__ uint64_t group_key(uint64_t h0, uint32_t set) {
  uint64_t z = h0 ^ ((uint64_t)(set + 1) * 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  return z ? z : 1ull;
}

struct GroupSlot {
  unsigned long long key;
  unsigned long long code;  // cached blocks << 48 | chain length << 32 | (0xffffffff - r)
};

// Work counters at the end of the workspace.
struct MatchCounters {
  unsigned long long n_long;       // leaders listed from the front of the leader list
  unsigned long long n_short;      // leaders listed from its back
  unsigned long long next_task;    // next (leader, decode group) task of the leader pass
};

// Leaders with at least this many cached blocks are listed first, so that the leader pass,
// which takes its tasks in list order, ends on short chains instead of waiting for a long
// one started last.
constexpr uint32_t kLongLeader = 2048;

// Blocks of one chain from p on that follow the run from position `run`, by one warp.
__device__ __forceinline__ uint32_t follow_run(const unsigned long long* __restrict__ run_keys,
                                               uint32_t cap, const uint64_t* __restrict__ chain,
                                               uint32_t p, uint32_t n, uint32_t run,
                                               uint32_t lane) {
  constexpr int U = 4;
  const uint32_t start = p;
  for (;;) {
    bool same[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t i = p + 32 * u + lane, rp = run + 32 * u + lane;
      const uint64_t ck = i < n ? __ldg(chain + i) : 0ull;
      const unsigned long long rk = i < n && rp < cap ? __ldg(run_keys + rp) : 1ull;
      same[u] = ck != 0ull && ck == rk && rp < cap;
    }
    if (!__all_sync(0xffffffffu, same[0] && same[1] && same[2] && same[3])) {
      uint32_t lead = 0;
#pragma unroll
      for (int u = U - 1; u >= 0; --u) {
        const uint32_t part = ~__ballot_sync(0xffffffffu, same[u]);
        if (part) lead = 32u * u + (uint32_t)(__ffs(part) - 1);
      }
      return p + lead - start;
    }
    p += 32 * U;
    run += 32 * U;
  }
}

// What a chain's walk through its set's first index found: the run position of its first
// block (kNoRun: not there), how many blocks follow the run from it, and how many runs were
// followed.  The later runs' positions and lengths lie in the request's row of M, 3 entries
// each, until the match writes the row (more than 64 entries, as pools of one decode group are
// matched directly).
struct FirstRun {
  uint32_t pos;
  uint16_t len, runs;
};

constexpr uint32_t kMaxRuns = 8;  // runs followed per chain: more only refine the grouping
static_assert(3 * (kMaxRuns - 1) <= kGroup, "the later runs fit the request's row");

// A warp takes `per` <= 32 consecutive requests, as match_kernel does.
__global__ void __launch_bounds__(kDirectBlock, 16) group_scan_kernel(
    const void* __restrict__ index, uint32_t n_dgroups, uint32_t log2_cap, uint32_t n_sets,
    const uint64_t* __restrict__ chains, const uint64_t* __restrict__ chain_off, uint32_t R,
    const uint32_t* __restrict__ set_off, uint32_t per, GroupSlot* __restrict__ tab,
    uint32_t log2_slots, int32_t* __restrict__ set_of, uint64_t* __restrict__ gkey,
    FirstRun* __restrict__ first_run, uint16_t* __restrict__ M, uint32_t D) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t cap = 1u << log2_cap;
  const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  for (uint64_t t0 = warp * per; t0 < R; t0 += n_warps * per) {
    const uint32_t count = (uint32_t)min((uint64_t)per, R - t0);
    const uint32_t my_r = (uint32_t)t0 + lane;
    uint64_t my_c0 = 0, my_key = 0;
    uint32_t my_n = 0, my_pos = kNoRun, my_len = 0, my_cached = 0, my_runs = 0;
    int32_t my_set = -1;
    if (lane < count) {
      my_c0 = __ldg(chain_off + my_r);
      const uint64_t c1 = __ldg(chain_off + my_r + 1);
      my_set = find_set(set_off, n_sets, my_r);
      set_of[my_r] = my_set;
      if (my_set >= 0 && c1 > my_c0) {
        my_n = (uint32_t)min(c1 - my_c0, (uint64_t)65535);
        const uint64_t h0 = __ldg(chains + my_c0);
        my_key = group_key(h0, (uint32_t)my_set);
        unsigned long long pos = kNotFound;
        if (h0 != 0ull)
          pos = lookup(index_view(index, (uint64_t)my_set * n_dgroups, log2_cap, 8u).hash, h0,
                       log2_cap, nullptr);  // the match itself reports what it meets
        if (pos < cap) my_pos = (uint32_t)pos;
      }
    }
    for (uint32_t i = 0; i < count; ++i) {
      const uint32_t pos = __shfl_sync(0xffffffffu, my_pos, i);
      if (pos == kNoRun) continue;
      const uint32_t n = __shfl_sync(0xffffffffu, my_n, i);
      const uint64_t* chain = chains + __shfl_sync(0xffffffffu, my_c0, i);
      const IndexView ix = index_view(
          index, (uint64_t)__shfl_sync(0xffffffffu, my_set, i) * n_dgroups, log2_cap, 8u);
      const uint32_t len = follow_run(ix.keys, cap, chain, 0, n, pos, lane);
      uint16_t* path = M + (uint64_t)(t0 + i) * D;
      uint32_t p = len, runs = 1;
      for (; runs < kMaxRuns && p < n; ++runs) {
        const uint64_t key = __ldg(chain + p);
        if (key == 0ull) break;
        const unsigned long long at = lookup_warp(ix.hash, key, log2_cap, lane, nullptr);
        if (at >= cap) break;
        const uint32_t more = follow_run(ix.keys, cap, chain, p, n, (uint32_t)at, lane);
        if (more == 0) break;
        if (lane < 3)
          path[3 * (runs - 1) + lane] = (uint16_t)(lane == 0 ? at : lane == 1 ? at >> 16 : more);
        p += more;
      }
      if (lane == i) {
        my_len = len;
        my_cached = p;
        my_runs = runs;
      }
    }
    if (lane < count) {
      gkey[my_r] = my_key;  // 0: not grouped
      first_run[my_r] = FirstRun{my_pos, (uint16_t)my_len, (uint16_t)my_runs};
      if (my_key != 0ull) {
        const uint64_t mask = (1ull << log2_slots) - 1;
        const unsigned long long code = ((unsigned long long)my_cached << 48) |
                                        ((unsigned long long)my_n << 32) | (0xffffffffu - my_r);
        uint64_t slot = home_slot(my_key, log2_slots);
        for (uint64_t step = 0; step <= mask; ++step) {
          const unsigned long long prev = atomicCAS(&tab[slot].key, 0ull, my_key);
          if (prev == 0ull || prev == my_key) {
            atomicMax(&tab[slot].code, code);
            break;
          }
          slot = (slot + 1) & mask;
        }
      }
    }
  }
}

// A member's common prefix with its leader, in the place of its group key: the length, and
// whether it is exact (else the chains agree at least so far and are compared from there).
constexpr uint64_t kLcpExact = 1ull << 32;

__global__ void group_resolve_kernel(const GroupSlot* __restrict__ tab, uint32_t log2_slots,
                                     uint32_t R, uint32_t* __restrict__ leader_of,
                                     const int32_t* __restrict__ set_of,
                                     uint32_t* __restrict__ leaders, uint64_t* __restrict__ gkey,
                                     const FirstRun* __restrict__ first_run,
                                     const uint16_t* __restrict__ M, uint32_t D,
                                     MatchCounters* counters) {
  const uint64_t mask = (1ull << log2_slots) - 1;
  for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < R; r += gridDim.x * blockDim.x) {
    const uint64_t key = gkey[r];  // written by the scan pass
    uint32_t lead = r, cached = 0;
    if (key != 0ull) {
      uint64_t slot = home_slot(key, log2_slots);
      for (uint64_t step = 0; step <= mask; ++step) {
        const unsigned long long k = tab[slot].key;
        if (k == key) {
          const unsigned long long code = tab[slot].code;
          const uint32_t L = 0xffffffffu - (uint32_t)(code & 0xffffffffull);
          // a leader from another table set (64-bit key collision) is never used
          if (L < R && __ldg(set_of + L) == __ldg(set_of + r)) lead = L;
          cached = (uint32_t)(code >> 48);
          break;
        }
        if (k == 0ull) break;
        slot = (slot + 1) & mask;
      }
    }
    leader_of[r] = lead;
    if (lead == r) {  // long chains from the front of the list, the rest from its back
      if (cached >= kLongLeader) leaders[atomicAdd(&counters->n_long, 1ull)] = r;
      else leaders[R - 1 - atomicAdd(&counters->n_short, 1ull)] = r;
    } else {
      // Chains that agree follow the same runs.  So the chain that left their common run
      // first parts from the other there, and so do chains whose next runs differ, or of
      // which only one goes on: a block's run depends on its hash alone.
      const FirstRun a = first_run[r], b = first_run[lead];
      uint64_t lcp = 0;
      if (a.pos == b.pos && a.pos != kNoRun) {
        uint32_t x = a.len, y = b.len;
        lcp = min(x, y);
        bool parted = x != y;
        for (uint32_t i = 1; !parted; ++i) {
          if (i == a.runs && i == b.runs) break;  // they agree so far
          parted = i == a.runs || i == b.runs;
          if (parted) break;
          const uint16_t* pa = M + (uint64_t)r * D + 3 * (i - 1);
          const uint16_t* pb = M + (uint64_t)lead * D + 3 * (i - 1);
          parted = pa[0] != pb[0] || pa[1] != pb[1];
          if (parted) break;
          x = pa[2];
          y = pb[2];
          lcp += min(x, y);
          parted = x != y;
        }
        if (parted) lcp |= kLcpExact;
      }
      gkey[r] = lcp;
    }
  }
}

// Chain r's extent clamped to 65535 blocks; false on a bad request (flagged).
__device__ __forceinline__ bool chain_extent(const uint64_t* __restrict__ chain_off,
                                             const uint32_t* __restrict__ set_off,
                                             uint32_t n_sets, const int32_t* __restrict__ set_of,
                                             uint32_t r, uint32_t lane, int* status,
                                             int32_t& set, uint64_t& c0, uint64_t& n) {
  set = set_of ? __ldg(set_of + r) : find_set(set_off, n_sets, r);
  c0 = __ldg(chain_off + r);
  const uint64_t c1 = __ldg(chain_off + r + 1);
  if (set < 0 || c1 < c0) {
    if (lane == 0) flag_status(status, NETKV_DEV_ERANGE);
    return false;
  }
  n = c1 - c0;
  if (n > 65535) {
    if (lane == 0) flag_status(status, NETKV_DEV_EDOMAIN);
    n = 65535;
  }
  return true;
}

__device__ __forceinline__ void store_hits(uint16_t* __restrict__ M, uint64_t row, uint32_t q0,
                                           uint32_t ng, uint32_t lane, const GroupHits& h) {
  if (lane < ng) M[row + q0 + lane] = (uint16_t)h.lo;
  if (lane + 32 < ng) M[row + q0 + lane + 32] = (uint16_t)h.hi;
}

// Leader pass: one task per (leader, decode group), taken in order from a global counter
// by whole warps, so long and short chains balance across the GPU.  Bound by the dependent
// steps of the longest chains, so steps are 256 blocks: 8 leaders x 16 groups of up to 7,680
// blocks 57 us (69 at 128 a step), 50 leaders x 64 groups 97 us.  A block of 8 warps per long
// leader, 1,024 blocks a step: 58 and 209 us.
__global__ void __launch_bounds__(kMatchBlock, 2) match_leaders_kernel(
    const void* __restrict__ index, uint32_t D, uint32_t log2_cap, uint32_t n_sets,
    const uint64_t* __restrict__ chains, const uint64_t* __restrict__ chain_off, uint32_t R,
    const uint32_t* __restrict__ set_off, const int32_t* __restrict__ set_of,
    const uint32_t* __restrict__ leaders, MatchCounters* counters, uint16_t* __restrict__ M,
    int* status) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t n_dgroups = (D + kGroup - 1) / kGroup;
  const unsigned long long n_long = *((volatile unsigned long long*)&counters->n_long);
  const unsigned long long total =
      (n_long + *((volatile unsigned long long*)&counters->n_short)) * n_dgroups;
  for (;;) {
    unsigned long long t = 0;
    if (lane == 0) t = atomicAdd(&counters->next_task, 1ull);
    t = __shfl_sync(0xffffffffu, t, 0);
    if (t >= total) break;
    const uint64_t li = t / n_dgroups;
    const uint32_t r = __ldg(leaders + (li < n_long ? li : (uint64_t)R - 1 - (li - n_long)));
    const uint32_t q = (uint32_t)(t - li * n_dgroups);
    const uint32_t q0 = q * kGroup, ng = min(kGroup, D - q0);
    GroupHits h = {0u, 0u};
    int32_t set;
    uint64_t c0, n;
    if (chain_extent(chain_off, set_off, n_sets, set_of, r, lane, status, set, c0, n)) {
      h.lo = h.hi = (uint32_t)n;
      const unsigned long long alive = ng >= 64 ? ~0ull : ((1ull << ng) - 1);
      const IndexView ix = index_view(index, (uint64_t)set * n_dgroups + q, log2_cap, 8u);
      scan_chain<8, 8>(ix, log2_cap, chains + c0, 0, n, alive, h, lane, status);
    }
    store_hits(M, (uint64_t)r * D, q0, ng, lane, h);
  }
}

// Full match, one task per (request, decode group): pools of one group, and any pool without
// a workspace.  A warp takes `per` <= 32 consecutive tasks: first lane i reads task i's
// chain extent and first block and looks the block up, all tasks side by side; then the
// warp scans one chain after another, whose first step needs no further address.
// Blocks are small so that a long chain holds back few other warps, and steps of 128
// blocks keep enough loads in flight at 32 warps an SM (64 registers).  Bound by latency and
// issue: 1,024 replicas (8 decodes, 1.02 M requests) 1.05 ms, 4.8 KB of DRAM traffic a
// request (4.7 TB/s).  Matching the members of a group against their leader's chain, after
// a grouping and a leader pass, took 1.38 ms there, 130 us against 14 for 1,000 requests,
// 37 against 4 for one, and 1.20 ms against 0.60 for 32,000 requests whose chains lie in
// host memory, where the leader's chain crosses the link for every member.  Steps of 64 and
// 96 blocks: 1.39 and 1.18 ms (in host memory 0.59 and 0.58); 32 blocks first: 1.26 ms; 24
// blocks an SM (40 registers): spills, no faster.  Many requests on shallow caches of 33 .. 64
// decodes still favour the grouping: 64,000 requests whose hits end within 1,024 blocks 202 us
// against 125, within 16 101 against 93.
template <int kMB>
__global__ void __launch_bounds__(kDirectBlock, 16) match_kernel(
    const void* __restrict__ index, uint32_t D, uint32_t log2_cap, uint32_t n_sets,
    const uint64_t* __restrict__ chains, const uint64_t* __restrict__ chain_off, uint32_t R,
    const uint32_t* __restrict__ set_off, uint32_t per, uint16_t* __restrict__ M, int* status) {
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint32_t n_dgroups = (D + kGroup - 1) / kGroup;
  const uint64_t total = (uint64_t)R * n_dgroups;
  for (uint64_t t0 = warp * per; t0 < total; t0 += n_warps * per) {
    const uint32_t count = (uint32_t)min((uint64_t)per, total - t0);
    uint64_t my_c0 = 0;  // lane i: task t0 + i
    uint32_t my_n = 0, my_pos = 0;
    int32_t my_set = -1;  // < 0: a bad request, hits 0
    if (lane < count) {
      const uint64_t task = t0 + lane;
      const uint32_t r = (uint32_t)(n_dgroups == 1 ? task : task / n_dgroups);
      const uint32_t q = (uint32_t)(task - (uint64_t)r * n_dgroups);
      my_c0 = __ldg(chain_off + r);
      const uint64_t c1 = __ldg(chain_off + r + 1);
      my_set = find_set(set_off, n_sets, r);
      if (my_set < 0 || c1 < my_c0) {
        flag_status(status, NETKV_DEV_ERANGE);
        my_set = -1;
      } else if (c1 > my_c0) {
        if (c1 - my_c0 > 65535) flag_status(status, NETKV_DEV_EDOMAIN);
        my_n = (uint32_t)min(c1 - my_c0, (uint64_t)65535);
        const uint64_t key = __ldg(chains + my_c0);
        unsigned long long pos = kNotFound;
        if (key != 0ull)
          pos = lookup(index_view(index, (uint64_t)my_set * n_dgroups + q, log2_cap, kMB).hash,
                       key, log2_cap, status);
        else
          flag_status(status, NETKV_DEV_EDOMAIN);
        my_pos = pos == kNotFound ? kNoRun : (uint32_t)min(pos, 1ull << log2_cap);
      }
    }
    for (uint32_t i = 0; i < count; ++i) {
      const uint64_t task = t0 + i;
      const uint32_t r = (uint32_t)(n_dgroups == 1 ? task : task / n_dgroups);
      const uint32_t q = (uint32_t)(task - (uint64_t)r * n_dgroups);
      const uint32_t q0 = q * kGroup, ng = min(kGroup, D - q0);
      const int32_t set = __shfl_sync(0xffffffffu, my_set, i);
      const uint32_t n = __shfl_sync(0xffffffffu, my_n, i);
      const uint32_t pos = __shfl_sync(0xffffffffu, my_pos, i);
      const uint64_t c0 = __shfl_sync(0xffffffffu, my_c0, i);
      GroupHits h = {0u, 0u};
      if (set >= 0 && pos != kNoRun) {  // else every decode misses block 0
        h.lo = h.hi = n;
        const unsigned long long alive = ng >= 64 ? ~0ull : ((1ull << ng) - 1);
        scan_chain<4, kMB>(index_view(index, (uint64_t)set * n_dgroups + q, log2_cap, kMB),
                           log2_cap, chains + c0, 0, n, alive, h, lane, status, pos);
      }
      store_hits(M, (uint64_t)r * D, q0, ng, lane, h);
    }
  }
}

// One group of a member walked on from block lcp, at run position `pos`: the decodes whose
// leader's hit (ml) reaches lcp go on, the others keep it.  (32 blocks a step instead of 128:
// 32,000 requests of 1,024 blocks on deep caches of 4,096 decodes 435 us, now 322.)
__device__ __forceinline__ void scan_member(IndexView ix, uint32_t log2_cap,
                                         const uint64_t* __restrict__ chain, uint32_t lcp,
                                         uint32_t n, unsigned long long pos,
                                         const uint16_t* __restrict__ ml,
                                         uint16_t* __restrict__ mr, uint32_t ng, int* status) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t mlo = lane < ng ? (uint32_t)__ldg(ml + lane) : 0u;
  const uint32_t mhi = lane + 32 < ng ? (uint32_t)__ldg(ml + lane + 32) : 0u;
  GroupHits h;
  h.lo = mlo < lcp ? mlo : n;
  h.hi = mhi < lcp ? mhi : n;
  const uint32_t alo = __ballot_sync(0xffffffffu, lane < ng && mlo >= lcp);
  const uint32_t ahi = __ballot_sync(0xffffffffu, lane + 32 < ng && mhi >= lcp);
  const unsigned long long alive = (unsigned long long)alo | ((unsigned long long)ahi << 32);
  scan_chain<4, 8>(ix, log2_cap, chain, lcp, n, alive, h, lane, status, pos);
  store_hits(mr, 0, 0, ng, lane, h);
}

// Member pass: one warp per member.  With lcp = |common prefix of h_r and h_L|, every decode
// has M_r[d] = min(M_L[d], lcp) unless M_L[d] >= lcp and block lcp of h_r is cached on d.  So
// the member's row is one elementwise pass over the leader's row (16 bytes a lane when the
// rows are 16-byte aligned), and block lcp is then probed in the groups where some leader
// hit reaches lcp, up to 32 groups at once with one lane per group; a group whose probe
// finds the block is walked again by the whole warp.
// Bound by the rows it writes: 32,000 requests on 4,096 decodes 100 us, 8,192 on 1,024 11 us
// (147 and 14 with one row chunk a lane in flight and groups noted one by one).  With only the
// first run's length known, whose end most members share with their leader, both chains were
// read on from there: 164 and 47 us, and 778 against 36 with the chains in host memory.  With
// leaders chosen by chain length, the members whose cached prefix ran past their leader's walked
// all 64 groups of the pool again: 3.9 ms (6.6 ms at 32 blocks a step).
__global__ void __launch_bounds__(kMatchBlock, 4) match_members_wide_kernel(
    const void* __restrict__ index, uint32_t D, uint32_t log2_cap, uint32_t n_sets,
    const uint64_t* __restrict__ chains, const uint64_t* __restrict__ chain_off, uint32_t R,
    const uint32_t* __restrict__ set_off, const uint32_t* __restrict__ leader_of,
    const int32_t* __restrict__ set_of, const uint64_t* __restrict__ known_lcp,
    uint16_t* __restrict__ M, int* status) {
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint32_t n_dgroups = (D + kGroup - 1) / kGroup;
  const bool vec = (D % 8u == 0) && ((reinterpret_cast<uintptr_t>(M) & 15u) == 0);
  const uint32_t n8 = D / 8u;  // 16-byte chunks of a row (vector form)

  for (uint64_t rr = warp; rr < R; rr += n_warps) {
    const uint32_t r = (uint32_t)rr;
    const uint32_t lead = __ldg(leader_of + r);
    if (lead == r) continue;  // leaders were matched by the leader pass
    const uint64_t known = __ldg(known_lcp + r);
    const uint64_t row = (uint64_t)r * D;
    int32_t set;
    uint64_t c0, n;
    if (!chain_extent(chain_off, set_off, n_sets, set_of, r, lane, status, set, c0, n)) {
      const GroupHits z = {0u, 0u};
      for (uint32_t q = 0; q < n_dgroups; ++q)
        store_hits(M, row, q * kGroup, min(kGroup, D - q * kGroup), lane, z);
      continue;
    }
    const uint64_t* __restrict__ own = chains + c0;
    const uint16_t* __restrict__ ml = M + (uint64_t)lead * D;
    uint16_t* __restrict__ mr = M + row;

    uint64_t lcp = known & (kLcpExact - 1);
    if (!(known & kLcpExact)) {  // compare the chains from there, 128 blocks a step
      const uint64_t l0 = __ldg(chain_off + lead);
      const uint64_t nl = min(__ldg(chain_off + lead + 1) - l0, (uint64_t)65535);
      const uint64_t* __restrict__ lch = chains + l0;
      // the leader's largest hit: blocks past it decide nothing
      uint32_t mmax = 0;
      if (vec) {
        for (uint32_t c = lane; c < n8; c += 32) {
          const uint4 v = __ldg(reinterpret_cast<const uint4*>(ml) + c);
          const uint32_t m2 = __vmaxu2(__vmaxu2(v.x, v.y), __vmaxu2(v.z, v.w));
          mmax = max(mmax, max(m2 & 0xffffu, m2 >> 16));
        }
      } else {
        for (uint32_t d = lane; d < D; d += 32) mmax = max(mmax, (uint32_t)__ldg(ml + d));
      }
      mmax = __reduce_max_sync(0xffffffffu, mmax);
      const uint64_t cap = min(n, min(nl, (uint64_t)mmax + 1));
      const uint64_t from = min(lcp, cap);
      lcp = cap;
      for (uint64_t base = from; base < cap; base += 128) {
        uint64_t a[4], b[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint64_t i = base + 32 * k + lane;
          a[k] = i < cap ? __ldg(own + i) : 0ull;
          b[k] = i < cap ? __ldg(lch + i) : 0ull;
        }
        uint64_t found = cap;
#pragma unroll
        for (int k = 3; k >= 0; --k) {
          const uint32_t diff = __ballot_sync(0xffffffffu, a[k] != b[k]);
          if (diff) found = base + 32 * k + (uint64_t)(__ffs(diff) - 1);
        }
        if (found < cap) {
          lcp = found;
          break;
        }
      }
    }
    // M_r = min(M_L, lcp), 32 groups at a time; where a leader hit reaches lcp (bit j of `reached`:
    // group g0 + j), block lcp is then looked up, a group a lane
    const uint32_t lcp_u = (uint32_t)lcp, lcp2 = lcp_u | (lcp_u << 16);
    for (uint32_t g0 = 0; g0 < n_dgroups; g0 += 32) {
      uint32_t reached = 0;
      if (vec) {
#pragma unroll
        for (uint32_t k0 = 0; k0 < 8; k0 += 4) {  // 256 decodes = 4 groups each
          if (g0 + 4 * k0 >= n_dgroups) break;
          uint4 x[4];
#pragma unroll
          for (uint32_t k = 0; k < 4; ++k) {
            const uint32_t c = 8 * g0 + 32 * (k0 + k) + lane;
            x[k] = make_uint4(0u, 0u, 0u, 0u);
            if (c < n8) x[k] = __ldg(reinterpret_cast<const uint4*>(ml) + c);
          }
#pragma unroll
          for (uint32_t k = 0; k < 4; ++k) {
            const uint32_t c = 8 * g0 + 32 * (k0 + k) + lane;
            const uint32_t m2 = __vmaxu2(__vmaxu2(x[k].x, x[k].y), __vmaxu2(x[k].z, x[k].w));
            const bool reach = c < n8 && max(m2 & 0xffffu, m2 >> 16) >= lcp_u;
            if (c < n8)
              reinterpret_cast<uint4*>(mr)[c] =
                  make_uint4(__vminu2(x[k].x, lcp2), __vminu2(x[k].y, lcp2),
                             __vminu2(x[k].z, lcp2), __vminu2(x[k].w, lcp2));
            // lanes 8 q .. 8 q + 7 hold the q-th of the four groups
            const uint32_t fb = __ballot_sync(0xffffffffu, reach);
#pragma unroll
            for (uint32_t q = 0; q < 4; ++q)
              reached |= ((fb >> (8 * q)) & 0xffu) ? 1u << (4 * (k0 + k) + q) : 0u;
          }
        }
      } else {
        for (uint32_t q = g0; q < min(n_dgroups, g0 + 32); ++q) {
          const uint32_t q0 = q * kGroup, ng = min(kGroup, D - q0);
          const uint32_t mlo = lane < ng ? (uint32_t)__ldg(ml + q0 + lane) : 0u;
          const uint32_t mhi = lane + 32 < ng ? (uint32_t)__ldg(ml + q0 + lane + 32) : 0u;
          GroupHits h;
          h.lo = min(mlo, lcp_u);
          h.hi = min(mhi, lcp_u);
          store_hits(M, row, q0, ng, lane, h);
          const bool reach = (lane < ng && mlo >= lcp_u) || (lane + 32 < ng && mhi >= lcp_u);
          if (__any_sync(0xffffffffu, reach)) reached |= 1u << (q - g0);
        }
      }
      if (lcp >= n || !reached) continue;  // decodes with M_L >= lcp may hit block lcp
      unsigned long long pos = kNotFound;
      if ((reached >> lane) & 1u) {
        const uint64_t key = __ldg(own + lcp);
        if (key == 0ull) flag_status(status, NETKV_DEV_EDOMAIN);
        else pos = lookup(index_view(index, (uint64_t)set * n_dgroups + g0 + lane, log2_cap, 8u).hash,
                          key, log2_cap, status);
      }
      uint32_t hit = __ballot_sync(0xffffffffu, pos != kNotFound);
      while (hit) {
        const uint32_t j = __ffs(hit) - 1, q = g0 + j;
        hit &= hit - 1;
        const unsigned long long pj = __shfl_sync(0xffffffffu, pos, j);
        __syncwarp();  // the row's minima are written
        scan_member(index_view(index, (uint64_t)set * n_dgroups + q, log2_cap, 8u), log2_cap, own,
                    lcp_u, (uint32_t)n, pj, ml + q * kGroup, mr + q * kGroup,
                    min(kGroup, D - q * kGroup), status);
      }
    }
  }
}

uint32_t group_log2_slots(uint32_t R) {
  uint32_t l = 1;
  while ((1ull << l) < 2ull * R) ++l;
  return l;
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Workspace: group table | leader_of [R] | set_of [R] | leader list [R] | group keys, then
// known common prefixes [R] | first runs [R] | counters.  Used for pools of several decode groups.
struct WorkspaceLayout {
  size_t table, leader_of, set_of, leaders, gkey, first_run, counters, total;
};

WorkspaceLayout workspace_layout(uint32_t R) {
  WorkspaceLayout w;
  w.table = 0;
  w.leader_of = align_up(sizeof(GroupSlot) << group_log2_slots(R), 256);
  w.set_of = w.leader_of + align_up(sizeof(uint32_t) * (size_t)R, 256);
  w.leaders = w.set_of + align_up(sizeof(int32_t) * (size_t)R, 256);
  w.gkey = w.leaders + align_up(sizeof(uint32_t) * (size_t)R, 256);
  w.first_run = w.gkey + align_up(sizeof(uint64_t) * (size_t)R, 256);
  w.counters = w.first_run + align_up(sizeof(FirstRun) * (size_t)R, 256);
  w.total = w.counters + align_up(sizeof(MatchCounters), 256);
  return w;
}

// Blocks of a persistent grid: every SM filled to the kernel's occupancy.
template <typename Kernel>
int persistent_grid(Kernel kernel, int block) {
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, 0);
  return (sms > 0 ? sms : 1) * (per_sm > 0 ? per_sm : 1);
}
int leader_grid() { return persistent_grid(match_leaders_kernel, kMatchBlock); }

// The direct match.  A warp takes several tasks where every resident warp still gets
// kWaves turns (the card's last turns are then short), at most kPerWarp.
constexpr uint32_t kPerWarp = 8, kWaves = 8;
uint32_t tasks_per_warp(uint64_t tasks, int sms) {
  const uint64_t turns = tasks / ((uint64_t)sms * 32 * kWaves);
  return turns < 1 ? 1u : turns < kPerWarp ? (uint32_t)turns : kPerWarp;
}
netkv_status launch_match(const void* index, uint32_t D, uint32_t log2_cap, uint32_t n_sets,
                          const uint64_t* chains, const uint64_t* chain_off, uint32_t R,
                          const uint32_t* set_off, uint16_t* M, int* status, int sms,
                          cudaStream_t s) {
  const uint64_t tasks = (uint64_t)R * ((D + kGroup - 1) / kGroup);
  const uint32_t per = tasks_per_warp(tasks, sms);
  const uint64_t per_block = (uint64_t)per * (kDirectBlock / 32);
  const uint64_t blocks = (tasks + per_block - 1) / per_block;
  const unsigned grid = (unsigned)(blocks < (1u << 24) ? blocks : (1u << 24));
#define NETKV_MATCH(MB)                                                                      \
  match_kernel<MB><<<grid, kDirectBlock, 0, s>>>(index, D, log2_cap, n_sets, chains,         \
                                                 chain_off, R, set_off, per, M, status)
  switch (mask_bytes_of(D)) {
    case 1: NETKV_MATCH(1); break;
    case 2: NETKV_MATCH(2); break;
    case 4: NETKV_MATCH(4); break;
    default: NETKV_MATCH(8); break;
  }
#undef NETKV_MATCH
  return netkv_launch_status();
}

// Whether a call's indices are built by one block each.  Few of them: one list after another
// takes 3 us a list or more, the passes about 45 us for their launches (us, one block / passes;
// 1 index of 8 lists of 16 keys 34 / 46, of 500 35 / 53, of 2,000 92 / 61; 16 lists of 16 41 /
// 53, of 500 74 / 58).  Many: the blocks fill the card, and the passes go over the slots four
// times (256 indices of 8 lists: 1,000 keys each 68 / 114, 2,000 137 / 184, 10,000 968 / 672;
// of 16 lists: 1,000 121 / 155, 2,000 237 / 244, 10,000 1,916 / 911).  Larger lists that share
// nothing favour one block too (300 indices of 8 lists of 50,000: 7,925 / 9,981), but the host
// cannot tell them from lists with shared prefixes.
bool serial_build(uint64_t n_index, uint32_t D, uint32_t log2_cap, uint32_t sms) {
  const uint32_t lists = D < kGroup ? D : kGroup;
  if ((lists <= 12 && log2_cap <= 13) || (lists <= 16 && log2_cap <= 11)) return true;
  return 2 * n_index >= sms && (lists <= 12 ? log2_cap <= 14 : lists <= 32 && log2_cap <= 13);
}

}  // namespace

extern "C" size_t netkv_cache_index_bytes(uint32_t n_sets, uint32_t D, uint32_t log2_capacity) {
  if (log2_capacity < 1 || log2_capacity > 31) return 0;
  return (size_t)n_sets * ((D + kGroup - 1) / kGroup) *
         index_stride(log2_capacity, mask_bytes_of(D));
}

extern "C" netkv_status netkv_cache_build(void* d_index, uint32_t n_sets, uint32_t D,
                                          uint32_t log2_capacity, const uint64_t* d_keys,
                                          const uint64_t* d_key_off, int* d_status,
                                          netkv_stream_t stream) {
  if (!d_index || !d_key_off || D == 0 || log2_capacity < 1 || log2_capacity > 31)
    return NETKV_EINVAL;
  if (!aligned_to(d_index, 16) || !aligned_to(d_key_off, 8) || (d_keys && !aligned_to(d_keys, 8)))
    return NETKV_EINVAL;
  if (n_sets == 0) return NETKV_OK;
  cudaStream_t s = (cudaStream_t)stream;
  NETKV_CUDA_TRY(cudaMemsetAsync(d_index, 0, netkv_cache_index_bytes(n_sets, D, log2_capacity), s));
  if (!d_keys) return NETKV_OK;
  BuildArgs a;
  a.index = d_index;
  a.n_index = (uint64_t)n_sets * ((D + kGroup - 1) / kGroup);
  a.D = D;
  a.log2_cap = log2_capacity;
  a.keys = d_keys;
  a.key_off = d_key_off;
  a.status = d_status;
  int dev = 0, sms = 0;
  NETKV_CUDA_TRY(cudaGetDevice(&dev));
  NETKV_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const unsigned per_index = (unsigned)(a.n_index < (1u << 20) ? a.n_index : (1u << 20));
  if (serial_build(a.n_index, D, log2_capacity, (uint32_t)sms)) {
    build_serial_kernel<true><<<per_index, kBuildBlock, 0, s>>>(a);
    return netkv_launch_status();
  }
  // blocks per index: one per 2,048 slots, more where the indices alone leave SMs idle
  uint64_t parts = (1ull << log2_capacity) / 2048;
  const uint64_t fill = ((uint64_t)sms * 8 + a.n_index - 1) / a.n_index;
  if (parts > kPartsMax) parts = kPartsMax;
  if (parts < fill) parts = fill;
  a.parts = (uint32_t)parts;
  const uint64_t blocks = a.n_index * a.parts;
  const unsigned grid = (unsigned)(blocks < (1u << 30) ? blocks : (1u << 30));
  build_insert_kernel<<<grid, kPassBlock, 0, s>>>(a);
  build_mark_kernel<<<grid, kPassBlock, 0, s>>>(a);
  build_count_kernel<<<per_index, kBuildBlock, 0, s>>>(a);
  build_place_kernel<<<grid, kPassBlock, 0, s>>>(a);
  build_wipe_kernel<<<grid, kPassBlock, 0, s>>>(a);
  build_masks_kernel<<<grid, kPassBlock, 0, s>>>(a);
  build_serial_kernel<false><<<per_index, kBuildBlock, 0, s>>>(a);
  return netkv_launch_status();
}

extern "C" size_t netkv_prefix_match_workspace_size(uint32_t R) {
  if (R == 0) return 0;
  return workspace_layout(R).total;
}

extern "C" netkv_status netkv_prefix_match(const void* d_index, uint32_t D,
                                           uint32_t log2_capacity, uint32_t n_sets,
                                           const uint64_t* d_chains, const uint64_t* d_chain_off,
                                           uint32_t R, const uint32_t* d_set_off,
                                           void* d_workspace, size_t workspace_bytes,
                                           uint16_t* d_M, int* d_status, netkv_stream_t stream) {
  if (!d_index || !d_chain_off || !d_M || D == 0 || n_sets == 0) return NETKV_EINVAL;
  if (log2_capacity < 1 || log2_capacity > 31) return NETKV_EINVAL;
  if (n_sets > 1 && !d_set_off) return NETKV_EINVAL;
  if (!aligned_to(d_index, 16) || !aligned_to(d_chain_off, 8) || !aligned_to(d_M, 2) ||
      (d_chains && !aligned_to(d_chains, 8)) || (d_set_off && !aligned_to(d_set_off, 4)) ||
      (d_workspace && !aligned_to(d_workspace, 256)))
    return NETKV_EINVAL;
  if (R == 0) return NETKV_OK;
  if (!d_chains || R > 0x7fffffffu) return NETKV_EINVAL;
  if (d_workspace && workspace_bytes < netkv_prefix_match_workspace_size(R)) return NETKV_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  const void* index = d_index;
  int dev = 0, sms = 0;
  NETKV_CUDA_TRY(cudaGetDevice(&dev));
  NETKV_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const uint64_t tasks = (uint64_t)R * ((D + kGroup - 1) / kGroup);
  // a few requests: every (request, group) has a warp at once, and sharing, six launches
  // long, cannot end before the longest of them (34 requests on 1,218 decodes: 20 us, not 55)
  if (!d_workspace || D <= kGroup || tasks <= (uint64_t)sms * 32)
    return launch_match(index, D, log2_capacity, n_sets, d_chains, d_chain_off, R, d_set_off, d_M,
                        d_status, sms, s);
  const uint32_t lg = group_log2_slots(R);
  const WorkspaceLayout L = workspace_layout(R);
  char* ws = reinterpret_cast<char*>(d_workspace);
  GroupSlot* tab = reinterpret_cast<GroupSlot*>(ws + L.table);
  uint32_t* leader_of = reinterpret_cast<uint32_t*>(ws + L.leader_of);
  int32_t* set_of = reinterpret_cast<int32_t*>(ws + L.set_of);
  uint32_t* leaders = reinterpret_cast<uint32_t*>(ws + L.leaders);
  uint64_t* gkey = reinterpret_cast<uint64_t*>(ws + L.gkey);
  MatchCounters* counters = reinterpret_cast<MatchCounters*>(ws + L.counters);
  NETKV_CUDA_TRY(cudaMemsetAsync(tab, 0, sizeof(GroupSlot) << lg, s));
  NETKV_CUDA_TRY(cudaMemsetAsync(counters, 0, sizeof(MatchCounters), s));
  const unsigned rgrid = (unsigned)((R + 255) / 256 < 65535u * 16 ? (R + 255) / 256 : 65535u * 16);
  FirstRun* first_run = reinterpret_cast<FirstRun*>(ws + L.first_run);
  const uint32_t per = tasks_per_warp(R, sms);
  const uint64_t sblocks = ((uint64_t)R + per * (kDirectBlock / 32) - 1) / (per * (kDirectBlock / 32));
  const unsigned sgrid = (unsigned)(sblocks < (1u << 24) ? sblocks : (1u << 24));
  group_scan_kernel<<<sgrid, kDirectBlock, 0, s>>>(
      index, (D + kGroup - 1) / kGroup, log2_capacity, n_sets, d_chains, d_chain_off, R, d_set_off,
      per, tab, lg, set_of, gkey, first_run, d_M, D);
  group_resolve_kernel<<<rgrid, 256, 0, s>>>(tab, lg, R, leader_of, set_of, leaders, gkey,
                                             first_run, d_M, D, counters);
  match_leaders_kernel<<<leader_grid(), kMatchBlock, 0, s>>>(
      index, D, log2_capacity, n_sets, d_chains, d_chain_off, R, d_set_off, set_of, leaders,
      counters, d_M, d_status);
  const uint64_t warps_per_block = kMatchBlock / 32;
  const uint64_t mblocks = ((uint64_t)R + warps_per_block - 1) / warps_per_block;
  const unsigned mgrid = (unsigned)(mblocks < (1u << 24) ? mblocks : (1u << 24));
  match_members_wide_kernel<<<mgrid, kMatchBlock, 0, s>>>(index, D, log2_capacity, n_sets,
                                                          d_chains, d_chain_off, R, d_set_off,
                                                          leader_of, set_of, gkey, d_M,
                                                          d_status);
  return netkv_launch_status();
}

// ---------------------------------------------------------------------------------
// netkv_prefix_match_static: the prefix match for callers that cannot allocate device
// memory (see include/netkv.h).  Its workspace is this fixed device array, shared by
// every call on a device.  Host code cannot use the array's name as a device address, so
// the address is looked up with the device current: on every call made outside a stream
// capture (a device reset reloads the module and may move the array), and from the
// last lookup on that device during a capture.
// ---------------------------------------------------------------------------------
#include <mutex>

namespace {

constexpr size_t kStaticScratchBytes = 32ull << 20;  // 32 MiB per device
static __device__ __align__(256) unsigned char g_prefix_scratch[kStaticScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mutex;
void* g_scratch_addr[kMaxDevices] = {};

// Device address of g_prefix_scratch on the current device.
netkv_status static_scratch(cudaStream_t stream, void** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return NETKV_ECUDA;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(stream, &cap) != cudaSuccess) {
    cudaGetLastError();
    return NETKV_ECUDA;
  }
  std::lock_guard<std::mutex> lock(g_scratch_mutex);
  if (cap == cudaStreamCaptureStatusNone || !g_scratch_addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_prefix_scratch) != cudaSuccess || !p) {
      cudaGetLastError();
      return NETKV_ECUDA;
    }
    g_scratch_addr[dev] = p;
  }
  *out = g_scratch_addr[dev];
  return NETKV_OK;
}

}  // namespace

static_assert(NETKV_PREFIX_MATCH_STATIC_MAX_R > 0, "limit must be positive");

extern "C" netkv_status netkv_prefix_match_static(const void* d_index, uint32_t D,
                                                  uint32_t log2_capacity, uint32_t n_sets,
                                                  const uint64_t* d_chains,
                                                  const uint64_t* d_chain_off, uint32_t R,
                                                  const uint32_t* d_set_off, uint16_t* d_M,
                                                  int* d_status, netkv_stream_t stream) {
  if (R > NETKV_PREFIX_MATCH_STATIC_MAX_R ||
      netkv_prefix_match_workspace_size(R) > kStaticScratchBytes)
    return NETKV_ELIMIT;
  void* scratch = nullptr;
  const netkv_status st = static_scratch((cudaStream_t)stream, &scratch);
  if (st != NETKV_OK) return st;
  return netkv_prefix_match(d_index, D, log2_capacity, n_sets, d_chains, d_chain_off, R,
                            d_set_off, scratch, kStaticScratchBytes, d_M, d_status, stream);
}
