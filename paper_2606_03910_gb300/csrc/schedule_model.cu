// The greedy's walks with one CTA per stream: warp 0 walks the stream's events in order, the
// other warps ("producers") work one window of events ahead and put what an arrival's
// candidates contribute besides the stream's own state into shared memory.
//
//   plain            base scores precomputed in global memory (base_kernel): copied
//   self-contention  Eq. 4's n_inflight: network and prefix terms without contention, and
//                    the parts contention needs, computed by the producers
//   load model       Sec. IV-B: network and prefix terms and missed tokens, by the producers
//
// So an arrival costs the walker one or two shared-memory loads, a fused multiply-add and a
// comparison per decode, and a warp reduction; windows are double-buffered and the two
// sides meet at one block barrier a window.  Scores are those of schedule_kernel bit for
// bit (the same expressions on the same values); that kernel, which evaluates the
// candidates between two events, spends 1.3 us an event on the last two forms.
//   schedule_small_kernel  pools of at most 32 decodes: lane d holds decode d's state in
//                          registers and the argmin is one reduction and one ballot
//   schedule_model_kernel  larger pools, self-contention and load model: the state lies in
//                          shared memory, a lane takes pairs of decodes
// Bound by the walker's chain of dependent instructions per event.
#include <math.h>

#include "score.cuh"

namespace {

constexpr uint32_t kBadCode = 0xffffffffu;
constexpr uint32_t kMaxWindow = 32;         // events per window: one a lane
constexpr int kAhead = 4;                   // candidates a producer thread has in flight
constexpr size_t kModelSmem = 227u * 1024u; // dynamic shared memory of one CTA

enum EventType : uint32_t { kNoEvent = 0, kArrival = 1, kDeparture = 2, kBadArrival = 3 };

// An event with what its candidates share, filled one window ahead.
// ref: where a departure's decode is known from: kRefGlobal (dd, read from global memory),
// kRefPrev | slot (its arrival in the window before), kRefOwn | slot (earlier in its own
// window); kRefSlow: released by itself, not with the sums.  count: the window's arrivals
// before a departure; for an arrival whose request departs once in its window, 1 + that
// departure's count, else 0.
struct __align__(16) ModelEvent {
  uint4 lp;        // the prefill's links
  float4 ubp;      // and level bottlenecks
  uint32_t code, type, l, pr;
  long long now;   // arrival time (self-contention)
  int32_t dd;
  uint32_t miss;   // a departure's missed tokens on dd (load model)
  uint32_t k, ref, count, pad;
};
constexpr uint32_t kRefGlobal = 0u, kRefPrev = 0x100u, kRefOwn = 0x200u, kRefSlow = 0x400u;
constexpr uint32_t kSumTokens = 1u << 27;  // below: a window's sum of 32 fits in 32 bits

enum Walk { kPlain = 0, kContend = 1, kModel = 2 };

// A candidate under self-contention: apart from its score without contention, the parts
// that contention needs (read only while a counter of the prefill is up).
struct __align__(16) XferRow {
  float s_eff, bb, miss;
  uint32_t tau;
};
// Whole microseconds of a transfer time (at most 2^31 - 1).
__device__ __forceinline__ int32_t whole_us(float T) {
  const float us = T * 1.0e6f;
  return (int32_t)(us < 2147483520.0f ? __float2ll_rn(us) : 2147483647ll);
}
// (float)x of a load: through int32 when it fits (the same value, without the slow 64-bit
// conversion, which stays out of line so that it is not evaluated on the common path)
__device__ __noinline__ float wide_to_float(int64_t x) { return (float)x; }
__device__ __forceinline__ float load_to_float(int64_t x) {
  if (__builtin_expect(x == (int64_t)(int32_t)x, 1)) return (float)(int32_t)x;
  return wide_to_float(x);
}
__device__ __forceinline__ float latency_of(const TopoArgs& t, uint32_t tau) {
  return tau == 0 ? t.lat[0] : tau == 1 ? t.lat[1] : tau == 2 ? t.lat[2] : t.lat[3];
}

// Byte offsets of the dynamic shared memory.
// Rows of candidates are padded to an even number of decodes, so that pairs load as one.
__host__ __device__ inline uint32_t row_stride(uint32_t D) { return (D + 1u) & ~1u; }

struct ModelLayout {
  uint32_t win;
  uint32_t ev, arr, narr, wd, wmiss, wb, ws, wx, state, tok, term, held, cnt, heap, rel, base, rows, dt,
      total;
};

ModelLayout model_layout(Walk walk, bool small, uint32_t D, uint32_t P, uint32_t heap_cap,
                         uint32_t win) {
  ModelLayout a;
  uint32_t at = 0;
  auto take = [&](size_t bytes) {
    const uint32_t o = at;
    at += (uint32_t)((bytes + 15) / 16 * 16);
    return o;
  };
  const bool infl = walk == kContend;
  const size_t cand = (size_t)2 * win * row_stride(D);
  a.win = win;
  a.ev = take(2 * win * sizeof(ModelEvent));
  a.arr = take(2 * kMaxWindow * 4);
  a.narr = take(2 * 4);
  // state and results of the larger pools; the small walk keeps both in registers
  a.wd = take(small ? 0 : 2 * kMaxWindow * 4);
  a.wmiss = take(small ? 0 : 2 * kMaxWindow * 4);
  a.wb = take(small ? 0 : kMaxWindow * 4);
  a.ws = take(small ? 0 : kMaxWindow * 4);
  a.wx = take(small ? 0 : kMaxWindow * 4);
  a.state = take(small ? 0 : (size_t)D * 8);              // load or free bytes
  a.tok = take(small || walk != kModel ? 0 : (size_t)D * 8);
  a.term = take(small ? 0 : (size_t)row_stride(D) * 8);               // (tokens that fit, load term)
  a.held = take(small || walk != kModel ? 0 : (size_t)D * 4);
  a.cnt = take(infl ? (size_t)(P < 32 ? 32 : P) * 4 : 0);
  a.heap = take(infl ? (size_t)heap_cap * 8 : 0);
  a.rel = take(small ? (size_t)(kMaxWindow + 1) * 32 * (walk == kModel ? 8 : 4) : 0);
  a.base = take(cand * (walk == kModel ? 8 : 4));
  a.rows = take(infl ? cand * sizeof(XferRow) : 0);
  a.dt = take(infl ? cand * sizeof(int2) : 0);
  a.total = at;
  return a;
}

struct ModelArgs {
  TopoArgs t;
  const netkv_weights* W;
  uint32_t R, n_snap;
  const uint32_t *len, *prefill, *snap;
  const uint16_t* M;
  const float* UB;
  const float* base;          // plain: [R][D] base scores
  const uint32_t* events;
  const uint64_t* event_off;
  const int64_t* state_init;  // loads, or free bytes
  int32_t* dec;
  float *best, *second;
  int64_t* state_final;
  int* status;
  const int64_t* arrival_us;  // self-contention
  uint32_t inflight_cap, heap_cap;
  int32_t* xfer_us;
  LoadModel lm;               // load model
  const int32_t* held_init;
  int32_t* held_final;
  ModelLayout lay;
};

// The shared memory of a block, by name.
struct ModelShared {
  ModelEvent* ev;    // [2][win]
  uint32_t* arr;     // [2][kMaxWindow] slots of a window's arrivals
  uint32_t* narr;    // [2]
  float* base;       // [2][win][row_stride(D)]
  uint2* cand;       // load model: (score, missed tokens)
  XferRow* rows;     // [2][win][row_stride(D)]
  int2* dt;          // [2][win][row_stride(D)] uncontended transfer time in us, tier
  uint32_t* cnt;     // self-contention: n_inflight, byte `tier` of cnt[prefill rank]
  __device__ ModelShared(unsigned char* smem, const ModelLayout& l)
      : ev(reinterpret_cast<ModelEvent*>(smem + l.ev)),
        arr(reinterpret_cast<uint32_t*>(smem + l.arr)),
        narr(reinterpret_cast<uint32_t*>(smem + l.narr)),
        base(reinterpret_cast<float*>(smem + l.base)),
        cand(reinterpret_cast<uint2*>(smem + l.base)),
        rows(reinterpret_cast<XferRow*>(smem + l.rows)),
        dt(reinterpret_cast<int2*>(smem + l.dt)),
        cnt(reinterpret_cast<uint32_t*>(smem + l.cnt)) {}
};

// The producers: in step k of the block they fill window k while the walker walks window
// k - 1; every step ends with a block barrier.
// Warps 4, 8, ... share warp 0's scheduler and only keep the barriers: a producer there took
// issue slots from the walker (262 decodes under the load model: 459 us with all warps
// producing, of which 68 were theirs).
template <Walk kWalk, int BT>
__device__ __forceinline__ void produce(const ModelArgs& a, const netkv_weights& w,
                                        const ModelShared& S, uint64_t e0, uint64_t e1,
                                        uint64_t n_win) {
  constexpr uint32_t NP = BT == 64 ? 32u : BT / 4 * 3;  // producing threads
  const TopoArgs& t = a.t;
  const uint32_t wid = threadIdx.x >> 5;
  if (wid % 4 == 0) {
    for (uint64_t k = 0; k <= n_win; ++k) __syncthreads();
    return;
  }
  const uint32_t D = t.D, win = a.lay.win;
  const uint32_t ptid = (wid - 1 - wid / 4) * 32 + (threadIdx.x & 31);
  const uint32_t step_q = NP / D, step_d = NP % D;
  bool have = ptid < win && e0 + ptid < e1;  // whether the lane has an event in the window
  uint32_t code = have ? __ldg(a.events + e0 + ptid) : kBadCode;
  uint32_t prev_r = kBadCode;  // lane j: event j of the window before: its request, if an arrival
  for (uint64_t k = 0; k <= n_win; ++k) {
    if (k < n_win) {
      ModelEvent* ev = S.ev + (k & 1) * win;
      uint32_t* arr = S.arr + (k & 1) * kMaxWindow;
      if (ptid < 32) {
        ModelEvent x;
        x.lp = make_uint4(0, 0, 0, 0);
        x.ubp = make_float4(0.f, 0.f, 0.f, 0.f);
        x.code = code;
        x.type = kNoEvent;
        x.l = x.pr = x.miss = x.k = x.count = x.pad = 0;
        x.ref = kRefGlobal;
        x.now = 0;
        x.dd = -1;
        const uint32_t r = code & 0x7fffffffu;
        const uint64_t e = e0 + (k + 1) * win + ptid;
        const bool have_next = ptid < win && e < e1;
        const uint32_t next = have_next ? __ldg(a.events + e) : kBadCode;
        if (!have) {
        } else if (r >= a.R) {
          flag_status(a.status, NETKV_DEV_ERANGE);
        } else if (code >> 31) {
          x.type = kDeparture;
          x.l = __ldg(a.len + r);
          x.dd = __ldcg(a.dec + r);  // by the walker, up to the window before the walked one
          if (kWalk == kModel && x.dd >= 0 && (uint32_t)x.dd < D)
            x.miss = x.l - min(16u * (uint32_t)__ldg(a.M + (uint64_t)r * D + x.dd), x.l);
        } else {
          x.l = __ldg(a.len + r);
          x.pr = __ldg(a.prefill + r);
          x.k = __ldg(a.snap + r);
          if (kWalk == kContend) x.now = __ldg(a.arrival_us + r);
          if (x.pr < t.P && x.k < a.n_snap && x.l != 0) {
            x.type = kArrival;
            if (kWalk != kPlain) {
              const uint32_t pinst = __ldg(t.pre + x.pr);
              x.lp = __ldg(t.links + pinst);
              x.ubp = __ldg(reinterpret_cast<const float4*>(a.UB) + (uint64_t)x.k * t.N + pinst);
            }
          } else {
            x.type = kBadArrival;
            flag_status(a.status, x.l == 0 ? NETKV_DEV_EDOMAIN : NETKV_DEV_ERANGE);
          }
        }
        code = next;
        have = have_next;
        // the window's arrivals, in order, and each departure's arrival when that lies in
        // this window or the one before (their decisions are not recorded yet)
        const bool is_arr = x.type == kArrival || x.type == kBadArrival;
        const bool is_dep = x.type == kDeparture;
        const uint32_t any_arr = __ballot_sync(0xffffffffu, is_arr);
        const uint32_t list = __ballot_sync(0xffffffffu, x.type == kArrival);
        const uint32_t deps = __ballot_sync(0xffffffffu, is_dep);
        const uint32_t below = (1u << ptid) - 1u;
        const uint32_t er = x.type == kNoEvent ? kBadCode : r;
        if (deps) {
          for (uint32_t j = 0; j < win; ++j) {
            const uint32_t rj = __shfl_sync(0xffffffffu, prev_r, j);
            if (is_dep && rj == r) x.ref = kRefPrev | j;
          }
          const uint32_t same = __match_any_sync(0xffffffffu, er);
          const uint32_t mate = same & any_arr & below;               // a departure's arrival
          const uint32_t leave = same & deps & ~below & ~(1u << ptid);  // an arrival's departures
          if (is_dep) {
            x.count = __popc(list & below);
            if (mate) {
              const uint32_t slot = 31u - __clz(mate);
              x.ref = kRefOwn | slot;
              // the arrival's dispatch releases it, unless it is large or departs twice
              if (__popc(same & deps & ~((2u << slot) - 1u)) != 1) x.ref |= kRefSlow;
            }
            if (x.l >= kSumTokens) x.ref |= kRefSlow;
          } else if (x.type == kArrival && __popc(leave) == 1 && x.l < kSumTokens) {
            x.count = 1u + __popc(list & ((1u << (__ffs(leave) - 1)) - 1u));
          }
        }
        prev_r = is_arr ? r : kBadCode;
        if (ptid < win) ev[ptid] = x;
        if (x.type == kArrival) arr[__popc(list & below)] = ptid;
        if (ptid == 0) S.narr[k & 1] = __popc(list);
      }
      if (BT == 64) __syncwarp();
      else asm volatile("bar.sync 1, %0;" ::"n"(NP) : "memory");
      // candidates (arrival, decode), decodes fastest, kAhead of a thread in flight
      const uint32_t na = S.narr[k & 1];
      uint32_t q = ptid / D, d = ptid % D;
      while (q < na) {
        uint32_t ci[kAhead], cd[kAhead], m[kAhead], inst[kAhead];
        uint4 ld[kAhead];
        float ubd[kAhead];
        int tau[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
          ci[u] = q < na ? arr[q] : kNone;
          cd[u] = d;
          if (ci[u] != kNone) {
            const uint64_t at = (uint64_t)(ev[ci[u]].code & 0x7fffffffu) * D + d;
            if (kWalk == kPlain) {
              ubd[u] = __ldg(a.base + at);
            } else {
              inst[u] = __ldg(t.dec + d);
              m[u] = __ldg(a.M + at);
            }
          }
          q += step_q;
          d += step_d;
          if (d >= D) {
            d -= D;
            ++q;
          }
        }
        if (kWalk != kPlain) {
#pragma unroll
          for (int u = 0; u < kAhead; ++u)
            if (ci[u] != kNone) ld[u] = __ldg(t.links + inst[u]);
#pragma unroll
          for (int u = 0; u < kAhead; ++u)
            if (ci[u] != kNone) {
              const ModelEvent& x = ev[ci[u]];
              tau[u] = tier_of(x.lp, ld[u]);
              ubd[u] = __ldg(a.UB + ((uint64_t)x.k * t.N + inst[u]) * 4 + tau[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
          if (ci[u] == kNone) continue;
          const size_t at = ((k & 1) * win + ci[u]) * (size_t)row_stride(D) + cd[u];
          if (kWalk == kPlain) {
            S.base[at] = ubd[u];
            continue;
          }
          const ModelEvent& x = ev[ci[u]];
          const float ubp = pick4(x.ubp, tau[u]), lat = latency_of(t, (uint32_t)tau[u]);
          if (kWalk == kContend) {
            const XferParts p = xfer_parts(w, x.l, m[u], ubp, ubd[u], a.status);
            const float T = xfer_time(p, 0u, lat);
            S.base[at] = w.w_net * T + w.w_prefix * p.miss;
            S.rows[at] = XferRow{p.s_eff, p.bb, p.miss, (uint32_t)tau[u]};
            S.dt[at] = make_int2(whole_us(T), tau[u]);
          } else {
            const float b = base_score(w, x.l, m[u], ubp, ubd[u], lat, a.status);
            S.cand[at] = make_uint2(__float_as_uint(b), x.l - min(16u * m[u], x.l));
          }
        }
      }
    }
    __syncthreads();  // window k is ready, window k - 1 has been walked
  }
}

// The pending completions of a stream and its counters.  The lanes of the walker hold 32 of
// them, one each, in no order (lowering a counter, floored at zero, commutes); more go to a
// heap kept by lane 0, out of line.
__device__ __forceinline__ void lower_counter(uint32_t* cnt, uint32_t pt) {
  uint32_t* c = cnt + (pt >> 2);
  const uint32_t sh = 8u * (pt & 3u);
  if ((*c >> sh) & 0xffu) *c -= 1u << sh;
}
__device__ __noinline__ uint32_t heap_settle(unsigned long long* a, uint32_t n, uint32_t cap,
                                             uint32_t* cnt, long long now) {
  DoneHeap h = {a, n, cap};
  while (h.n > 0 && (int64_t)(h.a[0] >> 16) <= now) {
    lower_counter(cnt, (uint32_t)(h.a[0] & 0xffffu));
    h.pop();
  }
  return h.n;
}
__device__ __noinline__ void heap_push(unsigned long long* a, uint32_t n, uint32_t cap,
                                       unsigned long long key) {
  DoneHeap h = {a, n, cap};
  h.push(key);
}
template <bool kRegs>  // counters of at most 32 prefill ranks: lane p holds rank p's
struct Completions {
  static constexpr unsigned long long kFree = ~0ull;  // above every key: prefill < 2^14 - 1
  unsigned long long key;  // time in us << 16 | prefill rank << 2 | tier
  uint32_t in_heap;        // the same in every lane
  uint32_t mine;           // kRegs: the lane's counters
  __device__ Completions() : key(kFree), in_heap(0), mine(0) {}
  // The counters of prefill pr, a byte per tier.
  __device__ __forceinline__ uint32_t counters(const uint32_t* cnt, uint32_t pr) const {
    return kRegs ? __shfl_sync(0xffffffffu, mine, pr) : cnt[pr];
  }
  // Transfers completed by `now` lower their counters (Algorithm 1 line 14's callback).
  __device__ __forceinline__ void settle(const ModelArgs& a, unsigned char* smem, uint32_t* cnt,
                                         long long now, uint32_t lane) {
    const bool due = key != kFree && (int64_t)(key >> 16) <= now;
    uint32_t dm = __ballot_sync(0xffffffffu, due);
    if (!dm && !in_heap) return;
    while (dm) {
      const uint32_t j = __ffs(dm) - 1;
      dm &= dm - 1;
      if (kRegs) {
        const uint32_t pt = __shfl_sync(0xffffffffu, (uint32_t)key & 0xffffu, j);
        const uint32_t sh = 8u * (pt & 3u);
        if (lane == pt >> 2 && ((mine >> sh) & 0xffu)) mine -= 1u << sh;
      } else {
        if (lane == j) lower_counter(cnt, (uint32_t)key & 0xffffu);
        __syncwarp();
      }
    }
    if (due) key = kFree;
    if (in_heap) {
      if (kRegs) cnt[lane] = mine;  // the heap lowers them in memory
      __syncwarp();
      if (lane == 0)
        in_heap = heap_settle(reinterpret_cast<unsigned long long*>(smem + a.lay.heap), in_heap,
                              a.heap_cap, cnt, now);
      in_heap = __shfl_sync(0xffffffffu, in_heap, 0);
      __syncwarp();
      if (kRegs) mine = cnt[lane];
    }
  }
  // A dispatch on tier tau of prefill pr, whose counters are cw: the counter and the
  // completion at now + dt.
  __device__ __forceinline__ void dispatch(const ModelArgs& a, unsigned char* smem, uint32_t* cnt,
                                           long long now, int32_t dt, uint32_t pr, uint32_t tau,
                                           uint32_t cw, uint32_t lane) {
    const uint32_t free = __ballot_sync(0xffffffffu, key == kFree);
    const unsigned long long k = ((unsigned long long)(now + dt) << 16) |
                                 ((unsigned long long)pr << 2) | tau;
    const uint32_t sh = 8u * tau;
    const uint32_t at = free ? (uint32_t)(__ffs(free) - 1) : 0u;
    const bool full = 32u - __popc(free) + in_heap >= a.heap_cap;
    const bool up = ((cw >> sh) & 0xffu) < a.inflight_cap;
    if (kRegs && up && lane == pr) mine += 1u << sh;
    if (lane == at) {
      if (!kRegs && up) cnt[pr] = cw + (1u << sh);
      if (full) flag_status(a.status, NETKV_DEV_EFULL);
      else if (free) key = k;
      else heap_push(reinterpret_cast<unsigned long long*>(smem + a.lay.heap), in_heap, a.heap_cap, k);
    }
    if (!full && !free) ++in_heap;
    if (!kRegs || !free) __syncwarp();
  }
};

// The score of a candidate under contention cw (the counters of its prefill's tiers).
__device__ __forceinline__ float contended(const TopoArgs& t, const netkv_weights& w,
                                           const XferRow& x, uint32_t cw, float uncontended) {
  const uint32_t n = (cw >> (8u * x.tau)) & 0xffu;
  if (n == 0) return uncontended;
  const XferParts p = {x.s_eff, x.bb, x.miss};
  const float T = xfer_time(p, n, latency_of(t, x.tau));
  return w.w_net * T + w.w_prefix * p.miss;
}

// kRegs: at most 32 prefill ranks (self-contention).  Blocks of 128 threads are for few
// streams: registers without spills; blocks of 64 for many: residency.
template <Walk kWalk, int BT, bool kRegs>
__global__ void __launch_bounds__(BT, BT >= 128 ? 512 / BT : 1024 / BT)
    schedule_small_kernel(ModelArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const TopoArgs& t = a.t;
  const uint32_t D = t.D, win = a.lay.win, lane = threadIdx.x & 31;
  const uint32_t stream = blockIdx.x;
  const netkv_weights w = a.W[stream];
  const ModelShared S(smem, a.lay);
  const uint64_t e0 = a.event_off[stream], e1 = a.event_off[stream + 1];
  const uint64_t n_win = e1 > e0 ? (e1 - e0 + win - 1) / win : 0;
  if (threadIdx.x >= 32) {
    produce<kWalk, BT>(a, w, S, e0, e1, n_win);
    return;
  }

  // ---- the walker: lane d holds decode d
  const bool mine = lane < D;
  uint32_t* rel = reinterpret_cast<uint32_t*>(smem + a.lay.rel);  // [kMaxWindow + 1][32]
  uint32_t* reln = rel + (kMaxWindow + 1) * 32;                   // load model: departures
  for (uint32_t q = lane; q < (kMaxWindow + 1) * 32; q += 32) {
    rel[q] = 0u;
    if (kWalk == kModel) reln[q] = 0u;
  }
  int64_t state = kWalk == kModel ? a.lm.m0 : 0;  // load, or free bytes
  int32_t held = 0;
  if (mine && a.state_init) state = a.state_init[(uint64_t)stream * D + lane];
  if (kWalk == kModel && mine && a.held_init) held = a.held_init[(uint64_t)stream * D + lane];
  const int64_t bpt = (int64_t)w.bytes_per_token;
  // what the last dispatch took on its decode's lane (tokens, or missed tokens of one
  // request), applied with the releases before the next arrival
  uint32_t own = 0, own_n = 0;
  Completions<kRegs> done_at;
  if (kWalk == kContend && !kRegs)
    for (uint32_t p = lane; p < t.P; p += 32) S.cnt[p] = 0u;
  __syncwarp();

  int32_t prev_d = -1;  // lane j: event j of the window before: its decision
  uint32_t prev_miss = 0;  // and its missed tokens there
  for (uint64_t k = 0; k <= n_win; ++k) {
    if (k > 0) {
      const uint32_t buf = (uint32_t)((k - 1) & 1);
      const ModelEvent* ev = S.ev + buf * win;
      // lane i prepares event i
      uint32_t type = kNoEvent, r = kBadCode, l_ev = 0, miss_ev = 0, pr_ev = 0, ref = 0, count = 0;
      int32_t dd = -1;
      long long now_ev = 0;
      if (lane < win) {
        const ModelEvent& x = ev[lane];
        type = x.type;
        l_ev = x.l;
        dd = x.dd;
        miss_ev = x.miss;
        ref = x.ref;
        count = x.count;
        if (kWalk == kContend) {
          pr_ev = x.pr;
          now_ev = x.now;
        }
        r = x.code & 0x7fffffffu;
      }
      const bool is_arr = type == kArrival || type == kBadArrival;
      const uint32_t arrivals = __ballot_sync(0xffffffffu, type == kArrival);
      const bool slow = type == kDeparture && (ref & kRefSlow);
      const uint32_t my_bj = type == kArrival ? count : 0u;
      {
        const int32_t pd = __shfl_sync(0xffffffffu, prev_d, ref & 31u);
        const uint32_t pm = kWalk == kModel ? __shfl_sync(0xffffffffu, prev_miss, ref & 31u) : 0u;
        if (ref & kRefPrev) {
          dd = pd;
          miss_ev = pm;
        }
      }
      if (type == kDeparture && !(ref & (kRefOwn | kRefSlow)) && dd >= 0 && (uint32_t)dd < D) {
        // tokens released before the window's count-th arrival
        atomicAdd(&rel[count * 32 + dd], kWalk == kModel ? miss_ev : l_ev);
        if (kWalk == kModel) atomicAdd(&reln[count * 32 + dd], 1u);
      }
      __syncwarp();
      const uint32_t leaving = __ballot_sync(0xffffffffu, my_bj != 0u);
      uint32_t left = __ballot_sync(0xffffffffu, slow);  // slow departures not applied yet
      int32_t my_d = -1, my_x = -1;  // lane i: event i's decision, transfer time,
      uint32_t my_miss = 0, my_b = kNoKey, my_s = kNoKey;  // missed tokens there, score keys
      // the departures of slots in `bits`, one by one
      auto apply = [&](uint32_t bits) {
        while (bits) {
          const uint32_t j = __ffs(bits) - 1;
          bits &= bits - 1;
          int32_t d = __shfl_sync(0xffffffffu, dd, j);
          const uint32_t l = __shfl_sync(0xffffffffu, l_ev, j);
          uint32_t m = __shfl_sync(0xffffffffu, miss_ev, j);
          const uint32_t rf = __shfl_sync(0xffffffffu, ref, j);
          const int32_t ds = __shfl_sync(0xffffffffu, my_d, rf & 31u);
          const uint32_t ms = __shfl_sync(0xffffffffu, my_miss, rf & 31u);
          if (rf & kRefOwn) {
            d = ds;
            m = ms;
          }
          if (mine && d == (int32_t)lane) {
            if (kWalk == kModel) {
              state += (int64_t)m * bpt;
              held -= 1;
            } else {
              state -= (int64_t)l;
            }
          }
        }
      };
      // an arrival's length, this lane's candidate and the releases before it: read one
      // arrival ahead
      uint32_t l_n = 0, rel_n = 0, reln_n = 0, miss_n = 0, pr_n = 0;
      long long now_n = 0;
      float net_n = 0.f;
      auto fetch = [&](uint32_t i) {
        const size_t row = (buf * win + i) * (size_t)row_stride(D);
        l_n = __shfl_sync(0xffffffffu, l_ev, i);
        if (kWalk == kContend) {
          pr_n = __shfl_sync(0xffffffffu, pr_ev, i);
          now_n = __shfl_sync(0xffffffffu, now_ev, i);
        }
        if (mine) {
          if (kWalk == kModel) {
            const uint2 c = S.cand[row + lane];
            net_n = __uint_as_float(c.x);
            miss_n = c.y;
          } else {
            net_n = S.base[row + lane];
          }
        }
      };
      auto fetch_rel = [&](uint32_t b) {
        rel_n = rel[b * 32 + lane];
        rel[b * 32 + lane] = 0u;
        if (kWalk == kModel) {
          reln_n = reln[b * 32 + lane];
          reln[b * 32 + lane] = 0u;
        }
      };
      // the last dispatch and the releases since
      auto advance = [&]() {
        if (kWalk == kModel) {
          state += ((int64_t)rel_n - (int64_t)own) * bpt;
          held += (int32_t)own_n - (int32_t)reln_n;
          own_n = 0;
        } else {
          state += (int64_t)own - (int64_t)rel_n;
        }
        own = 0;
      };
      uint32_t todo = arrivals, b = 0;
      if (todo) fetch(__ffs(todo) - 1);
      fetch_rel(0);
      while (todo) {
        const uint32_t i = __ffs(todo) - 1;
        todo &= todo - 1;
        const uint32_t l = l_n, miss = miss_n, pr = pr_n;
        const long long now = now_n;
        float net = net_n;
        advance();
        const uint32_t before = left & ((1u << i) - 1u);
        if (before) {
          apply(before);
          left &= ~before;
        }
        ++b;
        if (todo) fetch(__ffs(todo) - 1);
        fetch_rel(b);
        uint32_t cw = 0;
        const size_t row = (buf * win + i) * (size_t)row_stride(D);
        if (kWalk == kContend) {
          done_at.settle(a, smem, S.cnt, now, lane);
          cw = done_at.counters(S.cnt, pr);
          if (cw && mine) net = contended(t, w, S.rows[row + lane], cw, net);
        }
        bool feasible;
        float sc;
        if (kWalk == kModel) {
          feasible = mine && state >= (int64_t)miss * bpt + a.lm.m_min;
          sc = net + w.w_load * load_term(a.lm, held);
        } else {
          feasible = mine && state + (int64_t)l <= w.cap_tokens;
          sc = __fmaf_rn(w.w_load, w.theta_s_per_token * load_to_float(state), net);
        }
        const uint32_t key = feasible ? score_key(sc) : kNoKey;
        const uint32_t kb = __reduce_min_sync(0xffffffffu, key);
        const uint32_t at_best = __ballot_sync(0xffffffffu, key == kb);
        const uint32_t one = __reduce_min_sync(0xffffffffu, key == kb ? kNoKey : key);
        const int32_t dstar = kb == kNoKey ? -1 : (int32_t)(__ffs(at_best) - 1);
        if (dstar == (int32_t)lane) {
          own = kWalk == kModel ? miss : l;
          own_n = 1;
        }
        if (leaving >> i & 1u) {
          // the request departs in this window: its release waits with the others, or
          // cancels the dispatch where no arrival lies between
          const uint32_t bj = __shfl_sync(0xffffffffu, my_bj, i) - 1u;
          if (dstar == (int32_t)lane) {
            if (bj == b) {
              own = own_n = 0;
            } else {
              rel[bj * 32 + lane] += own;
              if (kWalk == kModel) reln[bj * 32 + lane] += 1u;
            }
          }
        }
        int32_t xfer = -1;
        if (kWalk == kContend && dstar >= 0) {
          const int2 tt = S.dt[row + dstar];
          const uint32_t tau = (uint32_t)tt.y, n = (cw >> (8u * tau)) & 0xffu;
          xfer = tt.x;
          if (n) {
            const XferRow x = S.rows[row + dstar];
            xfer = whole_us(xfer_time(XferParts{x.s_eff, x.bb, x.miss}, n, latency_of(t, tau)));
          }
          done_at.dispatch(a, smem, S.cnt, now, xfer, pr, tau, cw, lane);
        }
        const uint32_t taken =
            kWalk == kModel ? __shfl_sync(0xffffffffu, miss, dstar < 0 ? 0 : dstar) : 0u;
        if (lane == i) {
          my_d = dstar;
          my_miss = taken;
          my_x = xfer;
          my_b = kb;
          my_s = __popc(at_best) >= 2 ? kb : one;
        }
      }
      advance();  // after the window's last arrival
      apply(left);
      if (is_arr) {
        a.dec[r] = my_d;
        a.best[r] = key_score(my_b);
        a.second[r] = key_score(my_s);
        if (kWalk == kContend) a.xfer_us[r] = my_x;
      }
      prev_d = my_d;
      prev_miss = my_miss;
    }
    __syncthreads();
  }
  if (mine) {
    a.state_final[(uint64_t)stream * D + lane] = state;
    if (kWalk == kModel) a.held_final[(uint64_t)stream * D + lane] = held;
  }
}

// A decode's feasibility and load term, 8 bytes: (headroom, theta * load), a request of l
// tokens fits iff l <= headroom; load model: (free tokens + 1, T_queue + T_decode), a
// candidate fits iff its missed tokens are below the first.  There the free bytes above m_min
// are counted in whole tokens once and then change by the missed tokens of each dispatch
// and departure: floor((f - b * S) / b) = floor(f / b) - S.  That needs 0 < bytes_per_token
// < 2^31 (products of 32-bit token counts then stay in 63 bits); a stream with other bytes,
// and a request of 2^32 - 1 tokens, compare bytes instead.
template <Walk kWalk, int BT>
__global__ void __launch_bounds__(BT, BT >= 256 ? 512 / BT : 1024 / BT)
    schedule_model_kernel(ModelArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const TopoArgs& t = a.t;
  const uint32_t D = t.D, win = a.lay.win, lane = threadIdx.x & 31;
  const uint32_t stream = blockIdx.x;
  const netkv_weights w = a.W[stream];
  const ModelShared S(smem, a.lay);
  const uint64_t e0 = a.event_off[stream], e1 = a.event_off[stream + 1];
  const uint64_t n_win = e1 > e0 ? (e1 - e0 + win - 1) / win : 0;
  int32_t* s_wd = reinterpret_cast<int32_t*>(smem + a.lay.wd);          // [2][kMaxWindow]
  uint32_t* s_wmiss = reinterpret_cast<uint32_t*>(smem + a.lay.wmiss);  // [2][kMaxWindow]
  uint32_t* s_wb = reinterpret_cast<uint32_t*>(smem + a.lay.wb);
  uint32_t* s_ws = reinterpret_cast<uint32_t*>(smem + a.lay.ws);
  int32_t* s_wx = reinterpret_cast<int32_t*>(smem + a.lay.wx);
  int64_t* s_state = reinterpret_cast<int64_t*>(smem + a.lay.state);  // load, or free bytes
  int64_t* s_tok = reinterpret_cast<int64_t*>(smem + a.lay.tok);      // load model: in tokens
  uint2* s_hl = reinterpret_cast<uint2*>(smem + a.lay.term);
  int32_t* s_held = reinterpret_cast<int32_t*>(smem + a.lay.held);
  const int64_t bpt = (int64_t)w.bytes_per_token;
  const bool in_tokens = kWalk != kModel || (bpt > 0 && bpt < (1ll << 31));
  // `tok` whole tokens free: the bound that a candidate's missed tokens stay below
  auto below = [](int64_t tok) -> uint32_t {
    return tok < 0 ? 0u : tok >= 0xfffffffell ? 0xffffffffu : (uint32_t)tok + 1u;
  };
  auto hl_of_load = [&](int64_t ld) -> uint2 {
    return make_uint2(headroom(w.cap_tokens, ld),
                      __float_as_uint(w.theta_s_per_token * load_to_float(ld)));
  };
  // decode d after `delta` tokens more (load model: `delta` missed tokens of `n` requests less)
  auto change = [&](uint32_t d, int64_t delta, int32_t n) {
    if (kWalk == kModel) {
      const int64_t tok = s_tok[d] + delta;
      const int32_t h = s_held[d] - n;
      s_state[d] += delta * bpt;
      s_tok[d] = tok;
      s_held[d] = h;
      s_hl[d] = make_uint2(below(tok), __float_as_uint(load_term(a.lm, h)));
    } else {
      const int64_t ld = s_state[d] + delta;
      s_state[d] = ld;
      s_hl[d] = hl_of_load(ld);
    }
  };
  for (uint32_t d = threadIdx.x; d < D; d += BT) {  // the initial state, by the whole block
    int64_t x = kWalk == kModel ? a.lm.m0 : 0;
    if (a.state_init) x = a.state_init[(uint64_t)stream * D + d];
    s_state[d] = x;
    if (kWalk == kModel) {
      // x - m_min in whole tokens, rounded down, kept where a call's changes cannot overflow
      const int64_t f = x < INT64_MIN + a.lm.m_min ? INT64_MIN : x - a.lm.m_min;
      const int64_t tok = !in_tokens ? 0 : f / bpt - (f % bpt < 0 ? 1 : 0);
      s_tok[d] = max(INT64_MIN / 2, min(INT64_MAX / 2, tok));
      s_held[d] = a.held_init ? a.held_init[(uint64_t)stream * D + d] : 0;
      change(d, 0, 0);
    } else {
      s_hl[d] = hl_of_load(x);
    }
  }
  if (threadIdx.x == 0 && (D & 1u)) s_hl[D] = make_uint2(0u, 0u);  // the padding fits nothing
  if (kWalk == kContend)
    for (uint32_t p = threadIdx.x; p < t.P; p += BT) S.cnt[p] = 0u;
  __syncthreads();
  if (threadIdx.x >= 32) {
    produce<kWalk, BT>(a, w, S, e0, e1, n_win);
    return;
  }

  // ---- the walker: lane i takes decodes 2 i, 2 i + 1, 2 i + 64, ...
  Completions<false> done_at;
  for (uint64_t k = 0; k <= n_win; ++k) {
    if (k > 0) {
      const uint32_t buf = (uint32_t)((k - 1) & 1);
      const ModelEvent* ev = S.ev + buf * win;
      int32_t* wd = s_wd + buf * kMaxWindow;
      uint32_t* wmiss = s_wmiss + buf * kMaxWindow;
      const int32_t* pd = s_wd + (buf ^ 1) * kMaxWindow;
      const uint32_t* pmiss = s_wmiss + (buf ^ 1) * kMaxWindow;
      // lane i prepares event i
      uint32_t type = kNoEvent, r = kBadCode, my_l = 0, my_miss = 0, my_pr = 0, ref = 0;
      int32_t my_dd = -1;
      long long my_now = 0;
      if (lane < win) {
        const ModelEvent& x = ev[lane];
        type = x.type;
        my_l = x.l;
        my_pr = x.pr;
        my_now = x.now;
        my_dd = x.dd;
        my_miss = x.miss;
        ref = x.ref;
        r = x.code & 0x7fffffffu;
        if (ref & kRefPrev) {
          my_dd = pd[ref & 31u];
          my_miss = pmiss[ref & 31u];
        }
        if (type == kBadArrival) {
          wd[lane] = -1;
          s_wb[lane] = s_ws[lane] = kNoKey;
          s_wx[lane] = -1;
        }
      }
      const bool is_arr = type == kArrival || type == kBadArrival;
      const uint32_t dep_mask = __ballot_sync(0xffffffffu, type == kDeparture);
      uint32_t arr_mask = __ballot_sync(0xffffffffu, type == kArrival);
      uint32_t done = 0;  // events before `done` are applied
      __syncwarp();       // results of bad arrivals are visible
      // the departures between the last arrival and event `upto`, all at once: they commute
      auto depart = [&](uint32_t upto) {
        const uint32_t lo = done >= 32 ? 0u : ~0u << done;
        const uint32_t hi = upto >= 32 ? ~0u : (1u << upto) - 1u;
        const uint32_t bm = dep_mask & lo & hi;
        done = upto;
        if (!bm) return;
        uint32_t d = kNone, miss = my_miss;
        if ((bm >> lane) & 1u) {
          int32_t dd = my_dd;
          if (ref & kRefOwn) {
            dd = wd[ref & 31u];
            miss = wmiss[ref & 31u];
          }
          if (dd >= 0 && (uint32_t)dd < D) d = (uint32_t)dd;
        }
        const int64_t delta = kWalk == kModel ? (int64_t)miss : -(int64_t)my_l;
        // each lane releases its own decode; departures of one decode (rare) go one by one
        const bool one = __popc(bm) == 1;
        const uint32_t peers = one ? 0u : __match_any_sync(0xffffffffu, d);
        if (!one && __any_sync(0xffffffffu, d != kNone && __popc(peers) > 1)) {
          uint32_t rest = __ballot_sync(0xffffffffu, d != kNone);
          while (rest) {
            const uint32_t src = __ffs(rest) - 1;
            rest &= rest - 1;
            if (lane == src) change(d, delta, 1);
            __syncwarp();
          }
        } else if (d != kNone) {
          change(d, delta, 1);
        }
        __syncwarp();
      };
      while (arr_mask) {
        const uint32_t i = __ffs(arr_mask) - 1;
        arr_mask &= arr_mask - 1;
        const uint32_t l = __shfl_sync(0xffffffffu, my_l, i);
        const size_t row = (buf * win + i) * (size_t)row_stride(D);
        depart(i);
        done = i + 1;
        uint32_t pr = 0, cw = 0;
        long long now = 0;
        if (kWalk == kContend) {
          pr = __shfl_sync(0xffffffffu, my_pr, i);
          now = __shfl_sync(0xffffffffu, my_now, i);
          done_at.settle(a, smem, S.cnt, now, lane);
          cw = done_at.counters(S.cnt, pr);
        }
        // Each lane's best and second-best of its decodes: with base scores in two independent
        // chains (even and odd ranks) merged at the end (1,024 decodes: 107 against 133 us for
        // 128 arrivals on each of 64 streams), else in one (262 decodes under the load model:
        // 423 against 456 us).
        constexpr bool kTwo = kWalk == kPlain;
        const float inf = __int_as_float(0x7f800000);
        float b = inf, s2 = inf, bo = inf, so = inf;
        uint32_t ci = kNone, co = kNone;
        auto visit = [](float& cb, float& cs, uint32_t& cc, uint32_t d, bool feasible, float sc) {
          const bool take = feasible && (cc == kNone || sc < cb);
          cs = take ? cb : (feasible ? fminf(cs, sc) : cs);
          cb = take ? sc : cb;
          cc = take ? d : cc;
        };
        if (kWalk == kModel && (!in_tokens || l == kNone)) {  // see below(): 2^32 - 1 is a bound
          for (uint32_t d = lane; d < D; d += 32) {  // ranks rise within a lane, as below
            const uint2 c = S.cand[row + d];
            visit(b, s2, ci, d, s_state[d] >= (int64_t)c.y * bpt + a.lm.m_min,
                  __uint_as_float(c.x) + w.w_load * __uint_as_float(s_hl[d].y));
          }
        } else {
          constexpr int kUnroll = kWalk == kPlain ? 4 : 2;
#pragma unroll kUnroll
          for (uint32_t d = 2 * lane; d < D; d += 64) {
            const uint4 hl = *reinterpret_cast<const uint4*>(s_hl + d);
            if (kWalk == kModel) {
              const uint4 c = *reinterpret_cast<const uint4*>(S.cand + row + d);
              visit(b, s2, ci, d, c.y < hl.x,
                    __uint_as_float(c.x) + w.w_load * __uint_as_float(hl.y));
              visit(b, s2, ci, d + 1, c.w < hl.z,
                    __uint_as_float(c.z) + w.w_load * __uint_as_float(hl.w));
            } else {
              float2 net = *reinterpret_cast<const float2*>(S.base + row + d);
              if (kWalk == kContend && cw) {
                net.x = contended(t, w, S.rows[row + d], cw, net.x);
                if (d + 1 < D) net.y = contended(t, w, S.rows[row + d + 1], cw, net.y);
              }
              // load + l <= cap (l >= 1 here)
              visit(b, s2, ci, d, l <= hl.x,
                    __fmaf_rn(w.w_load, __uint_as_float(hl.y), net.x));
              visit(kTwo ? bo : b, kTwo ? so : s2, kTwo ? co : ci, d + 1, l <= hl.z,
                    __fmaf_rn(w.w_load, __uint_as_float(hl.w), net.y));
            }
          }
        }
        if (kTwo) {
          const bool other = bo < b || (bo == b && co < ci);
          s2 = other ? fminf(so, b) : fminf(s2, bo);
          b = other ? bo : b;
          ci = other ? co : ci;
        }
        // (key, rank) argmin and second key: the rank and the second depend only on the key
        const uint32_t key = ci == kNone ? kNoKey : score_key(b);
        const uint32_t kb = __reduce_min_sync(0xffffffffu, key);
        const bool at_best = key == kb;
        const uint32_t bi = __reduce_min_sync(0xffffffffu, at_best ? ci : kNone);
        const uint32_t ties = __popc(__ballot_sync(0xffffffffu, at_best));
        const uint32_t one = __reduce_min_sync(0xffffffffu, at_best ? score_key(s2) : key);
        const uint32_t ks = ties >= 2 ? kb : one;
        const int32_t dstar = kb == kNoKey ? -1 : (int32_t)bi;
        int32_t xfer = -1;
        uint32_t miss = 0;
        if (dstar >= 0) {
          if (kWalk == kModel) miss = S.cand[row + dstar].y;
          if (lane == 0) {
            if (kWalk == kModel) change((uint32_t)dstar, -(int64_t)miss, -1);
            else change((uint32_t)dstar, (int64_t)l, 0);
          }
          if (kWalk == kContend) {
            const int2 tt = S.dt[row + dstar];
            const uint32_t tau = (uint32_t)tt.y, n = (cw >> (8u * tau)) & 0xffu;
            xfer = tt.x;
            if (n) {
              const XferRow x = S.rows[row + dstar];
              xfer = whole_us(xfer_time(XferParts{x.s_eff, x.bb, x.miss}, n, latency_of(t, tau)));
            }
            done_at.dispatch(a, smem, S.cnt, now, xfer, pr, tau, cw, lane);
          }
        }
        if (lane == 0) {
          wd[i] = dstar;
          wmiss[i] = miss;
          s_wb[i] = kb;
          s_ws[i] = ks;
          s_wx[i] = xfer;
        }
        __syncwarp();
      }
      depart(32);  // departures after the window's last arrival
      if (is_arr) {
        a.dec[r] = wd[lane];
        a.best[r] = key_score(s_wb[lane]);
        a.second[r] = key_score(s_ws[lane]);
        if (kWalk == kContend) a.xfer_us[r] = s_wx[lane];
      }
    }
    __syncthreads();
  }
  for (uint32_t d = lane; d < D; d += 32) {
    a.state_final[(uint64_t)stream * D + d] = s_state[d];
    if (kWalk == kModel) a.held_final[(uint64_t)stream * D + d] = s_held[d];
  }
}

// The attribute is per device: set before every launch that needs it.
template <typename Kernel>
netkv_status launch_walk(Kernel kernel, const ModelArgs& a, uint32_t n_streams, uint32_t bt,
                         cudaStream_t s) {
  if (a.lay.total > 48u * 1024u)
    NETKV_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)kModelSmem));
  kernel<<<n_streams, bt, a.lay.total, s>>>(a);
  return netkv_launch_status();
}

// Whether a stream's walk by one warp pays.  The rows of a window leave room for few CTAs an SM
// over large pools, where the other kernels score with several warps a stream, and the packed
// per-event walk puts 2 or 4 streams of up to 16 decodes into a warp.  60 requests a stream,
// this walk against the other (us):
//   base scores      577 decodes, 608 streams 200 / 327, 912 513 / 475; 1,024, 304 141 / 187,
//                    456 314 / 270
//   self-contention  16 decodes, 2,432 streams 131 / 140, 4,864 205 / 160; 8, 3,648 144 / 164,
//                    4,864 178 / 166; 96, 608 145 / 262, 760 350 / 281; 192, 304 119 / 139, 456
//                    252 / 162, 760 1,024 / 289; 32 and 64 at 4,864 575 / 691 and 1,018 / 1,600
//   load model       8 decodes, 4,864 streams 102 / 117, 7,296 148 / 124; 16, 2,432 85 / 101,
//                    3,648 146 / 110; 32, 1,216 72 / 76, 2,432 156 / 90; 192, 608 112 / 203, 760
//                    256 / 223; 577, 304 121 / 192, 456 445 / 350; 800, 152 98 / 168, 304
//                    245 / 204
template <Walk kWalk>
bool walk_pays(uint32_t D, uint32_t n_streams, uint32_t sms) {
  const uint32_t per_sm = (n_streams + sms - 1) / sms;
  const uint64_t pool = (uint64_t)D * n_streams;
  if (kWalk == kPlain) return D <= 512 || (pool <= 512u * 1024u && per_sm <= (D <= 800 ? 4u : 2u));
  if (D > 96 && pool > 256u * 1024u) return false;
  if (kWalk == kContend) {
    if (D <= 16) return per_sm <= (D <= 8 ? 28u : 20u);
    return D <= 64 || per_sm <= (D <= 128 ? 4u : 2u);
  }
  if (D <= 32) return per_sm <= (D <= 8 ? 32u : D <= 16 ? 16u : 8u);
  return D <= 128 || per_sm <= (D <= 400 ? 4u : D <= 600 ? 2u : 1u);
}

// Launches the walk when the pool fits: false (and nothing launched) otherwise.  Windows of
// 32 events hide the producers' round trips best; shorter ones where the rows of a larger
// pool need the memory, or more streams than the card's SMs hold at once.
template <Walk kWalk>
bool launch_model(ModelArgs& a, uint32_t n_streams, cudaStream_t s, netkv_status* result) {
  *result = NETKV_OK;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    *result = NETKV_ECUDA;
    return true;
  }
  const uint32_t D = a.t.D;
  const bool small = D <= 32;
  if (!walk_pays<kWalk>(D, n_streams, (uint32_t)sms)) return false;
  // producers enough for a window's candidates (about 16 arrivals) in a few rounds while
  // every stream is resident
  uint32_t bt = 64u;
  if (small) {
    if (kWalk != kPlain && n_streams <= 4u * (uint32_t)sms) bt = 128u;
  } else {
    bt = D <= 96 || (kWalk == kPlain && D <= 512) ? 256u : 512u;
    while (bt > 64u && (uint64_t)n_streams * bt > (uint64_t)sms * 512u) bt /= 2;
  }
  const uint32_t per_sm = (n_streams + (uint32_t)sms - 1) / (uint32_t)sms;
  const uint32_t most = 1024u / bt < per_sm ? 1024u / bt : per_sm;
  uint32_t win = 0;
  for (uint32_t x = kMaxWindow; x >= 8; x /= 2) {
    const ModelLayout l = model_layout(kWalk, small, D, a.t.P, a.heap_cap, x);
    if (l.total > kModelSmem) continue;
    win = x;
    if ((size_t)l.total * most <= kModelSmem) break;
  }
  if (win == 0) return false;
  a.lay = model_layout(kWalk, small, D, a.t.P, a.heap_cap, win);
  const bool regs = kWalk == kContend && a.t.P <= 32;
  if (small && bt == 128u) {
    if (regs) *result = launch_walk(schedule_small_kernel<kWalk, 128, kWalk == kContend>, a, n_streams, bt, s);
    else *result = launch_walk(schedule_small_kernel<kWalk, 128, false>, a, n_streams, bt, s);
  } else if (small) {
    if (regs) *result = launch_walk(schedule_small_kernel<kWalk, 64, kWalk == kContend>, a, n_streams, bt, s);
    else *result = launch_walk(schedule_small_kernel<kWalk, 64, false>, a, n_streams, bt, s);
  } else if (bt == 64u) {
    *result = launch_walk(schedule_model_kernel<kWalk, 64>, a, n_streams, bt, s);
  } else if (bt == 128u) {
    *result = launch_walk(schedule_model_kernel<kWalk, 128>, a, n_streams, bt, s);
  } else if (bt == 256u) {
    *result = launch_walk(schedule_model_kernel<kWalk, 256>, a, n_streams, bt, s);
  } else {
    *result = launch_walk(schedule_model_kernel<kWalk, 512>, a, n_streams, bt, s);
  }
  return true;
}

}  // namespace

bool launch_model_inflight(const TopoArgs& t, uint32_t n_streams, const netkv_weights* d_w,
                           uint32_t R, const uint32_t* d_len, const uint32_t* d_prefill,
                           const uint32_t* d_snap, const int64_t* d_arrival_us,
                           const uint16_t* d_M, const float* d_UB, uint32_t n_snap,
                           const uint32_t* d_events, const uint64_t* d_event_off,
                           uint32_t inflight_cap, uint32_t heap_cap, const int64_t* d_load_init,
                           int32_t* d_dec, float* d_best, float* d_second, int32_t* d_xfer_us,
                           int64_t* d_load_final, int* d_status, cudaStream_t s,
                           netkv_status* result) {
  ModelArgs a = {};
  a.t = t;
  a.W = d_w;
  a.R = R;
  a.n_snap = n_snap;
  a.len = d_len;
  a.prefill = d_prefill;
  a.snap = d_snap;
  a.M = d_M;
  a.UB = d_UB;
  a.events = d_events;
  a.event_off = d_event_off;
  a.state_init = d_load_init;
  a.dec = d_dec;
  a.best = d_best;
  a.second = d_second;
  a.state_final = d_load_final;
  a.status = d_status;
  a.arrival_us = d_arrival_us;
  a.inflight_cap = inflight_cap;
  a.heap_cap = heap_cap;
  a.xfer_us = d_xfer_us;
  return launch_model<kContend>(a, n_streams, s, result);
}

bool launch_model_load(const TopoArgs& t, uint32_t n_streams, const netkv_weights* d_w,
                       float t_a, float t_b, int32_t beta_max, int64_t m_min, int64_t m0,
                       uint32_t R, const uint32_t* d_len, const uint32_t* d_prefill,
                       const uint32_t* d_snap, const uint16_t* d_M, const float* d_UB,
                       uint32_t n_snap, const uint32_t* d_events, const uint64_t* d_event_off,
                       const int64_t* d_m_init, const int32_t* d_n_init, int32_t* d_dec,
                       float* d_best, float* d_second, int64_t* d_m_final, int32_t* d_n_final,
                       int* d_status, cudaStream_t s, netkv_status* result) {
  ModelArgs a = {};
  a.t = t;
  a.W = d_w;
  a.R = R;
  a.n_snap = n_snap;
  a.len = d_len;
  a.prefill = d_prefill;
  a.snap = d_snap;
  a.M = d_M;
  a.UB = d_UB;
  a.events = d_events;
  a.event_off = d_event_off;
  a.state_init = d_m_init;
  a.dec = d_dec;
  a.best = d_best;
  a.second = d_second;
  a.state_final = d_m_final;
  a.status = d_status;
  a.lm = LoadModel{t_a, t_b, beta_max, m_min, m0};
  a.held_init = d_n_init;
  a.held_final = d_n_final;
  return launch_model<kModel>(a, n_streams, s, result);
}

bool launch_model_plain(const TopoArgs& t, uint32_t n_streams, const netkv_weights* d_w,
                        uint32_t R, const uint32_t* d_len, const uint32_t* d_prefill,
                        const uint32_t* d_snap, uint32_t n_snap, const uint32_t* d_events,
                        const uint64_t* d_event_off, const int64_t* d_load_init, int32_t* d_dec,
                        float* d_best, float* d_second, int64_t* d_load_final,
                        const float* d_base, int* d_status, cudaStream_t s,
                        netkv_status* result) {
  ModelArgs a = {};
  a.t = t;
  a.W = d_w;
  a.R = R;
  a.n_snap = n_snap;
  a.len = d_len;
  a.prefill = d_prefill;
  a.snap = d_snap;
  a.base = d_base;
  a.events = d_events;
  a.event_off = d_event_off;
  a.state_init = d_load_init;
  a.dec = d_dec;
  a.best = d_best;
  a.second = d_second;
  a.state_final = d_load_final;
  a.status = d_status;
  return launch_model<kPlain>(a, n_streams, s, result);
}
