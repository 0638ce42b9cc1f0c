// Scores, score keys and the state of the greedy's variants, shared by the greedy kernels.
#pragma once

#include "netkv_internal.cuh"

// Decision-independent part of a candidate's score (Algorithm 1 lines 5-8, Eq. 2, Eq. 3):
// w_net * (s_eff / min(UB_p[tau], UB_d[tau]) + L_tau) + w_prefix * (l - 16 M) / l.
__device__ __forceinline__ float base_score(const netkv_weights& w, uint32_t l, uint32_t m,
                                            float ub_p, float ub_d, float lat_tau, int* status) {
  uint32_t lam = 16u * m;
  if (m > l / 16u) {
    flag_status(status, NETKV_DEV_EDOMAIN);
    lam = lam < l ? lam : l;
  }
  const uint32_t miss_tok = l - lam;
  const float bb = fminf(ub_p, ub_d);
  const float s_eff = (float)((int64_t)miss_tok * (int64_t)w.bytes_per_token);
  const float T = s_eff / bb + lat_tau;
  const float miss = (float)miss_tok / (float)l;
  return w.w_net * T + w.w_prefix * miss;
}

// Level bottlenecks of an instance with links `l` in one utilisation row:
// (B_0 (1-u_0), min with B_1 (1-u_1), ...), the same fp32 expression as the oracle build's
// level-bottleneck pass, so a score computed from the row equals one computed from UB.
__device__ __forceinline__ float4 level_bottlenecks_of(const TopoArgs& t,
                                                       const float* __restrict__ row,
                                                       const uint4& l, int* status) {
  const float u0 = __ldg(row + l.x), u1 = __ldg(row + l.y);
  const float u2 = __ldg(row + l.z), u3 = __ldg(row + l.w);
  if (!(u0 >= 0.0f && u0 < 1.0f && u1 >= 0.0f && u1 < 1.0f && u2 >= 0.0f && u2 < 1.0f &&
        u3 >= 0.0f && u3 < 1.0f))
    flag_status(status, NETKV_DEV_EDOMAIN);
  float4 b;
  b.x = t.bw[0] * (1.0f - u0);
  b.y = fminf(b.x, t.bw[1] * (1.0f - u1));
  b.z = fminf(b.y, t.bw[2] * (1.0f - u2));
  b.w = fminf(b.z, t.bw[3] * (1.0f - u3));
  return b;
}

namespace {

constexpr uint32_t kNone = 0xffffffffu;

// Order-preserving 32-bit keys of fp32 scores, so that warp-wide redux minima give the
// (score, rank) argmin; kNoKey (above every float's key) stands for "no candidate".
constexpr uint32_t kNoKey = 0xffffffffu;
__device__ __forceinline__ uint32_t score_key(float x) {
  const uint32_t u = __float_as_uint(__fadd_rn(x, 0.0f));  // -0 and +0 tie, as compared
  return u ^ ((uint32_t)((int32_t)u >> 31) | 0x80000000u);
}
__device__ __forceinline__ float key_score(uint32_t k) {
  if (k == kNoKey) return __int_as_float(0x7f800000);
  return __uint_as_float(k ^ ((k >> 31) ? 0x80000000u : 0xffffffffu));
}
// Block-free argmin over the 32 lanes of a warp: (best key, its lowest rank, second key),
// where a lane offers (key, rank, key of its own runner-up).
__device__ __forceinline__ void warp_argmin_keys(uint32_t& key, uint32_t& rank, uint32_t& key2) {
  const uint32_t bk = __reduce_min_sync(0xffffffffu, key);
  const uint32_t br = __reduce_min_sync(0xffffffffu, key == bk ? rank : kNone);
  // the winning lane offers its runner-up; every other lane its best
  const uint32_t sk = __reduce_min_sync(0xffffffffu, (key == bk && rank == br) ? key2 : key);
  key = bk;
  rank = br;
  key2 = sk;
}

// Tokens that still fit a decode, at most 2^32 - 1: load + l <= cap iff l <= headroom (l >= 1).
// The unsigned difference is exact where cap > load, also where the signed one overflows.
__device__ __forceinline__ uint32_t headroom(int64_t cap, int64_t load) {
  const uint64_t h = (uint64_t)cap - (uint64_t)load;
  return cap <= load ? 0u : h >= 0xffffffffull ? 0xffffffffu : (uint32_t)h;
}

// The paper's compute-load model (Sec. III-C, IV-B) as kernel parameters.
struct LoadModel {
  float t_a, t_b;      // t_iter(beta) = t_a + t_b * beta
  int32_t beta_max;
  int64_t m_min, m0;
};

// w_load's factor for a decode that holds `held` requests: T_queue + T_decode (Sec. IV-B).
__device__ __forceinline__ float load_term(const LoadModel& lm, int32_t held) {
  const int32_t beta = min(held, lm.beta_max);
  const int32_t blocked = (held - beta) - (lm.beta_max - beta);
  const float t_queue = (blocked > 0 ? (float)blocked : 0.0f) * (lm.t_a + lm.t_b * (float)beta);
  const float t_decode = lm.t_a + lm.t_b * (float)(beta + 1);
  return t_queue + t_decode;
}

// Self-contention (Eq. 4's n_inflight, Algorithm 1 lines 5 and 14, Sec. V-C): the parts of
// a candidate's score that do not depend on the counters ...
struct XferParts {
  float s_eff, bb, miss;  // bytes to move, Bbot, missed fraction
};
__device__ __forceinline__ XferParts xfer_parts(const netkv_weights& w, uint32_t l, uint32_t m,
                                                float ub_p, float ub_d, int* status) {
  uint32_t lam = 16u * m;
  if (m > l / 16u) {
    flag_status(status, NETKV_DEV_EDOMAIN);
    lam = lam < l ? lam : l;
  }
  const uint32_t miss_tok = l - lam;
  XferParts x;
  x.bb = fminf(ub_p, ub_d);
  x.s_eff = (float)((int64_t)miss_tok * (int64_t)w.bytes_per_token);
  x.miss = (float)miss_tok / (float)l;
  return x;
}
// ... its transfer time, the bandwidth being divided by 1 + n ...
__device__ __forceinline__ float xfer_time(const XferParts& x, uint32_t n, float lat_tau) {
  const float b_eff = n ? x.bb / (float)(1u + n) : x.bb;
  return x.s_eff / b_eff + lat_tau;
}
// ... and its network and prefix terms; T is returned for the completion time.
__device__ __forceinline__ float contended_score(const netkv_weights& w, uint32_t l, uint32_t m,
                                                 float ub_p, float ub_d, float lat_tau,
                                                 uint32_t n, float& T, int* status) {
  const XferParts x = xfer_parts(w, l, m, ub_p, ub_d, status);
  T = xfer_time(x, n, lat_tau);
  return w.w_net * T + w.w_prefix * x.miss;
}

// Pending transfer completions of one stream: a binary min-heap in shared memory kept by
// the stream's lead thread, keys (completion time in us << 16) | (prefill rank << 2) | tier.
struct DoneHeap {
  unsigned long long* a;
  uint32_t n, cap;
  __device__ bool push(unsigned long long k) {
    if (n == cap) return false;
    uint32_t i = n++;
    while (i > 0) {
      const uint32_t p = (i - 1) >> 1;
      if (a[p] <= k) break;
      a[i] = a[p];
      i = p;
    }
    a[i] = k;
    return true;
  }
  __device__ void pop() {
    const unsigned long long k = a[--n];
    if (n == 0) return;
    uint32_t i = 0;
    for (;;) {
      uint32_t c = 2 * i + 1;
      if (c >= n) break;
      if (c + 1 < n && a[c + 1] < a[c]) ++c;
      if (a[c] >= k) break;
      a[i] = a[c];
      i = c;
    }
    a[i] = k;
  }
};

}  // namespace

// The walks with producers (schedule_model.cu); false when the pool or its tables do not fit, or
// another walk serves so many streams faster: nothing is launched.
bool launch_model_plain(const TopoArgs& t, uint32_t n_streams, const netkv_weights* d_w,
                        uint32_t R, const uint32_t* d_len, const uint32_t* d_prefill,
                        const uint32_t* d_snap, uint32_t n_snap, const uint32_t* d_events,
                        const uint64_t* d_event_off, const int64_t* d_load_init, int32_t* d_dec,
                        float* d_best, float* d_second, int64_t* d_load_final,
                        const float* d_base, int* d_status, cudaStream_t s,
                        netkv_status* result);
bool launch_model_inflight(const TopoArgs& t, uint32_t n_streams, const netkv_weights* d_w,
                           uint32_t R, const uint32_t* d_len, const uint32_t* d_prefill,
                           const uint32_t* d_snap, const int64_t* d_arrival_us,
                           const uint16_t* d_M, const float* d_UB, uint32_t n_snap,
                           const uint32_t* d_events, const uint64_t* d_event_off,
                           uint32_t inflight_cap, uint32_t heap_cap, const int64_t* d_load_init,
                           int32_t* d_dec, float* d_best, float* d_second, int32_t* d_xfer_us,
                           int64_t* d_load_final, int* d_status, cudaStream_t s,
                           netkv_status* result);
bool launch_model_load(const TopoArgs& t, uint32_t n_streams, const netkv_weights* d_w,
                       float t_a, float t_b, int32_t beta_max, int64_t m_min, int64_t m0,
                       uint32_t R, const uint32_t* d_len, const uint32_t* d_prefill,
                       const uint32_t* d_snap, const uint16_t* d_M, const float* d_UB,
                       uint32_t n_snap, const uint32_t* d_events, const uint64_t* d_event_off,
                       const int64_t* d_m_init, const int32_t* d_n_init, int32_t* d_dec,
                       float* d_best, float* d_second, int64_t* d_m_final, int32_t* d_n_final,
                       int* d_status, cudaStream_t s, netkv_status* result);
