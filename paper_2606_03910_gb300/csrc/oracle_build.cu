// Network cost oracle (Sec. III-D Eq. 3 and Eq. 4, Sec. III-E) with per-link congestion.
//
// level_bottleneck_kernel: UB[s][i][k] = min_{h<=k} B_h (1 - u[s][link_h(i)]), one
//   thread per (snapshot, instance), one 16-byte store each.  With directed links
//   (kDir) a prefill instance's climb reads the upward row and a decode instance's the
//   downward row: the directions a transfer from prefill to decode crosses them in.
// oracle_build_kernel: C[s][p][d] = kv / min(UB[s][p][tau], UB[s][d][tau]) + L_tau.
//   In the paper-literal per-tier mode (kTier) UB[s][i][k] = B_k (1 - c[s][k]) for every
//   instance, from four congestion values per snapshot.
//   Division is monotone (correctly rounded, positive operands), so
//   kv / min(a, b) == max(kv / a, kv / b) exactly; each block therefore divides once per
//   (instance, level) it touches and the per-pair work is a tier test, a max and an
//   add.  No scratch memory: the quotients of the block's instances are recomputed from
//   the utilisation row.  When the call also asks for UB, the blocks that hold an
//   instance's bottlenecks first write them, so both outputs take one launch.
#include "netkv_internal.cuh"

namespace {

constexpr int kBlock = 256;
constexpr int kPerThread = 4;
constexpr uint32_t kPTile = 256;  // prefill ranks staged at a time, one a thread
// Pairs of a call from which the deep form runs: four rows a thread in flight at 3 blocks an SM
// instead of two at 4.  Snapshots of 2,048 x 8,192 (us, two rows / four): 1 20.8 / 24.5, 8
// 96.2 / 97.8, 16 173 / 168, 32 324 / 310, 1,000 9,232 / 9,167.
constexpr uint64_t kDeepPairs = 1ull << 28;

__device__ __forceinline__ bool util_ok(float u) { return u >= 0.0f && u < 1.0f; }

// Level bottlenecks of instance `links` in one utilisation row.
__device__ __forceinline__ float4 level_bottlenecks(const TopoArgs& t, const float* __restrict__ row,
                                                    const uint4& l, int* status) {
  const float u0 = __ldg(row + l.x), u1 = __ldg(row + l.y);
  const float u2 = __ldg(row + l.z), u3 = __ldg(row + l.w);
  if (!(util_ok(u0) && util_ok(u1) && util_ok(u2) && util_ok(u3)))
    flag_status(status, NETKV_DEV_EDOMAIN);
  float4 b;
  b.x = t.bw[0] * (1.0f - u0);
  b.y = fminf(b.x, t.bw[1] * (1.0f - u1));
  b.z = fminf(b.y, t.bw[2] * (1.0f - u2));
  b.w = fminf(b.z, t.bw[3] * (1.0f - u3));
  return b;
}

// Paper-literal per-tier maps (Sec. III-E): level k's bandwidth B_k (1 - c_k) from the
// snapshot's four per-tier congestion values, with no minimum over lower levels.
__device__ __forceinline__ float4 tier_bandwidths(const TopoArgs& t, const float* __restrict__ c,
                                                  int* status) {
  const float c0 = __ldg(c), c1 = __ldg(c + 1), c2 = __ldg(c + 2), c3 = __ldg(c + 3);
  if (!(util_ok(c0) && util_ok(c1) && util_ok(c2) && util_ok(c3)))
    flag_status(status, NETKV_DEV_EDOMAIN);
  return make_float4(t.bw[0] * (1.0f - c0), t.bw[1] * (1.0f - c1), t.bw[2] * (1.0f - c2),
                     t.bw[3] * (1.0f - c3));
}

__device__ __forceinline__ float4 quotients(float kv, const float4& b) {
  return make_float4(kv / b.x, kv / b.y, kv / b.z, kv / b.w);
}

template <bool kDir, bool kTier = false>
__global__ void __launch_bounds__(kBlock) level_bottleneck_kernel(
    TopoArgs t, const float* __restrict__ util, const float* __restrict__ util_down,
    uint32_t n_snap, float4* __restrict__ UB, int* status) {
  const uint64_t total = (uint64_t)n_snap * t.N;
  for (uint64_t idx = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t s = idx / t.N;
    const uint32_t i = (uint32_t)(idx - s * t.N);
    const uint4 l = __ldg(t.links + i);
    const float* rows = (kDir && __ldg(t.role + i)) ? util_down : util;
    UB[idx] = kTier ? tier_bandwidths(t, util + s * 4, status)
                    : level_bottlenecks(t, rows + s * t.n_links, l, status);
  }
}

// A block takes one snapshot, the prefill ranks [y * p_span, (y + 1) * p_span) and
// 4 * tx decode ranks: tx = 2^log2_tx thread columns own four decodes each, kept in
// registers, and the 256 / tx thread rows walk the staged prefill ranks side by side, so
// that small pools fill a block too.  Bound by the writes of C: a warp stores 512
// contiguous bytes of a row (kVec), or four times 128 where rows are not 16-byte
// aligned, with an evict-first hint.  Instances are numbered pod by pod, so a prefill
// whose pod lies outside the pods of the thread's decodes is of tier 3 with all of them:
// that test replaces four tier tests and the selections by tier for all but the few
// pairs that share a pod (issue slots: about 20 instructions per four pairs, not 80).
// util_down: the decode side's rows (the downward utilisations of directed links; the
// same pointer as util for undirected links).
template <bool kVec, bool kTier, bool kDeep>
__global__ void __launch_bounds__(kBlock, kDeep ? 3 : 4) oracle_build_kernel(
    TopoArgs t, const float* __restrict__ util, const float* __restrict__ util_down,
    uint32_t n_snap, float kv, float* __restrict__ C, float4* __restrict__ UB, uint32_t p_span,
    uint32_t log2_tx, int* status) {
  __shared__ float4 s_q[kPTile];
  __shared__ uint4 s_l[kPTile];
  __shared__ float2 s_far[kPTile];  // tier-3 quotient and pod link
  const float4 lat = make_float4(t.lat[0], t.lat[1], t.lat[2], t.lat[3]);
  const uint32_t tx = 1u << log2_tx, ty = kBlock >> log2_tx;
  const uint32_t col = threadIdx.x & (tx - 1), row = threadIdx.x >> log2_tx;
  // decode of slot j: d0 + j * dstep
  const uint32_t dstep = kVec ? 1u : min(tx, 32u);
  const uint32_t d0 = blockIdx.x * (kPerThread * tx) +
                      (kVec ? col * kPerThread
                            : col / dstep * (kPerThread * dstep) + col % dstep);
  const uint32_t p_beg = blockIdx.y * p_span, p_end = min(t.P, p_beg + p_span);

  for (uint32_t s = blockIdx.z; s < n_snap; s += gridDim.z) {
    const float* row_u = util + (uint64_t)s * (kTier ? 4u : t.n_links);
    const float* row_d = util_down + (uint64_t)s * (kTier ? 4u : t.n_links);
    uint4 ld[kPerThread];
    float4 qd[kPerThread];
    uint32_t pod_lo = 0xffffffffu, pod_hi = 0u;
#pragma unroll
    for (int j = 0; j < kPerThread; ++j) {
      const uint32_t d = d0 + j * dstep;
      ld[j] = make_uint4(0, 0, 0, 0);
      qd[j] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (d < t.D) {
        const uint32_t inst = __ldg(t.dec + d);
        ld[j] = __ldg(t.links + inst);
        const float4 b = kTier ? tier_bandwidths(t, row_u, status)
                               : level_bottlenecks(t, row_d, ld[j], status);
        if (UB && blockIdx.y == 0 && row == 0) UB[(uint64_t)s * t.N + inst] = b;
        qd[j] = quotients(kv, b);
        pod_lo = min(pod_lo, ld[j].w);
        pod_hi = max(pod_hi, ld[j].w);
      }
    }
    float* crow = C + (uint64_t)s * t.P * t.D;
    for (uint32_t p0 = p_beg; p0 < p_end; p0 += kPTile) {
      const uint32_t np = min(kPTile, p_end - p0);
      __syncthreads();
      if (threadIdx.x < np) {
        const uint32_t inst = __ldg(t.pre + p0 + threadIdx.x);
        const uint4 l = __ldg(t.links + inst);
        const float4 b = kTier ? tier_bandwidths(t, row_u, status)
                               : level_bottlenecks(t, row_u, l, status);
        if (UB && blockIdx.x == 0) UB[(uint64_t)s * t.N + inst] = b;
        const float4 q = quotients(kv, b);
        s_l[threadIdx.x] = l;
        s_q[threadIdx.x] = q;
        s_far[threadIdx.x] = make_float2(q.w, __uint_as_float(l.w));
      }
      __syncthreads();
      if (d0 >= t.D) continue;
#pragma unroll kDeep ? 4 : 2
      for (uint32_t k = row; k < np; k += ty) {
        const float2 far = s_far[k];
        const uint32_t pod = __float_as_uint(far.y);
        float c[kPerThread];
        if (pod < pod_lo || pod > pod_hi) {
#pragma unroll
          for (int j = 0; j < kPerThread; ++j) c[j] = fmaxf(far.x, qd[j].w) + lat.w;
        } else {
          const float4 qp = s_q[k];
          const uint4 lp = s_l[k];
#pragma unroll
          for (int j = 0; j < kPerThread; ++j) {
            const int tau = tier_of(lp, ld[j]);
            c[j] = fmaxf(pick4(qp, tau), pick4(qd[j], tau)) + pick4(lat, tau);
          }
        }
        float* out = crow + (uint64_t)(p0 + k) * t.D + d0;
        if (kVec) {
          __stcs(reinterpret_cast<float4*>(out), make_float4(c[0], c[1], c[2], c[3]));
        } else {
#pragma unroll
          for (int j = 0; j < kPerThread; ++j)
            if (d0 + j * dstep < t.D) __stcs(out + j * dstep, c[j]);
        }
      }
    }
  }
}

}  // namespace

enum OracleMode { kLinks = 0, kDirected = 1, kTiers = 2 };

static netkv_status oracle_build(netkv_topology_t topo, const float* d_util, const float* d_util_down,
                          int mode, uint32_t n_snap, double kv_bytes, float* d_C,
                          float* d_UB, int* d_status, netkv_stream_t stream) {
  if (!topo || !d_util || !d_util_down || (!d_C && !d_UB)) return NETKV_EINVAL;
  if (!(kv_bytes > 0) || !(kv_bytes < 3.0e38)) return NETKV_EINVAL;
  if (!aligned_to(d_util, 4) || !aligned_to(d_util_down, 4) || (d_C && !aligned_to(d_C, 4)) ||
      (d_UB && !aligned_to(d_UB, 16)))
    return NETKV_EINVAL;
  if (n_snap == 0) return NETKV_OK;
  const TopoArgs t = topo_args(topo);
  cudaStream_t s = (cudaStream_t)stream;
  if (!d_C) {
    const uint64_t total = (uint64_t)n_snap * t.N;
    const uint64_t blocks = (total + kBlock - 1) / kBlock;
    const unsigned grid = (unsigned)(blocks < (1u << 20) ? blocks : (1u << 20));
    if (mode == kTiers)
      level_bottleneck_kernel<false, true><<<grid, kBlock, 0, s>>>(
          t, d_util, d_util, n_snap, reinterpret_cast<float4*>(d_UB), d_status);
    else if (mode == kDirected)
      level_bottleneck_kernel<true><<<grid, kBlock, 0, s>>>(
          t, d_util, d_util_down, n_snap, reinterpret_cast<float4*>(d_UB), d_status);
    else
      level_bottleneck_kernel<false><<<grid, kBlock, 0, s>>>(
          t, d_util, d_util, n_snap, reinterpret_cast<float4*>(d_UB), d_status);
    return netkv_launch_status();
  }
  // Thread columns to cover D four decodes a thread, at most 256; then the prefill ranks are
  // split until the card has kBlocksPerSm blocks an SM.  A block's set-up (16 gathers
  // and divisions a thread) is worth at least kMinRows prefill ranks per thread row.
  // 2,048 x 8,192 pairs with UB (kernel time): one snapshot 20.8 us (491 us as 8 blocks of all
  // prefill ranks); 32 snapshots, in the two-row form, 324 us (528 us as 256 blocks; 387 us with
  // 4 blocks an SM wanted), in the deep form that they take 310 us = 6.9 TB/s of writes.
  constexpr uint32_t kBlocksPerSm = 16, kMinRows = 16;
  uint32_t log2_tx = 0;
  while (log2_tx < 8 && (uint32_t)kPerThread << log2_tx < t.D) ++log2_tx;
  const uint32_t gx = (t.D + (kPerThread << log2_tx) - 1) / (kPerThread << log2_tx);
  const uint32_t gz = n_snap < 65535u ? n_snap : 65535u;
  int dev = 0, sms = 0;
  NETKV_CUDA_TRY(cudaGetDevice(&dev));
  NETKV_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const uint64_t have = (uint64_t)gx * gz, want = (uint64_t)sms * kBlocksPerSm;
  const uint32_t rows = kMinRows * (kBlock >> log2_tx);
  const uint32_t most = (t.P + rows - 1) / rows;
  const uint64_t need = (want + have - 1) / have;
  uint32_t gy = need < most ? (uint32_t)need : most;
  if (gy > 65535u) gy = 65535u;
  const uint32_t p_span = (t.P + gy - 1) / gy;
  const dim3 grid(gx, (t.P + p_span - 1) / p_span, gz);
  const bool vec = (t.D % 4 == 0) && aligned_to(d_C, 16);
  const float* down = mode == kDirected ? d_util_down : d_util;
  float4* ub = reinterpret_cast<float4*>(d_UB);
  const bool deep = (uint64_t)n_snap * t.P * t.D >= kDeepPairs;
#define NETKV_BUILD(VEC, TIER)                                                             \
  if (deep)                                                                                \
    oracle_build_kernel<VEC, TIER, true><<<grid, kBlock, 0, s>>>(                          \
        t, d_util, down, n_snap, (float)kv_bytes, d_C, ub, p_span, log2_tx, d_status);     \
  else                                                                                     \
    oracle_build_kernel<VEC, TIER, false><<<grid, kBlock, 0, s>>>(                         \
        t, d_util, down, n_snap, (float)kv_bytes, d_C, ub, p_span, log2_tx, d_status)
  if (mode == kTiers) {
    if (vec) { NETKV_BUILD(true, true); }
    else { NETKV_BUILD(false, true); }
  } else {
    if (vec) { NETKV_BUILD(true, false); }
    else { NETKV_BUILD(false, false); }
  }
#undef NETKV_BUILD
  return netkv_launch_status();
}

extern "C" netkv_status netkv_oracle_build(netkv_topology_t topo, const float* d_util,
                                           uint32_t n_snap, double kv_bytes, float* d_C,
                                           float* d_UB, int* d_status, netkv_stream_t stream) {
  return oracle_build(topo, d_util, d_util, kLinks, n_snap, kv_bytes, d_C, d_UB, d_status, stream);
}

extern "C" netkv_status netkv_oracle_build_directed(netkv_topology_t topo, const float* d_util_up,
                                                    const float* d_util_down, uint32_t n_snap,
                                                    double kv_bytes, float* d_C, float* d_UB,
                                                    int* d_status, netkv_stream_t stream) {
  return oracle_build(topo, d_util_up, d_util_down, kDirected, n_snap, kv_bytes, d_C, d_UB,
                      d_status, stream);
}

extern "C" netkv_status netkv_oracle_build_tiers(netkv_topology_t topo, const float* d_c,
                                                 uint32_t n_snap, double kv_bytes, float* d_C,
                                                 float* d_UB, int* d_status,
                                                 netkv_stream_t stream) {
  return oracle_build(topo, d_c, d_c, kTiers, n_snap, kv_bytes, d_C, d_UB, d_status, stream);
}
