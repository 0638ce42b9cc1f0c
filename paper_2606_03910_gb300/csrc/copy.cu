// Bulk copies by SM loads and stores, for moving a step's inputs from pinned host memory
// to the device (and results back).  On a Grace-Blackwell node a kernel reading pinned
// host memory through unified addressing streams it over NVLink-C2C about twice as fast
// as the copy engines; the same kernel also copies device to device.
//
// A group of copies is one launch: the buffers are cut into chunks of 512 * U units of 16
// bytes, numbered one buffer after another, and the blocks stride over the chunks.  A small
// copy is bound by its launch and one round trip over the link (6.8 us each), which a group
// pays once: the ten inputs and four results of a step of 32 replicas took 95 us, now 72.
// Large groups are bound by the link; U = 4 loads a thread in flight where every resident
// block still gets several chunks, else 1, so that small groups use more SMs.
#include "netkv_internal.cuh"

namespace {

constexpr uint32_t kCopyThreads = 512;
constexpr uint32_t kCopyMax = 32;  // buffers of one launch

struct CopyGroup {
  uint32_t n;
  uint32_t first[kCopyMax + 1];  // each buffer's first chunk; the number of chunks
  const unsigned char* src[kCopyMax];
  unsigned char* dst[kCopyMax];
  uint64_t bytes[kCopyMax];
};

template <int U>
__global__ void __launch_bounds__(kCopyThreads) copy_kernel(const __grid_constant__ CopyGroup g) {
  constexpr uint64_t kChunk = (uint64_t)kCopyThreads * U;  // 16-byte units
  for (uint32_t chunk = blockIdx.x; chunk < g.first[g.n]; chunk += gridDim.x) {
    uint32_t c = 0;
    while (chunk >= g.first[c + 1]) ++c;  // ends at the latest with the last buffer
    const uint64_t n16 = g.bytes[c] / 16, tail = g.bytes[c] % 16;
    const uint4* src = reinterpret_cast<const uint4*>(g.src[c]);
    uint4* dst = reinterpret_cast<uint4*>(g.dst[c]);
    const uint64_t i0 = (uint64_t)(chunk - g.first[c]) * kChunk + threadIdx.x;
    uint4 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (i0 + u * kCopyThreads < n16) v[u] = __ldcs(src + i0 + u * kCopyThreads);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (i0 + u * kCopyThreads < n16) dst[i0 + u * kCopyThreads] = v[u];
    if (chunk == g.first[c] && threadIdx.x < tail)
      g.dst[c][n16 * 16 + threadIdx.x] = g.src[c][n16 * 16 + threadIdx.x];
  }
}

}  // namespace

extern "C" netkv_status netkv_copy_group_async(const netkv_copy* copies, uint32_t n,
                                               netkv_stream_t stream) {
  if (n == 0) return NETKV_OK;
  if (!copies) return NETKV_EINVAL;
  for (uint32_t i = 0; i < n; ++i)
    if (copies[i].bytes && (!copies[i].dst || !copies[i].src || !aligned_to(copies[i].dst, 16) ||
                            !aligned_to(copies[i].src, 16) || copies[i].bytes >> 40))
      return NETKV_EINVAL;
  int dev = 0, sms = 0;
  NETKV_CUDA_TRY(cudaGetDevice(&dev));
  NETKV_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  for (uint32_t i = 0; i < n;) {
    CopyGroup g;
    g.n = 0;
    uint64_t units = 0;
    for (; i < n && g.n < kCopyMax; ++i) {
      if (copies[i].bytes == 0) continue;
      g.src[g.n] = reinterpret_cast<const unsigned char*>(copies[i].src);
      g.dst[g.n] = reinterpret_cast<unsigned char*>(copies[i].dst);
      g.bytes[g.n++] = copies[i].bytes;
      units += (copies[i].bytes + 15) / 16;
    }
    if (g.n == 0) break;
    const uint64_t resident = (uint64_t)sms * 4;
    const bool deep = units > resident * 4 * kCopyThreads * 4;
    const uint64_t chunk = (uint64_t)kCopyThreads * (deep ? 4 : 1);
    g.first[0] = 0;
    for (uint32_t c = 0; c < g.n; ++c)
      g.first[c + 1] = g.first[c] + (uint32_t)(((g.bytes[c] + 15) / 16 + chunk - 1) / chunk);
    const unsigned grid = (unsigned)(g.first[g.n] < resident ? g.first[g.n] : resident);
    if (deep) copy_kernel<4><<<grid, kCopyThreads, 0, (cudaStream_t)stream>>>(g);
    else copy_kernel<1><<<grid, kCopyThreads, 0, (cudaStream_t)stream>>>(g);
    if (netkv_launch_status() != NETKV_OK) return NETKV_ECUDA;
  }
  return NETKV_OK;
}

extern "C" netkv_status netkv_copy_async(void* dst, const void* src, size_t bytes,
                                         netkv_stream_t stream) {
  const netkv_copy one = {dst, src, bytes};
  return netkv_copy_group_async(&one, 1, stream);
}
