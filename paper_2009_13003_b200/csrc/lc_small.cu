// Small vectors: the whole compress pass (Algorithm 1 steps 4-6, optionally step 7) in one launch and without a
// workspace: one CTA for a vector of one chunk, one cluster of CTAs for a vector of up to 32.
//
// For such a vector the four kernels of the general path are all launch latency; layers of
// a few hundred elements are common in per-layer use, and so are whole models of some ten thousand. Bound: latency, so every
// part of the pass is spread over all 16 warps. A thread loads its eight elements of a chunk once and keeps base and delta in
// registers through statistics, coding and the tracked state. Warp w takes the chunk's steps 2w and 2w + 1, so the codes
// of a thread are one contiguous piece of its lane's sub-stream: a scan over warps and lanes of the pieces' bit counts
// places them, and each thread ORs its piece into the chunk's image in shared memory, which leaves with 16-byte stores.
// In a cluster, the CTAs add their statistics to each other's in shared memory and read each other's chunk sizes there, each derives the same table, and
// hardware barriers take the place of kernel boundaries and of the encode pass's look-back. Same bytes as the general
// path. GPU time of a call: about 8 us at 1000 elements (18 us with one warp coding alone and the earlier table pass), 12.8 us at 61,706 (25.5 us in the general
// path; 14.8 us with the CTAs reading each other's statistics of the keys that occur, 26.9 of all 512).
#include "lc_small.cuh"

namespace lc {
namespace {

using namespace small;

constexpr uint32_t kMaxCluster = 16;

template <int M, bool CLUSTER>
__global__ void __launch_bounds__(kTableThreads)
small_compress_kernel(Control* ctl, const float* base, const float* cur, uint32_t n, int nbits, uint8_t* stream,
                      float* tracked_out, int keep_status) {
  extern __shared__ __align__(16) unsigned char s_small[];
  SmallShared<M>& S = *reinterpret_cast<SmallShared<M>*>(s_small);
  begin_next();
  const uint32_t tid = threadIdx.x;
  const bool first = !CLUSTER || cluster_rank() == 0;
  const int earlier = keep_status ? ctl->status : 0;  // the same for every thread: nothing here has written it yet
  if (earlier) {
    if (first) clear_header(stream);
    return;
  }
  const int err = small_vector<M, CLUSTER>(S, base, cur, n, nbits, stream, tracked_out, ctl);
  if (!first) return;
  if (err) clear_header(stream);
  if (tid == 0) {
    // what the general path clears and its table pass writes, as far as later readers look at it
    ctl->status = err;  // barriers (of the cluster) lie between the reads above and this
    ctl->ticket = 0;
    ctl->nsym = err ? 0 : S.T.nsym;
    ctl->wide = err ? 0 : S.T.wide;
    ctl->max_len = err ? 0 : S.T.max_len;
    ctl->payload_bits = err ? 0 : S.T.payload_bits;
  }
}

template <int M, bool CLUSTER>
cudaError_t launch_small(uint32_t ctas, Control* ctl, const float* base, const float* cur, uint32_t n, int nbits, uint8_t* stream,
                         float* tracked_out, bool keep_status, cudaStream_t cs) {
  static int state[kMaxDevices] = {};  // by device ordinal: 0 not looked at yet, 1 ready, 2 no room for such a cluster
  const int dev = current_device_index();
  if (dev < 0) return cudaErrorInvalidDevice;
  const auto kernel = small_compress_kernel<M, CLUSTER>;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kTableThreads);
  cfg.dynamicSmemBytes = sizeof(SmallShared<M>);
  cfg.stream = cs;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (state[dev] == 0) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallShared<M>));
    int fit = 1;
    if (e == cudaSuccess && CLUSTER) {
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      at[0].val.clusterDim = {kMaxCluster, 1, 1};
      cfg.gridDim = dim3(kMaxCluster);
      if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&fit, kernel, &cfg);
    }
    if (e != cudaSuccess) return e;
    state[dev] = fit > 0 ? 1 : 2;
  }
  if (state[dev] == 2) return cudaErrorNotSupported;
  if (!CLUSTER) {
    kernel<<<1, kTableThreads, sizeof(SmallShared<M>), cs>>>(ctl, base, cur, n, nbits, stream, tracked_out, keep_status ? 1 : 0);
    return cudaGetLastError();
  }
  cfg.gridDim = dim3(ctas);
  at[0].val.clusterDim = {ctas, 1, 1};
  return cudaLaunchKernelEx(&cfg, kernel, ctl, base, cur, n, nbits, stream, tracked_out, keep_status ? 1 : 0);
}

}  // namespace

cudaError_t launch_small_compress(Control* ctl, const float* base, const float* cur, uint64_t n, int nbits,
                                  uint8_t* stream, float* tracked_out, bool keep_status, cudaStream_t cs) {
  if (n == 0 || n > kSmallMaxElems) return cudaErrorInvalidValue;
  const uint32_t m = (uint32_t)n, chunks = (m + kChunkElems - 1) / kChunkElems;
  if (chunks == 1) return launch_small<1, false>(1, ctl, base, cur, m, nbits, stream, tracked_out, keep_status, cs);
  uint32_t ctas = 2;  // a power of two, so that every size is one the hardware schedules
  while (ctas < kMaxCluster && ctas < chunks) ctas *= 2;
  if (chunks <= ctas) return launch_small<1, true>(ctas, ctl, base, cur, m, nbits, stream, tracked_out, keep_status, cs);
  return launch_small<2, true>(ctas, ctl, base, cur, m, nbits, stream, tracked_out, keep_status, cs);
}

}  // namespace lc
