// Small vectors: the whole compress pass (Algorithm 1 steps 4-6, optionally step 7) in one CTA and one launch.
//
// For a vector of one chunk the three kernels of the general path and the memset before them are all launch latency;
// layers of a few hundred elements are common in per-layer use. Bound: latency, so every part of the pass is spread over
// all 16 warps. A thread loads its (at most) eight elements once and keeps base and delta in registers through
// statistics, coding and the tracked state. Warp w takes the chunk's steps 2w and 2w + 1, so the codes of a thread are
// one contiguous piece of its lane's sub-stream: a scan over warps and lanes of the pieces' bit counts places them, and
// each thread ORs its piece into the chunk's image in shared memory, which leaves with 16-byte stores. Same bytes as the
// general path. A call of 1000 elements: 20.4 us with one warp coding
// alone and the earlier table pass, now 10.3 us.
#include "lc_small.cuh"

namespace lc {
namespace {

using namespace small;

__global__ void __launch_bounds__(kTableThreads)
small_compress_kernel(Control* ctl, const float* base, const float* cur, uint32_t n, int nbits, uint8_t* stream,
                      float* tracked_out, int keep_status) {
  extern __shared__ __align__(16) unsigned char s_small[];
  SmallShared& S = *reinterpret_cast<SmallShared*>(s_small);
  const uint32_t tid = threadIdx.x;
  const int earlier = keep_status ? ctl->status : 0;  // the same for every thread: nothing here has written it yet
  if (earlier) {
    clear_header(stream);
    return;
  }
  const int err = small_vector(S, base, cur, n, nbits, stream, tracked_out, ctl);
  if (err) clear_header(stream);
  if (tid == 0) {
    // what the memset of the general path clears, as far as later readers look at it
    ctl->status = err;  // barriers lie between the reads above and this
    ctl->ticket = 0;
    ctl->nsym = err ? 0 : S.T.nsym;
    ctl->wide = err ? 0 : S.T.wide;
    ctl->max_len = err ? 0 : S.T.max_len;
    ctl->payload_bits = err ? 0 : S.T.payload_bits;
  }
}

}  // namespace

cudaError_t launch_small_compress(Control* ctl, const float* base, const float* cur, uint64_t n, int nbits,
                                  uint8_t* stream, float* tracked_out, bool keep_status, cudaStream_t cs) {
  if (n == 0 || n > kSmallMaxElems) return cudaErrorInvalidValue;
  static bool ready[kMaxDevices] = {};  // by device ordinal
  const int dev = current_device_index();
  if (dev < 0) return cudaErrorInvalidDevice;
  if (!ready[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(small_compress_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallShared));
    if (e != cudaSuccess) return e;
    ready[dev] = true;
  }
  small_compress_kernel<<<1, kTableThreads, sizeof(SmallShared), cs>>>(ctl, base, cur, (uint32_t)n, nbits, stream, tracked_out,
                                                                      keep_status ? 1 : 0);
  return cudaGetLastError();
}

}  // namespace lc
