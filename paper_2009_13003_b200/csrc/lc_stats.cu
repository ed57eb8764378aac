// Statistics pass: fused delta, (sign, exponent) key extraction, 512-bin histogram with per-bin
// minimum / maximum, and the 1-byte-per-element key plane for the encode pass.
//
// Paper: Algorithm 1 step 4 (delta against the tracked state) and Section 3.1.1, exponent-based
// quantization (bucket = identical sign and exponent; representative from the bucket's min and max).
//
// Bound: HBM. 8 bytes per element must be read; 1 byte per element is written.
//
// Two settings decide whether the pass reaches that bound. (1) The L1 cache: a kernel with this much dynamic
// shared memory gets the largest shared-memory carve-out by default, and the small L1 that is left cannot keep
// enough loads in flight (the pass then runs 15 % slower). The launcher asks for just the carve-out its
// resident CTAs need. (2) Plain cached loads (ld.global.nc): with the L1 available they are faster than loads
// that bypass it. Two CTAs of 12 warps per SM share 2 x 68 KB of tables; three CTAs of 8 warps would need a
// carve-out that leaves no L1.
//
// Design for a skewed histogram (a handful of exponents hold almost all elements):
//  * counts live in shared memory as cnt[slot][lane] (slot = the key with the sign moved to bit 0):
//    every lane of a warp owns its own column, so the
//    32 atomics of one warp instruction always hit 32 different banks and never the same address,
//    whatever the keys are;
//  * min / max are kept per key as a pair of running maxima (of ~bits and of bits: inside one key the
//    order of the bit patterns is the order of the mantissas). A lane first reads the pair with a
//    plain load and only issues an atomic when its value would improve it, which after the first few
//    elements almost never happens;
//  * counts are integers and min / max are order-free, so the result is deterministic.
#include "lc_stats.cuh"

namespace lc {
namespace {

using namespace stats;

template <bool MEAN>
__global__ void __launch_bounds__(kStatsThreads, MEAN ? 1 : 2)
stats_kernel(const float* __restrict__ base, const float* __restrict__ cur, uint64_t n, uint64_t nunits,
             Control* __restrict__ ctl, uint8_t* __restrict__ plane) {
  extern __shared__ __align__(16) uint32_t smem[];
  begin_next();
  // MEAN: cnt, then the two sum tables, then mm
  constexpr uint32_t kTables = MEAN ? 3 : 1;
  uint32_t* cnt = smem;
  uint2* mm = reinterpret_cast<uint2*>(smem + kTables * kCntWords);
  for (uint32_t i = threadIdx.x; i < kTables * kCntWords + 2 * kKeys; i += kStatsThreads) smem[i] = 0;
  __syncthreads();

  const uint32_t lane = threadIdx.x & 31;
  const uint64_t warp = (uint64_t)blockIdx.x * (kStatsThreads / 32) + (threadIdx.x >> 5);
  const uint64_t nwarps = (uint64_t)gridDim.x * (kStatsThreads / 32);
  Acc<MEAN> acc{cnt + lane, mm};

  stats_units<MEAN, true>(acc, base, cur, n, warp, nunits, nwarps, lane, plane);
  wait_previous();  // the bins are clear
  __syncthreads();
  fold_stats<MEAN>(cnt, mm, ctl->count, ctl->inv_min, ctl->max_bits, ctl->mant_sum);
}

}  // namespace

cudaError_t launch_stats(const float* base, const float* cur, uint64_t n, Control* ctl, uint8_t* plane,
                         cudaStream_t cs, bool mean, bool overlap) {
  const WorkspaceLayout W = workspace_layout(n);
  if (W.nunits == 0) return cudaSuccess;
  static int blocks_per_sm[kMaxDevices][2] = {}, sms[kMaxDevices] = {};  // by device ordinal and kernel variant
  const int dev = current_device_index();
  if (dev < 0) return cudaErrorInvalidDevice;
  const int v = mean ? 1 : 0;
  const uint32_t smem = mean ? kStatsSmemMean : kStatsSmem;
  const void* fn = mean ? reinterpret_cast<const void*>(stats_kernel<true>) : reinterpret_cast<const void*>(stats_kernel<false>);
  if (blocks_per_sm[dev][v] == 0) {
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    int nsm = 0;
    if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    int bps = 0;
    e = mean ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, stats_kernel<true>, kStatsThreads, smem)
             : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, stats_kernel<false>, kStatsThreads, smem);
    if (e != cudaSuccess) return e;
    if (bps < 1) bps = 1;
    // carve-out in percent of the SM's 228 KB: the resident CTAs' shared memory (plus 1 KB each that the system
    // reserves), rounded up
    const int carve = (int)(((uint64_t)bps * (smem + 1024) * 100 + 228 * 1024 - 1) / (228 * 1024)) + 1;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, carve < 100 ? carve : 100);
    if (e != cudaSuccess) return e;
    sms[dev] = nsm;
    blocks_per_sm[dev][v] = bps;
  }
  const uint64_t want = (W.nunits + kStatsThreads / 32 - 1) / (kStatsThreads / 32);
  const uint64_t full = (uint64_t)sms[dev] * blocks_per_sm[dev][v];
  const unsigned grid = (unsigned)(want < full ? want : full);
  if (mean) {
    // the 32-bit column sums of the variant hold for a bounded number of units per warp (see kMeanMaxUnitsPerWarp)
    const uint64_t nwarps = (uint64_t)grid * (kStatsThreads / 32);
    if ((W.nunits + nwarps - 1) / nwarps > kMeanMaxUnitsPerWarp) return cudaErrorInvalidConfiguration;
    return launch_kernel(overlap, stats_kernel<true>, grid, kStatsThreads, smem, cs, base, cur, n, W.nunits, ctl, plane);
  }
  return launch_kernel(overlap, stats_kernel<false>, grid, kStatsThreads, smem, cs, base, cur, n, W.nunits, ctl, plane);
}

}  // namespace lc
