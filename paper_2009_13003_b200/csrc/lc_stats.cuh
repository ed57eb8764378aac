// The statistics of a run of units in one CTA (see lc_stats.cu for the design): shared by the kernel for one vector and
// the kernel for the segments of a vector.
#pragma once
#include "lc_common.cuh"

namespace lc {
namespace stats {

constexpr int kStatsThreads = 384;
constexpr int kRows = 8;  // steps per unit
constexpr uint32_t kCntWords = kKeys * 32;
constexpr uint32_t kStatsSmem = (kCntWords + 2 * kKeys) * 4;  // 64 KB + 4 KB
// Mean-representative variant (format section 1.8): two more tables of the same shape hold, per key and lane, the
// sums of the low 12 and of the high 11 bits of the mantissa fields. A column receives at most 32 elements per warp
// and unit, so 32-bit sums hold for kMeanMaxUnitsPerWarp units per warp: 12 warps * 32 * 4095 * 2731 < 2^32.
constexpr uint32_t kStatsSmemMean = (3 * kCntWords + 2 * kKeys) * 4;  // 192 KB + 4 KB: one CTA per SM
constexpr uint64_t kMeanMaxUnitsPerWarp = 2731;

__device__ __forceinline__ float4 ld_stream(const float4* p) {
  float4 v;
  asm volatile("ld.global.nc.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p));
  return v;
}

// Slot of a delta's bucket in the shared-memory tables: (exponent field << 1) | sign. The two signs of one
// exponent are neighbours and 8 consecutive exponents fill the 16 bank pairs of a 64-bit access exactly once,
// so the few hot buckets of a vector (neighbouring exponents, both signs) rarely meet in a bank.
__device__ __forceinline__ uint32_t slot_of(uint32_t bits) { return ((bits >> 22) & 0x1FEu) | (bits >> 31); }
__device__ __forceinline__ uint32_t key_of_slot(uint32_t slot) { return ((slot & 1u) << 8) | (slot >> 1); }

// The plane bytes of four elements from their slots: slot ^ 1, and 0 where that is 256 or more; two at a time, in 16-bit halves.
__device__ __forceinline__ uint32_t plane_word(uint32_t k0, uint32_t k1, uint32_t k2, uint32_t k3) {
  const uint32_t lo = __vmins2(__byte_perm(k0, k1, 0x5410) ^ 0x00010001u, 0x01000100u);
  const uint32_t hi = __vmins2(__byte_perm(k2, k3, 0x5410) ^ 0x00010001u, 0x01000100u);
  return __byte_perm(lo, hi, 0x6420);
}

template <bool MEAN>
struct Acc {
  uint32_t* cnt_lane;  // &cnt[lane]
  uint2* mm;
  __device__ __forceinline__ void sum(uint32_t bits, uint32_t slot) {
    if (MEAN) {
      atomicAdd(cnt_lane + kCntWords + slot * 32, bits & 0xFFFu);
      atomicAdd(cnt_lane + 2 * kCntWords + slot * 32, (bits >> 12) & 0x7FFu);
    }
  }
  __device__ __forceinline__ void improve(uint32_t bits, uint32_t slot, uint2 cur) {
    if (~bits > cur.x) atomicMax(&mm[slot].x, ~bits);
    if (bits > cur.y) atomicMax(&mm[slot].y, bits);
  }
  __device__ __forceinline__ void add(uint32_t bits) {
    const uint32_t slot = slot_of(bits);
    atomicAdd(cnt_lane + slot * 32, 1u);
    sum(bits, slot);
    improve(bits, slot, mm[slot]);
  }
  // Four elements at once: the four reads of the running min / max pairs go out together, and one test
  // covers all eight comparisons, because after the first few elements none of them ever holds.
  __device__ __forceinline__ void add4(uint32_t d0, uint32_t d1, uint32_t d2, uint32_t d3, uint32_t k0, uint32_t k1,
                                       uint32_t k2, uint32_t k3) {
    const uint2 c0 = mm[k0], c1 = mm[k1], c2 = mm[k2], c3 = mm[k3];
    atomicAdd(cnt_lane + k0 * 32, 1u);
    atomicAdd(cnt_lane + k1 * 32, 1u);
    atomicAdd(cnt_lane + k2 * 32, 1u);
    atomicAdd(cnt_lane + k3 * 32, 1u);
    sum(d0, k0);
    sum(d1, k1);
    sum(d2, k2);
    sum(d3, k3);
    const bool any = (~d0 > c0.x) | (d0 > c0.y) | (~d1 > c1.x) | (d1 > c1.y) | (~d2 > c2.x) | (d2 > c2.y) |
                     (~d3 > c3.x) | (d3 > c3.y);
    if (any) {
      improve(d0, k0, c0);
      improve(d1, k1, c1);
      improve(d2, k2, c2);
      improve(d3, k3, c3);
    }
  }
};

// Units first, first + step, ... below `end` of the vector, one warp; PLANE: also the key plane.
template <bool MEAN, bool PLANE>
__device__ __forceinline__ void stats_units(Acc<MEAN>& acc, const float* __restrict__ base, const float* __restrict__ cur,
                                            uint64_t n, uint64_t first, uint64_t end, uint64_t step, uint32_t lane,
                                            uint8_t* __restrict__ plane) {
  for (uint64_t u = first; u < end; u += step) {
    const uint64_t i0 = u * kUnitElems;
    uint32_t ew[kRows];
    if (i0 + kUnitElems <= n) {
      const float4* b4 = reinterpret_cast<const float4*>(base + i0) + lane;
      const float4* c4 = reinterpret_cast<const float4*>(cur + i0) + lane;
      float4 b[kRows], c[kRows];
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        b[r] = ld_stream(b4 + 32 * r);
        c[r] = ld_stream(c4 + 32 * r);
      }
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        const uint32_t d0 = __float_as_uint(__fsub_rn(c[r].x, b[r].x));
        const uint32_t d1 = __float_as_uint(__fsub_rn(c[r].y, b[r].y));
        const uint32_t d2 = __float_as_uint(__fsub_rn(c[r].z, b[r].z));
        const uint32_t d3 = __float_as_uint(__fsub_rn(c[r].w, b[r].w));
        const uint32_t k0 = slot_of(d0), k1 = slot_of(d1), k2 = slot_of(d2), k3 = slot_of(d3);
        if (PLANE) ew[r] = plane_word(k0, k1, k2, k3);
        acc.add4(d0, d1, d2, d3, k0, k1, k2, k3);
      }
    } else {
      // ragged tail: the last units of the vector, element by element.
#pragma unroll 1
      for (int r = 0; r < kRows; ++r) {
        uint32_t word = 0;
        for (int e = 0; e < 4; ++e) {
          const uint64_t i = i0 + 128 * r + 4 * lane + e;
          uint32_t d = 0;
          if (i < n) {
            d = __float_as_uint(__fsub_rn(cur[i], base[i]));
            acc.add(d);
          }
          word |= (min(slot_of(d) ^ 1u, 256u) & 255u) << (8 * e);
        }
        ew[r] = word;
      }
    }
    if (PLANE) {
      uint4* ep = reinterpret_cast<uint4*>(plane + i0) + lane;
      ep[0] = make_uint4(ew[0], ew[1], ew[2], ew[3]);
      ep[32] = make_uint4(ew[4], ew[5], ew[6], ew[7]);
    }
  }
}

// Folds the 32 lane columns of each key and merges them into the global bins; all threads, behind a barrier. Returns
// whether this thread met a non-finite key.
template <bool MEAN>
__device__ __forceinline__ bool fold_stats(const uint32_t* cnt, const uint2* mm, unsigned long long* count, uint32_t* inv_min,
                                           uint32_t* max_bits, unsigned long long* mant_sum) {
  bool bad = false;
  for (uint32_t slot = threadIdx.x; slot < kKeys; slot += kStatsThreads) {
    uint32_t total = 0;
#pragma unroll 8
    for (uint32_t l = 0; l < 32; ++l) total += cnt[slot * 32 + ((l + threadIdx.x) & 31)];
    if (total != 0) {
      const uint32_t key = key_of_slot(slot);
      bad |= (key & 255u) == 255u;
      atomicAdd(&count[key], (unsigned long long)total);
      atomicMax(&inv_min[key], mm[slot].x);
      atomicMax(&max_bits[key], mm[slot].y);
      if (MEAN) {
        unsigned long long lo = 0, hi = 0;
        for (uint32_t l = 0; l < 32; ++l) {
          lo += cnt[kCntWords + slot * 32 + ((l + threadIdx.x) & 31)];
          hi += cnt[2 * kCntWords + slot * 32 + ((l + threadIdx.x) & 31)];
        }
        atomicAdd(&mant_sum[key], lo + (hi << 12));
      }
    }
  }
  return bad;
}

}  // namespace stats
}  // namespace lc
