// Pieces shared by the kernels of the encode pass: a lane's bit packers, the code tables in shared memory, and the
// out-of-line forms of coding a chunk (the vector's partial last chunk, and the rare cases).
#pragma once
#include "lc_common.cuh"

namespace lc {
namespace enc {

constexpr uint32_t kPackedLenShift = 26;                      // packed entry: length << 26 | code
constexpr uint32_t kPackedCodeMask = (1u << kPackedLenShift) - 1;
constexpr uint32_t kPackedMaxLen = 16;                        // two packed codes make one append of <= 32 bits
constexpr uint32_t kPackedLong = 63;                          // length field of a code that does not fit

struct Tables {
  uint32_t packed[256];  // by plane byte: length << 26 | code for codes of up to 16 bits, else length field 63
  uint2 full[256];       // by plane byte: {code, length} for codes of up to 32 bits
};

// Where the slow path gets an element's key from.
struct KeySource {
  const uint8_t* plane;  // used unless `wide`; in global or shared memory
  const float* base;
  const float* cur;
  bool wide;
  __device__ __forceinline__ uint32_t key(uint64_t c, uint32_t j, uint32_t lane, uint32_t e) const {
    if (wide) {
      const uint64_t i = c * kChunkElems + 128ull * j + 4 * lane + e;
      return __float_as_uint(__fsub_rn(cur[i], base[i])) >> 23;
    }
    const uint32_t b = plane[c * kChunkElems + (j >> 2) * 512 + lane * 16 + (j & 3) * 4 + e];
    return ((b & 1u) << 8) | (b >> 1);
  }
};

// Appends a code of at most 32 bits to the lane's bit accumulator and ORs completed 32-bit words into the
// chunk image at `dst` (shared or global memory).
struct OrPacker {
  unsigned long long acc;  // pending bits in the low `nb` bits
  uint32_t nb;
  uint32_t* dst;  // next word of the chunk this lane touches
  __device__ __forceinline__ void put(uint32_t code, uint32_t len) {
    acc = (acc << len) | code;
    nb += len;
    if (nb >= 32) {
      nb -= 32;
      atomicOr(dst, (uint32_t)(acc >> nb));
      dst += 1;
    }
  }
  __device__ __forceinline__ void flush() {
    if (nb > 0) atomicOr(dst, (uint32_t)(acc << (32 - nb)));
  }
};

// Slow, compact path (see the header). With dst == nullptr it only returns the lane's bit count;
// otherwise it ORs the lane's bits into the zeroed chunk image at dst, starting at bit lane_start.
// The plane bytes of four steps are read as one 16-byte vector, the way the fast path reads them. Codes come from the per-key table in global memory:
// passing the CTA's shared tables in as well was measured to cost the kernel's main loop 4 %.
static __device__ __noinline__ uint32_t chunk_slow(const EncEntry* __restrict__ enc, KeySource ks, uint64_t c,
                                            uint32_t lane, uint64_t n, uint32_t* dst, uint32_t lane_start) {
  OrPacker pk{0ull, lane_start & 31u, dst ? dst + (lane_start >> 5) : nullptr};
  uint32_t bits = 0;
  const bool from_plane = !ks.wide;
  for (uint32_t q = 0; q < kSteps / 4; ++q) {
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (from_plane) v = reinterpret_cast<const uint4*>(ks.plane + c * kChunkElems + q * 512)[lane];
    const uint32_t words[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (uint32_t r = 0; r < 4; ++r) {
      const uint32_t j = 4 * q + r;
#pragma unroll
      for (uint32_t e = 0; e < kGroup; ++e) {
        const uint64_t i = c * kChunkElems + 128ull * j + 4 * lane + e;
        if (i >= n) continue;
        uint32_t key;
        if (from_plane) {
          const uint32_t b = (words[r] >> (8 * e)) & 255u;
          key = ((b & 1u) << 8) | (b >> 1);
        } else {
          key = ks.key(c, j, lane, e);
        }
        const EncEntry en = enc[key];
        const uint32_t code_lo = en.code_lo, code_hi = en.code_hi, len = en.len;
        bits += len;
        if (dst) {
          if (len > 32) {
            pk.put(code_hi, len - 32);
            pk.put(code_lo, 32);
          } else {
            pk.put(code_lo, len);
          }
        }
      }
    }
  }
  if (dst) pk.flush();
  return bits;
}

__device__ __forceinline__ unsigned long long ld_tile(const unsigned long long* p) {
  return *reinterpret_cast<const volatile unsigned long long*>(p);
}
__device__ __forceinline__ void st_tile(unsigned long long* p, unsigned long long v) {
  *reinterpret_cast<volatile unsigned long long*>(p) = v;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Fast-path state of a lane: pending bits in hi:lo (low `nb` bits valid), next word slot in its column.
struct ColumnPacker {
  uint32_t hi, lo, nb;
  uint32_t dst;  // shared address of the next word of this lane's column (stride 128 bytes)
  uint32_t lim;  // shared address one past the column
  __device__ __forceinline__ void put(uint32_t code, uint32_t len) {
    // (hi:lo) = (hi:lo) << len | code, len <= 32
    hi = __funnelshift_lc(lo, hi, len);
    lo = __funnelshift_lc(0u, lo, len) | code;
    nb += len;
    // emit the oldest 32 pending bits once there are 32 or more, unless the column is full
    asm volatile(
        "{\n\t"
        ".reg .pred q;\n\t"
        ".reg .u32 w;\n\t"
        "setp.ge.u32 q, %0, 32;\n\t"
        "setp.lt.and.u32 q, %1, %4, q;\n\t"
        "@q sub.u32 %0, %0, 32;\n\t"
        "@q shf.r.clamp.b32 w, %3, %2, %0;\n\t"
        "@q st.shared.u32 [%1], w;\n\t"
        "@q add.u32 %1, %1, 128;\n\t"
        "}"
        : "+r"(nb), "+r"(dst)
        : "r"(hi), "r"(lo), "r"(lim)
        : "memory");
  }
};

// Packed table entries (shared address packed_addr) of the four plane bytes of `word`.
__device__ __forceinline__ void lookup4(uint32_t packed_addr, uint32_t word, uint32_t (&g)[4]) {
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const uint32_t b = __byte_perm(word, 0u, 0x4440 + e);  // plane byte of slot e
    // volatile: keeps the loads where they are written, one row ahead of their use
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(g[e]) : "r"(packed_addr + b * 4u));
  }
}

// Appends four codes whose packed entries are g, none of them the marker of a long code. Packed codes have at most 16
// bits, so two neighbours are joined into one append of at most 32 bits (half the accumulator and flush work).
__device__ __forceinline__ void put4_packed(ColumnPacker& pk, const uint32_t (&g)[4]) {
#pragma unroll
  for (int e = 0; e < 4; e += 2) {
    const uint32_t l0 = g[e] >> kPackedLenShift, l1 = g[e + 1] >> kPackedLenShift;
    const uint32_t c0 = g[e] & kPackedCodeMask, c1 = g[e + 1] & kPackedCodeMask;
    pk.put((c0 << l1) | c1, l0 + l1);
  }
}

// Ends a lane's column: writes the pending bits and returns the lane's bit count, or ~0 if the column was too small.
__device__ __forceinline__ uint32_t finish_column(const ColumnPacker& pk, uint32_t col0) {
  if (pk.nb >= 32 || (pk.nb > 0 && pk.dst >= pk.lim)) return 0xffffffffu;
  if (pk.nb > 0) asm volatile("st.shared.u32 [%0], %1;" ::"r"(pk.dst), "r"(pk.lo << (32 - pk.nb)) : "memory");
  return ((pk.dst - col0) >> 7) * 32 + pk.nb;
}

// Phase A for the vector's partial last chunk of `rem` elements: as for a whole chunk, with the slots beyond the end
// masked to empty codes and only the steps that hold elements visited. A kernel of its own size in miniature: one warp
// runs it once per call, and on vectors of a few thousand chunks everything else waits for that warp, so it must not
// take the element-by-element path (which took 20 us for the codes and 60 us for the tracked state). Out of line, so
// that it does not weigh on the registers of the main loop. Returns the lane's bit count, ~0 if a column overflowed.
static __device__ __noinline__ uint32_t code_partial(const Tables* tb, const uint4* ep, uint32_t rem, uint32_t lane,
                                              uint32_t col0, uint32_t lane_words) {
  ColumnPacker pk{0u, 0u, 0u, col0, col0 + lane_words * 128};
  const uint32_t packed_addr = smem_addr(tb->packed);
  const uint32_t rows = (rem + 127) / 128;
  uint4 nxt = *ep;
#pragma unroll 1
  for (uint32_t q = 0; 4 * q < rows; ++q) {
    const uint32_t words[4] = {nxt.x, nxt.y, nxt.z, nxt.w};
    if (q + 1 < kSteps / 4) nxt = ep[32 * (q + 1)];
    uint32_t g[4][4];
#pragma unroll
    for (uint32_t r = 0; r < 4; ++r) {
      lookup4(packed_addr, words[r], g[r]);
      const uint32_t first = (4 * q + r) * 128 + 4 * lane;
      const uint32_t have = first < rem ? rem - first : 0u;  // elements from this slot group on
#pragma unroll
      for (uint32_t e = 0; e < 4; ++e)
        if (e >= have) g[r][e] = 0u;  // no element: an empty code
    }
#pragma unroll
    for (uint32_t r = 0; r < 4; ++r) {
      if ((int)(g[r][0] | g[r][1] | g[r][2] | g[r][3]) < 0) {
#pragma unroll
        for (uint32_t e = 0; e < 4; ++e) {
          if (g[r][e] == 0u) continue;
          const uint2 f = tb->full[__byte_perm(words[r], 0u, 0x4440 + e)];
          pk.put(f.x, f.y);
        }
      } else {
        put4_packed(pk, g[r]);
      }
    }
  }
  return finish_column(pk, col0);
}

}  // namespace enc
}  // namespace lc
