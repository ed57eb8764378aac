// Pieces shared by the kernels of the encode pass: a lane's bit packers, the code tables in shared memory, and the
// out-of-line forms of coding a chunk (the vector's partial last chunk, and the rare cases).
#pragma once
#include "lc_common.cuh"

namespace lc {
namespace enc {

// ---- code tables ---------------------------------------------------------------------------------------------
// A table entry holds its code left-aligned in the upper 24 bits and the length in the low byte: the code is then appended
// with one shift by the number of pending bits, and adding two entries adds their lengths.
constexpr uint32_t kEntryLenMask = 255u;
constexpr uint32_t kEntryMaxLen = 24;
constexpr uint32_t kEntryLong = 100u;      // length of an entry without a code: it takes every sum of two beyond 32
constexpr uint32_t kSingleMaxLen = 16;     // codes in `single`: two of them make one append of at most 32 bits
constexpr uint32_t kPairSpan = 32;         // values a byte takes in the index of a pair
// Words from one value of a pair's second element to the next. An odd number above 32: the bank then depends on both elements. With 32 it
// was the first element's value, of which a vector has a dozen that are frequent: 4.6 to 5.4 wavefronts a lookup, with 37 it
// is 2.7 to 3.1 (counted for Gaussian, Laplace, log-normal and Student deltas in 4 to 6 bits; 33 3.8 to 4.1, 35 2.8 to 3.2, 39 to 45 as 37).
constexpr uint32_t kPairStride = 37;
constexpr uint32_t kPairWords = (kPairSpan - 1) * kPairStride + kPairSpan;
static_assert(4 * kPairWords < 65536, "two byte offsets in one word");

struct Tables {
  union {
    uint32_t pair[kPairWords];  // both codes of two neighbouring elements
    uint32_t single[256];                  // by plane byte
  };
  uint2 full[256];     // by plane byte: {code, length} for codes of up to 32 bits
  uint32_t scan[256];  // while the table is built
  uint32_t best, below, above;
  int32_t base;        // see build_tables
  uint32_t use_pair;
  uint32_t long_codes;  // set by the kernel: some code is longer than 32 bits
};
// They lie at the start of the dynamic shared memory, so that the out-of-line functions below need no pointer to them (as one more argument it cost the
// encode pass's main loop registers: 268 M elements 158 us instead of 148).
constexpr uint32_t kTablesBytes = (uint32_t)((sizeof(Tables) + 127) / 128 * 128);
__device__ __forceinline__ Tables& shared_tables() {
  extern __shared__ __align__(128) unsigned char s_tables[];
  return *reinterpret_cast<Tables*>(s_tables);
}

__device__ __forceinline__ uint32_t make_entry(uint32_t code, uint32_t len, uint32_t longest) {
  return len > longest ? kEntryLong : (len ? code << (32 - len) : 0u) | len;
}

// Builds the table the coding loop looks codes up in; `full` is there, `sym0_len` is the zero bucket's code length and
// kept(b) tells whether plane byte b's bucket has a symbol of its own. All threads of a CTA of 256; ends with a barrier.
//
// Two neighbouring elements are looked up together: a plane byte b counts as clamp(b - base, 0, 31), and the two make an
// index of 10 bits. The clamped values cover 16 exponents of both signs, which is all that 2^5 - 1 kept buckets usually
// span; all bytes below are the zero bucket then. If more than that is kept, the 32 values go where most elements are, and
// a pair with an element outside is marked and coded the long way. Unless less than one element in 256 is outside, single
// bytes are looked up instead (one row of 128 elements in three would take the long way, which costs as much as it saves).
// A vector with one used symbol has no code bits at all: no pair is marked then (with all of them marked, 268 M elements of
// one bucket took 653 us instead of 505).
template <class Kept>
__device__ __forceinline__ void build_tables(Tables& tb, uint32_t sym0_len, Kept kept) {
  const uint32_t b = threadIdx.x, lane = b & 31, warp = b >> 5;
  const bool is_kept = kept(b);
  const uint32_t my_len = tb.full[b].y;
  // the share of the elements that a code of this length stands for, out of 2^22
  const auto share = [](uint32_t len) { return len == 0 || len > 22 ? 0u : 1u << (22 - len); };
  const uint32_t mine = is_kept ? share(my_len) : 0u;
  uint32_t incl = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t v = __shfl_up_sync(0xffffffffu, incl, d);
    if ((int)lane >= d) incl += v;
  }
  const uint32_t ballot = __ballot_sync(0xffffffffu, is_kept);
  if (b == 0) tb.best = 0, tb.below = 255, tb.above = 0;
  __syncthreads();
  tb.scan[b] = incl;
  if (lane == 0 && ballot) {
    atomicMin(&tb.below, 32 * warp + __ffs(ballot) - 1);
    atomicMax(&tb.above, 32 * warp + 31 - __clz(ballot));
  }
  __syncthreads();
  for (uint32_t w = 0; w < warp; ++w) incl += tb.scan[32 * w + 31];
  __syncthreads();
  tb.scan[b] = incl;  // share of the kept bytes up to b
  __syncthreads();
  const uint32_t lowest = tb.below, highest = tb.above;  // of the kept bytes; 255 and 0 if there are none
  // candidate: base = b. Values 1..30 are bytes of their own; 0 and 31 stand for all beyond, if those are of one kind.
  {
    const uint32_t upto = tb.scan[min(b + 30, 255u)];
    uint32_t covered = upto - incl;
    if (lowest > b || lowest > highest) covered += share(sym0_len);
    if (highest <= b + 31 && b + 31 < 256) covered += tb.scan[b + 31] - upto;
    const uint32_t score = __reduce_max_sync(0xffffffffu, covered << 8 | b);  // covered <= 2^22
    if (lane == 0) atomicMax(&tb.best, score);
  }
  __syncthreads();
  const int32_t base = (int32_t)(tb.best & 255u);
  const uint32_t covered = tb.best >> 8, all = tb.scan[255] + share(sym0_len);
  const bool use_pair = lowest > highest || all - covered <= all >> 8;
  if (b == 0) {
    tb.base = base;
    tb.use_pair = use_pair ? 1u : 0u;
  }
  if (use_pair) {
    for (uint32_t k = b; k < kPairSpan * kPairSpan; k += 256) {
      const uint32_t v0 = k % kPairSpan, v1 = k / kPairSpan;  // clamped bytes of the first and second element
      const auto escapes = [&](uint32_t v) { return all == 0 ? false : v == 0 ? lowest <= (uint32_t)base && lowest <= highest : v == 31 && highest > (uint32_t)base + 31; };
      const uint2 f0 = tb.full[min(base + v0, 255u)], f1 = tb.full[min(base + v1, 255u)];
      const uint32_t len = f0.y + f1.y;
      tb.pair[v1 * kPairStride + v0] = escapes(v0) || escapes(v1) || f0.y > 32 || f1.y > 32 ? kEntryLong : make_entry(f0.x << (f1.y & 31) | f1.x, len, kEntryMaxLen);
    }
  } else {
    tb.single[b] = make_entry(tb.full[b].x, my_len, kSingleMaxLen);
  }
  __syncthreads();
}

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
    return key_of_byte(plane[c * kChunkElems + (j >> 2) * 512 + lane * 16 + (j & 3) * 4 + e]);
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

// Whether a chunk has elements that the plane does not identify (byte 0), in a vector that has some; the whole warp. Out of line: rare.
static __device__ __noinline__ bool has_escape(const uint8_t* plane, uint32_t c, uint32_t lane) {
  const uint4* p = reinterpret_cast<const uint4*>(plane + (uint64_t)c * kChunkElems) + lane;
  uint32_t zero = 0;
#pragma unroll
  for (uint32_t q = 0; q < kSteps / 4; ++q) {
    const uint4 v = __ldg(p + 32 * q);
    const auto of = [](uint32_t x) { return (x - 0x01010101u) & ~x & 0x80808080u; };  // not zero if one of x's bytes is
    zero |= of(v.x) | of(v.y) | of(v.z) | of(v.w);
  }
  return __any_sync(0xffffffffu, zero != 0);
}

// A whole chunk from the CTA's tables: with dst == nullptr returns the lane's bits, otherwise ORs them into the zeroed chunk image at `dst`. Plane bytes
// as the fast path reads them.
__device__ __forceinline__ uint32_t chunk_from_tables(const Tables& tb, const uint4* ep, uint32_t* dst, uint32_t lane_start) {
  uint32_t bits = 0;
  OrPacker pk{0ull, lane_start & 31u, dst ? dst + (lane_start >> 5) : nullptr};
  uint4 v = ep[0];
#pragma unroll 1
  for (uint32_t q = 0; q < kSteps / 4; ++q) {
    const uint4 nxt = ep[32 * (q + 1 < kSteps / 4 ? q + 1 : q)];
    const uint32_t words[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (uint32_t r = 0; r < 4; ++r) {
      uint2 f[kGroup];
#pragma unroll
      for (uint32_t e = 0; e < kGroup; ++e) {
        f[e] = tb.full[__byte_perm(words[r], 0u, 0x4440 + e)];
        bits += f[e].y;
      }
      if (dst) {
#pragma unroll
        for (uint32_t e = 0; e < kGroup; ++e) pk.put(f[e].x, f[e].y);
      }
    }
    v = nxt;
  }
  if (dst) pk.flush();
  return bits;
}

// Slow, compact path (see the header). With dst == nullptr it only returns the lane's bit count;
// otherwise it ORs the lane's bits into the zeroed chunk image at dst, starting at bit lane_start.
// The plane bytes of four steps are read as one 16-byte vector, the way the fast path reads them. Codes come from the per-key table in global memory.
// TABLES: the kernel keeps the CTA's code tables at the start of its dynamic shared memory (one launched without them has nothing there to read).
template <bool TABLES>
static __device__ __noinline__ uint32_t chunk_slow(const EncEntry* __restrict__ enc, KeySource ks, uint64_t c,
                                            uint32_t lane, uint64_t n, uint32_t* dst, uint32_t lane_start) {
  // A whole chunk that outgrew its columns or its image. (A vector of layers has some where exponents are rare, and a launch of one round of chunks waits for them:
  // 11.7 M elements in 62 layers, that have such a chunk, 88 us in 4 bits and 107 in 5 by the loop below, 62 and 70 so; 46.5 and 48 without one.)
  if constexpr (TABLES)
    if ((c + 1) * kChunkElems <= n && !ks.wide && !shared_tables().long_codes)
      return chunk_from_tables(shared_tables(), reinterpret_cast<const uint4*>(ks.plane + c * kChunkElems) + lane, dst, lane_start);
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
          key = key_of_byte((words[r] >> (8 * e)) & 255u);
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

// Fast-path state of a lane: pending bits at the top of `w` (`nb` < 32 of them), next word slot in its column.
struct ColumnPacker {
  uint32_t w, nb;
  uint32_t dst;  // shared address of the next word of this lane's column (stride 128 bytes)
  uint32_t lim;  // shared address one past the column
  // appends `len` <= 32 bits that stand left-aligned in `code` (zero below)
  __device__ __forceinline__ void put(uint32_t code, uint32_t len) {
    // the word that is complete with 32 or more bits is emitted, unless the column is full: nb then stays at 32 or more
    asm volatile(
        "{\n\t"
        ".reg .pred q;\n\t"
        ".reg .u32 t;\n\t"
        "shr.u32 t, %4, %1;\n\t"
        "or.b32 %0, %0, t;\n\t"
        "shf.r.wrap.b32 t, 0, %4, %1;\n\t"  // the bits that do not fit: code << (32 - nb), 0 if nb is 0
        "add.u32 %1, %1, %5;\n\t"
        "setp.ge.u32 q, %1, 32;\n\t"
        "setp.lt.and.u32 q, %2, %3, q;\n\t"
        "@q st.shared.u32 [%2], %0;\n\t"
        "@q mov.u32 %0, t;\n\t"
        "@q add.u32 %2, %2, 128;\n\t"
        "@q sub.u32 %1, %1, 32;\n\t"
        "}"
        : "+r"(w), "+r"(nb), "+r"(dst)
        : "r"(lim), "r"(code), "r"(len)
        : "memory");
  }
  // a code of at most 32 bits as `full` has it
  __device__ __forceinline__ void put_full(uint2 f) { put(f.y ? f.x << (32 - f.y) : 0u, f.y); }
  // two entries, lengths together at most 32
  __device__ __forceinline__ void put_two(uint32_t e0, uint32_t e1, uint32_t len) {
    put((e0 & ~kEntryLenMask) | __funnelshift_r(e1 & ~kEntryLenMask, 0u, e0), len);  // shift by the low 5 bits: e0's length
  }
};

// Entries of the two pairs of a row's plane bytes `word`: elements 0 and 1, elements 2 and 3. `neg_base`: -base in both
// halves. The four bytes are clamped two at a time, in 16-bit halves.
__device__ __forceinline__ uint2 lookup_pairs(const Tables& tb, uint32_t word, uint32_t neg_base) {
  const uint32_t v0 = __viaddmin_s16x2_relu(__byte_perm(word, 0u, 0x4240), neg_base, 0x001f001fu);  // elements 0, 2
  const uint32_t v1 = __viaddmin_s16x2_relu(__byte_perm(word, 0u, 0x4341), neg_base, 0x001f001fu);  // elements 1, 3
  const uint32_t at = (v1 * kPairStride + v0) * 4u;  // byte offsets of the two entries, one in each half
  const volatile char* t = reinterpret_cast<const volatile char*>(tb.pair);  // volatile: one row ahead of the use
  return make_uint2(*reinterpret_cast<const volatile uint32_t*>(t + (at & 0xffffu)),
                    *reinterpret_cast<const volatile uint32_t*>(t + (at >> 16)));
}
// One row (four elements) of which e holds the pairs' entries. A pair that is marked, or two that are longer than 32 bits
// together, send the warp the long way.
__device__ __forceinline__ void put_pairs(ColumnPacker& pk, const Tables& tb, uint32_t word, uint2 e) {
  const uint32_t len = (e.x + e.y) & kEntryLenMask;
  if (__builtin_expect(__any_sync(0xffffffffu, len > 32), 0)) {
#pragma unroll 1
    for (int k = 0; k < 4; ++k) pk.put_full(tb.full[(word >> (8 * k)) & 255u]);
  } else {
    pk.put_two(e.x, e.y, len);
  }
}

// The same with single bytes: entries of the four plane bytes, two appends of two.
__device__ __forceinline__ uint4 lookup_singles(const Tables& tb, uint32_t word) {
  const volatile uint32_t* t = tb.single;
  return make_uint4(t[word & 255u], t[(word >> 8) & 255u], t[(word >> 16) & 255u], t[word >> 24]);
}
__device__ __forceinline__ void put_singles(ColumnPacker& pk, const Tables& tb, uint32_t word, uint4 e) {
  const uint32_t l0 = (e.x + e.y) & kEntryLenMask, l1 = (e.z + e.w) & kEntryLenMask;
  if (__builtin_expect(__any_sync(0xffffffffu, max(l0, l1) > 32), 0)) {
#pragma unroll 1
    for (int k = 0; k < 4; ++k) pk.put_full(tb.full[(word >> (8 * k)) & 255u]);
  } else {
    pk.put_two(e.x, e.y, l0);
    pk.put_two(e.z, e.w, l1);
  }
}

// Codes a whole chunk's rows for one lane: `load(q)` gives the plane bytes of steps 4q .. 4q + 3, and row(word, j) is
// called behind step j. Plane bytes are read one q ahead, lookups run one row ahead of the appends (which depend on each
// other through the pending bits).
template <bool PAIR, class Load, class Row>
__device__ __forceinline__ void code_rows(ColumnPacker& pk, const Tables& tb, uint32_t neg_base, Load load, Row row) {
  uint4 now = load(0);
  if (PAIR) {
    uint2 a = lookup_pairs(tb, now.x, neg_base), b;
#pragma unroll 1
    for (int q = 0; q < (int)kSteps / 4; ++q) {
      const uint4 nxt = load(q + 1 < (int)kSteps / 4 ? q + 1 : q);
      b = lookup_pairs(tb, now.y, neg_base);
      put_pairs(pk, tb, now.x, a);
      row(now.x, 4 * q);
      a = lookup_pairs(tb, now.z, neg_base);
      put_pairs(pk, tb, now.y, b);
      row(now.y, 4 * q + 1);
      b = lookup_pairs(tb, now.w, neg_base);
      put_pairs(pk, tb, now.z, a);
      row(now.z, 4 * q + 2);
      a = lookup_pairs(tb, nxt.x, neg_base);  // first row of the next step (unused after the last step)
      put_pairs(pk, tb, now.w, b);
      row(now.w, 4 * q + 3);
      now = nxt;
    }
  } else {
    uint4 a = lookup_singles(tb, now.x), b;
#pragma unroll 1
    for (int q = 0; q < (int)kSteps / 4; ++q) {
      const uint4 nxt = load(q + 1 < (int)kSteps / 4 ? q + 1 : q);
      b = lookup_singles(tb, now.y);
      put_singles(pk, tb, now.x, a);
      row(now.x, 4 * q);
      a = lookup_singles(tb, now.z);
      put_singles(pk, tb, now.y, b);
      row(now.y, 4 * q + 1);
      b = lookup_singles(tb, now.w);
      put_singles(pk, tb, now.z, a);
      row(now.z, 4 * q + 2);
      a = lookup_singles(tb, nxt.x);
      put_singles(pk, tb, now.w, b);
      row(now.w, 4 * q + 3);
      now = nxt;
    }
  }
}

// Ends a lane's column: writes the pending bits and returns the lane's bit count, or ~0 if the column was too small.
__device__ __forceinline__ uint32_t finish_column(const ColumnPacker& pk, uint32_t col0) {
  if (pk.nb >= 32 || (pk.nb > 0 && pk.dst >= pk.lim)) return 0xffffffffu;
  if (pk.nb > 0) asm volatile("st.shared.u32 [%0], %1;" ::"r"(pk.dst), "r"(pk.w) : "memory");
  return ((pk.dst - col0) >> 7) * 32 + pk.nb;
}

// ORs a lane's `bits` bits from its column into the zeroed chunk image at `image` (shared or global memory), from bit `start` on.
__device__ __forceinline__ void or_column(const uint32_t* column, uint32_t lane, uint32_t bits, uint32_t start, uint32_t* image) {
  const uint32_t words = (bits + 31) >> 5, r = start & 31;
  uint32_t* out = image + (start >> 5);
  uint32_t prev = 0;
  for (uint32_t k = 0; k < words; ++k) {
    const uint32_t w = column[k * 32 + lane];
    atomicOr(out + k, __funnelshift_r(w, prev, r));
    prev = w;
  }
  const uint32_t tail = r ? prev << (32 - r) : 0u;
  if (tail) atomicOr(out + words, tail);
}

// Assembles a chunk's image in shared memory (`chunk_bytes` of it, 16-byte aligned) from the columns; the whole warp.
// Where every lane has 32 bits or more, a lane ends in another word than it begins in: it gets the bits of its first word that belong
// to the lane before out of that lane's register and writes every word that it completes with a plain store, and nothing has to be
// zeroed first. Otherwise (a partial chunk, codes of almost no bits) the lanes OR their words into the zeroed image.
__device__ __forceinline__ void assemble_chunk(const uint32_t* column, uint32_t lane, uint32_t bits, uint32_t start, uint32_t* image,
                                               uint32_t chunk_bytes) {
  if (__any_sync(0xffffffffu, bits < 32)) {
    uint4* im4 = reinterpret_cast<uint4*>(image);
    for (uint32_t k = lane; k < chunk_bytes / 16; k += 32) im4[k] = make_uint4(0, 0, 0, 0);
    __syncwarp();
    or_column(column, lane, bits, start, image);
    return;
  }
  const uint32_t r = start & 31, first = start >> 5, end = start + bits;
  const uint32_t whole = (end >> 5) - first;  // words that the lane completes, its first among them: 1 or more
  const uint32_t* col = column + lane;
  // what it leaves of the next word (a column is zero behind its bits, and may end before that word does)
  const uint32_t partial = __funnelshift_r(whole < (bits + 31) >> 5 ? col[whole * 32] : 0u, col[(whole - 1) * 32], r);
  const uint32_t carry = __shfl_up_sync(0xffffffffu, partial, 1);
  uint32_t* out = image + first;
  uint32_t prev = col[0];
  out[0] = prev >> r | (r ? carry : 0u);
#pragma unroll 4
  for (uint32_t k = 1; k < whole; ++k) {
    const uint32_t w = col[k * 32];
    out[k] = __funnelshift_r(w, prev, r);
    prev = w;
  }
  // the last lane's partial word, and zeros up to the end
  const uint32_t rest = __shfl_sync(0xffffffffu, partial, 31), at = __shfl_sync(0xffffffffu, end >> 5, 31) + lane;
  if (at < chunk_bytes / 4) image[at] = lane == 0 ? rest : 0u;
}

// Phase A for the vector's partial last chunk of `rem` elements: as for a whole chunk, with the slots beyond the end
// masked to empty codes and only the steps that hold elements visited. A kernel of its own size in miniature: one warp
// runs it once per call, and on vectors of a few thousand chunks everything else waits for that warp, so it must not
// take the element-by-element path (which took 20 us for the codes and 60 us for the tracked state). Out of line, so
// that it does not weigh on the registers of the main loop. Returns the lane's bit count, ~0 if a column overflowed.
static __device__ __noinline__ uint32_t code_partial(const Tables* tb, const uint4* ep, uint32_t rem, uint32_t lane,
                                              uint32_t col0, uint32_t lane_words) {
  ColumnPacker pk{0u, 0u, col0, col0 + lane_words * 128};
  const uint32_t rows = (rem + 127) / 128;
  uint4 nxt = *ep;
#pragma unroll 1
  for (uint32_t q = 0; 4 * q < rows; ++q) {
    const uint32_t words[4] = {nxt.x, nxt.y, nxt.z, nxt.w};
    if (q + 1 < kSteps / 4) nxt = ep[32 * (q + 1)];
    uint2 f[4][4];
#pragma unroll
    for (uint32_t r = 0; r < 4; ++r) {
      const uint32_t first = (4 * q + r) * 128 + 4 * lane;
#pragma unroll
      for (uint32_t e = 0; e < 4; ++e)  // no element: an empty code
        f[r][e] = first + e < rem ? tb->full[__byte_perm(words[r], 0u, 0x4440 + e)] : make_uint2(0u, 0u);
    }
#pragma unroll
    for (uint32_t r = 0; r < 4; ++r)
#pragma unroll
      for (uint32_t e = 0; e < 4; ++e) pk.put_full(f[r][e]);
  }
  return finish_column(pk, col0);
}

}  // namespace enc
}  // namespace lc
